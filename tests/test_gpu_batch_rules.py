"""Kernel variants chosen by the size of the batch give the same walks: blocks and tiles of the table
kernel when the configuration leaves them open, and the width of the short walks' step tail."""
import numpy as np
import pytest

import psl_workloads as W
from helpers import have_gpu, same_decisions, submit_spec

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def run(P, specs, keep, **kw):
    with P.Context(arena_bytes=2 << 30, max_walks=len(specs), **kw) as ctx:
        ids = [submit_spec(ctx, s) for s in specs]
        name = ctx.hot_variant()
        ctx.run()
        return name, [(ctx.trace(ids[q], specs[q].budget), ctx.best(ids[q])) for q in keep]


@pytest.mark.parametrize("L,walks,name", [(31, 400, "k_hot_batched<512,16,4>"), (1023, 400, "k_hot_batched<512,16,4>"),
                                          (4095, 64, "k_hot_batched<512,16,4>"), (8191, 64, "k_hot_batched<512,32,8>")])
def test_same_walks_in_any_batch(L, walks, name):
    import paper_2107_09801_gb300 as P
    specs = [W.WalkSpec(L=L, seed=q, alpha1=2 + q % 4, alpha2=8 + q % 5, budget=12, ls_lmt=2, topk=1 + q % 3) for q in range(walks)]
    keep = [0, 1, walks // 2, walks - 1]
    full, got = run(P, specs, keep, steps_per_graph=6)
    assert full == name
    few, want = run(P, [specs[q] for q in keep], range(len(keep)))  # 256 x 32, and eight-warp tail blocks
    assert few.startswith("k_hot_batched<256,32")
    for (tr, best), (tr0, best0) in zip(got, want):
        assert same_decisions(tr, tr0)
        assert best[0] == best0[0] and np.array_equal(best[1], best0[1])


@pytest.mark.parametrize("L,walks,lin", [(13500, 100, False), (20001, 80, False), (20001, 152, True), (20001, 160, False),
                                         (20001, 304, True), (32767, 90, False), (32767, 152, True), (65535, 77, True)])
def test_correlation_form_where_its_tiles_fill_the_sms(L, walks, lin):
    """On 152 SMs: a last wave of few tiles costs more than the lookups it saves."""
    import torch
    import paper_2107_09801_gb300 as P
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line depends on the number of SMs")
    n_lmt = 8192 if L == 13500 else 6912
    with P.Context(arena_bytes=walks * P.psl_walk_bytes(L, n_lmt, 0) + (64 << 20), max_walks=walks) as ctx:
        for q in range(walks):
            ctx.submit_ex(L, q, 4, 13, 10, n_lmt=n_lmt)
        assert (ctx.hot_variant() == "k_lin + k_quad") == lin


def test_autotuner_leaves_the_choice_open_when_there_is_none(tmp_path):
    """Tuning a batch that the correlation form scores stores nothing, and later batches keep the automatic rule."""
    import paper_2107_09801_gb300 as P
    cache = tmp_path / "tune.json"
    with P.Context(arena_bytes=1 << 30, max_walks=400, max_sms=2) as ctx:
        wid = ctx.submit_ex(70001, 1, 4, 13, 10)
        assert ctx.hot_variant() == "k_lin + k_quad"
        ctx.autotune(reps=1, cache=str(cache))
        assert not cache.exists()
        ctx.release(wid)
        ctx.set_max_sms(0)
        for q in range(400):
            ctx.submit_ex(1023, q, 4, 13, 10)
        assert ctx.hot_variant() == "k_hot_batched<512,16,4>"
        assert ctx.autotune(reps=1, cache=str(cache)) and cache.exists()


def test_kernel_name_of_a_mixed_batch():
    import paper_2107_09801_gb300 as P
    from paper_2107_09801_gb300 import binding as B
    with P.Context(arena_bytes=1 << 30, max_walks=8, max_sms=2) as ctx:
        for L in (1023, 40000, 70001):
            ctx.submit_ex(L, L, 4, 13, 10)
        full = ctx.hot_variant()
        table, _, rest = full.partition(" + ")
        assert table.startswith("k_hot_batched<") and rest == "k_lin + k_quad"
        for cap in range(1, len(full) + 2):  # truncated like snprintf, NUL-terminated, the full length returned
            buf = B.ct.create_string_buffer(b"x" * 63, 64)
            assert B.lib().psl_hot_variant(ctx.h, buf, cap) == len(full)
            assert buf.raw[:cap] == full.encode()[:cap - 1].ljust(cap, b"\0") and buf.raw[cap:cap + 1] == b"x"


@pytest.mark.parametrize("L,walks,name", [(255, 152, "k_hot_batched<256,32,4>"), (128, 120, "k_hot_batched<256,32,4>"),
                                          (255, 153, "k_hot_batched<512,16,4>"), (300, 114, "k_hot_batched<512,16,4>")])
def test_walks_of_one_small_block_each(L, walks, name):
    """On 152 SMs: blocks of 512 only when the blocks of 256 no longer have an SM each."""
    import torch
    import paper_2107_09801_gb300 as P
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line depends on the number of SMs")
    with P.Context(arena_bytes=walks * P.psl_walk_bytes(L, L, 0) + (64 << 20), max_walks=walks) as ctx:
        for q in range(walks):
            ctx.submit_ex(L, q, 4, 13, 10)
        assert ctx.hot_variant() == name


@pytest.mark.parametrize("base,extra,sms", [([(1023, 4, 13)] * 16, (1023, 4, 13), 8), ([(511, 2, 2)] * 4, (300, 4, 13), 8),
                                            ([(40000, 4, 13)] * 2, (1023, 4, 13), 2)])
def test_batches_that_take_other_kernels_and_return(base, extra, sms):
    """Graphs captured for one choice of kernels are used again when the batch returns to it."""
    import paper_2107_09801_gb300 as P
    spec = lambda q, t, budget: W.WalkSpec(L=t[0], seed=q, alpha1=t[1], alpha2=t[2], budget=budget, ls_lmt=3, n_lmt=6912)
    got = []
    for graph in (3, 0):
        with P.Context(arena_bytes=1 << 30, max_walks=32, max_sms=sms, steps_per_graph=graph) as ctx:
            specs = [spec(q, t, 33) for q, t in enumerate(base)]
            ids = [submit_spec(ctx, s) for s in specs]
            names, traces = set(), []
            for r in range(5):
                s = spec(100 + r, extra, 3)
                wid = submit_spec(ctx, s)
                names.add(ctx.hot_variant())
                ctx.step(3)
                traces.append(ctx.trace(wid, 3))
                ctx.release(wid)
                names.add(ctx.hot_variant())
                ctx.step(3)
            ctx.run()
            got.append(traces + [ctx.trace(i, 33) for i in ids])
    for tr, tr0 in zip(*got):
        assert len(tr) and same_decisions(tr, tr0)
    assert len(names) == 2 or base[0] == extra  # (there the step tail changes)


@pytest.mark.parametrize("batch,name", [([(131071, 1), (1023, 310)], "k_hot_batched<256,32,8>"),
                                        ([(16383, 1), (1023, 310)], "k_hot_batched<256,32,8>"),
                                        ([(16383, 1), (300, 2000)], "k_hot_batched<512,32,8>"),
                                        ([(8191, 50), (1023, 310)], "k_hot_batched<512,32,8>"),
                                        ([(2047, 4), (255, 120)], "k_hot_batched<512,16,4>")])
def test_few_long_walks_among_short_ones(batch, name):
    """On 152 SMs: the long walks' blocks finish last, and blocks of 256 spread them over more SMs."""
    import torch
    import paper_2107_09801_gb300 as P
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the line depends on the number of SMs")
    need = sum(n * P.psl_walk_bytes(L, 6912, 0) for L, n in batch)
    with P.Context(arena_bytes=need + (64 << 20), max_walks=sum(n for _, n in batch)) as ctx:
        for L, n in batch:
            for q in range(n):
                ctx.submit_ex(L, q, 4, 13, 10)
        assert ctx.hot_variant() == name
