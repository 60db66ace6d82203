"""The correlation form (psl_lin.cu): state it shares with the tables (a walk's fixed-point sums lie in the space
of their last partial scores), and its failure path."""
import numpy as np
import pytest

import psl_workloads as W
from helpers import have_gpu, same_decisions, submit_spec
import oracle as O

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def wrapping_seed(L, n_lmt):
    """A seed whose first window holds both ends of the sequence (their neighbours have the longest shifts)."""
    return next(s for s in range(100000) if O.splitmix64(s, (L + 63) // 64) % L in range(L - n_lmt // 2 - 50, L - n_lmt // 2 + 50))


@pytest.mark.parametrize("L", [30721, 46081])  # 16 k-chunks of 1920 and of 2880 shifts: the last two are full
def test_walk_tuned_on_the_tables_before_its_first_move(L):
    """The autotuner runs the tables, split 16 ways, on a walk that has made no move; with one tile for two SMs
    the correlation then adds its shares to what lies in that space."""
    import paper_2107_09801_gb300 as P
    spec = W.WalkSpec(L=L, seed=wrapping_seed(L, 8192), alpha1=4, alpha2=13, budget=6, n_lmt=8192, ls_lmt=2)
    res = []
    for tune in (True, False):
        with P.Context(arena_bytes=1 << 30, max_walks=1) as ctx:
            wid = submit_spec(ctx, spec)
            if tune:
                ctx.autotune(reps=1)
                assert ctx.hot_variant().startswith("k_hot")
                ctx.set_max_sms(2)
                assert ctx.hot_variant() == "k_lin + k_quad"
            ctx.run()
            assert ctx.poll(wid)["state"] == P.PSL_DONE
            res.append((ctx.trace(wid, spec.budget), ctx.best(wid)))
    (tr, best), (tr0, best0) = res
    assert same_decisions(tr, tr0)
    assert best[0] == best0[0] and np.array_equal(best[1], best0[1])


def run_stalled(P, specs, stall, products, **kw):
    with P.Context(arena_bytes=1 << 30, max_walks=16, **kw) as ctx:
        ids = [submit_spec(ctx, s) for s in specs]
        ctx.step(2)
        name = ctx.hot_variant()
        for q in stall:
            ctx.inject_stall(ids[q], products)
        ctx.run()
        extra = W.WalkSpec(L=511, seed=99, budget=10)  # the context stays usable
        wid = submit_spec(ctx, extra)
        ctx.run()
        assert ctx.poll(wid)["state"] == P.PSL_DONE
        return name, [(ctx.poll(i), ctx.trace(i, s.budget), ctx.best(i)) for i, s in zip(ids, specs)]


@pytest.mark.parametrize("products", [True, False])
@pytest.mark.parametrize("stall", [[0], [2], [0, 1, 4]])
def test_a_wait_that_runs_out_fails_only_that_walk(products, stall):
    """Walks of more tiles than the two blocks have, so that the items after a failed one are the same block's."""
    import paper_2107_09801_gb300 as P
    specs = [W.WalkSpec(L=L, seed=60 + q, alpha1=3, alpha2=11, budget=6, n_lmt=n, ls_lmt=3)
             for q, (L, n) in enumerate([(70001, 20000), (40000, 6912), (65535, 6912), (32769, 32769), (50001, 8192)])]
    name, got = run_stalled(P, specs, stall, products, max_sms=2, steps_per_graph=2)
    assert name == "k_lin + k_quad"
    _, want = run_stalled(P, specs, [], products)
    for q, ((st, tr, best), (_, tr0, best0)) in enumerate(zip(got, want)):
        if q in stall:
            assert st["state"] == P.PSL_ERROR and st["error"] == -5 and st["moves"] == 2  # PSL_ETIMEOUT
        else:
            assert st["state"] == P.PSL_DONE
            assert same_decisions(tr, tr0) and best[0] == best0[0] and np.array_equal(best[1], best0[1])


@pytest.mark.parametrize("L,n_lmt,sms", [(30721, 8192, 2), (65537, 4500, 2), (70001, 6912, 2), (90001, 8193, 4),
                                         (33000, 12001, 4), (40000, 40000, 10)])
def test_partners_split_over_two_items(L, n_lmt, sms):
    """Half as many tiles as SMs: two items share a tile's partners and add their sums up."""
    import paper_2107_09801_gb300 as P
    spec = W.WalkSpec(L=L, seed=wrapping_seed(L, n_lmt) if n_lmt < L else 5, alpha1=4, alpha2=13, budget=6, n_lmt=n_lmt,
                      ls_lmt=2)
    name, ((st, tr, best),) = run_stalled(P, [spec], [], False, max_sms=sms)
    assert name == "k_lin + k_quad" and st["state"] == P.PSL_DONE
    _, ((_, tr0, best0),) = run_stalled(P, [spec], [], False)
    assert same_decisions(tr, tr0)
    assert best[0] == best0[0] and np.array_equal(best[1], best0[1])
