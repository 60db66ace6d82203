"""Long walks scored by the correlation on the tensor cores and one lookup per five shifts (psl_lin.cu),
against the subset-sum tables: the same decisions, and scores within the bound of the exact values.

The library takes that path when the long walks' tiles fill half the SMs it may use, so a context of two
SMs takes it for one walk and a context of the whole GPU does not."""
import numpy as np
import pytest

import psl_workloads as W
from helpers import fp32_error_ratios, have_gpu, same_decisions, submit_spec
import oracle as O

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


def run(P, specs, **kw):
    with P.Context(arena_bytes=1 << 30, max_walks=16, **kw) as ctx:
        ids = [submit_spec(ctx, s) for s in specs]
        name = ctx.hot_variant()
        ctx.run()
        return name, [(ctx.trace(i, s.budget), ctx.export_state(i), ctx.best(i)) for i, s in zip(ids, specs)]


@pytest.mark.parametrize("L,n_lmt", [(20001, 6912), (20480, 8192), (32769, 32769), (33000, 5500), (40000, 1 << 20),
                                     (65536, 12000), (65537, 12289), (70001, 4500), (131072, 8193)])
def test_same_decisions_as_the_tables(L, n_lmt):
    import paper_2107_09801_gb300 as P
    specs = [W.WalkSpec(L=L, seed=L + n_lmt + q, alpha1=a1, alpha2=a2, budget=5, n_lmt=n_lmt, ls_lmt=2, topk=1 + q)
             for q, (a1, a2) in enumerate([(1, 16), (2, 9), (4, 13)])]
    name, got = run(P, specs, max_sms=2)
    assert name == "k_lin + k_quad"
    other, want = run(P, specs)
    assert other != name
    for spec, (tr, st, best), (tr0, st0, best0) in zip(specs, got, want):
        assert same_decisions(tr, tr0)
        assert np.array_equal(st["C"], st0["C"]) and np.array_equal(st["pivot"], st0["pivot"])
        assert best[0] == best0[0] and np.array_equal(best[1], best0[1])
        F0 = O.fitness(O.autocorr(O.init_seq(spec.L, spec.seed)), spec.alpha1)[0]
        assert max(fp32_error_ratios(tr, F0)) <= 1.0


def test_short_and_long_walks_together():
    import paper_2107_09801_gb300 as P
    specs = [W.WalkSpec(L=L, seed=7 + L, alpha1=3, alpha2=11, budget=8, ls_lmt=3) for L in (100, 4095, 16383, 20001, 40000)]
    name, got = run(P, specs, max_sms=2, steps_per_graph=4)
    _, want = run(P, specs)
    for (tr, st, best), (tr0, st0, best0) in zip(got, want):
        assert same_decisions(tr, tr0) and np.array_equal(st["C"], st0["C"]) and best[0] == best0[0]
