"""The split of a flip's change of F into a correlation and a quadratic part, and the tiling by which the
correlation is taken (psl_lin.cu): against the term-by-term definition, in plain integers.

For neighbour j, shifts k <= kin = min(j, L-1-j) have two partners and those up to kout = max(j, L-1-j)
one.  With coefficients A, B (two partners) and D, E (one),

    score(j) = sum_{k<=kin} A_k [s_{j+k} = s_{j-k}] + s_j sum_{p != j} g_{|p-j|} s_p + sum_{kin<k<=kout} E_k

with g = B where 2j-(L-1) <= p <= 2j, else D.  The kernel decides B or D per 64-position row and chunk and
adds the difference to the exact boundary afterwards.
"""
import numpy as np
import pytest

P, ROWS = 64, 128


def tiles(L, N, start):
    f = (start + 1) % L
    if N == L:
        segs, whole = [(0, L)], True
    else:
        segs, whole = [(f, min(N, L - f)), (0, N - min(N, L - f))], False
    out = [(s0 + x, min(P * ROWS, n - x)) for s0, n in segs for x in range(0, n, P * ROWS)]
    return out, whole, f


def kinds(g, tau):
    """Closed form of the kinds of rows in a chunk (bit 0 B, bit 1 D)."""
    jA, nb, qa, rmin, rmax = g
    b_lo, b_hi = max(-rmax, -((rmax - rmin) >> 1)), min(qa + nb - 1, (rmax + qa) >> 1)
    d_lo, d_hi = min(0, nb - 1 - rmax) - 1, qa + 1
    return (b_lo <= tau <= b_hi) | (2 if tau <= d_lo or tau >= d_hi else 0)


def e_step(E, j, L):
    kp, kc, op, oc = min(j - 1, L - j), min(j, L - 1 - j), max(j - 1, L - j), max(j, L - 1 - j)
    d = 0
    if kc > kp:
        d -= E[kc]
    if kc < kp:
        d += E[kp]
    if oc > op:
        d += E[oc]
    if oc < op:
        d -= E[op]
    return int(d)


@pytest.mark.parametrize("L,N,start", [(2, 2, 1), (3, 1, 0), (65, 20, 60), (300, 300, 17), (301, 100, 250), (301, 100, 299),
                                       (641, 640, 0), (700, 650, 600), (1000, 999, 998), (1001, 64, 467)])
def test_tiles_rows_and_boundary(L, N, start):
    rng = np.random.Generator(np.random.PCG64(L * 1000 + N))
    s = 1 - 2 * rng.integers(0, 2, L)
    B, D, E = (rng.integers(-1000, 1000, L) for _ in range(3))
    pad = np.zeros(6 * L + 4 * P * ROWS, dtype=np.int64)
    off = 3 * L + 2 * P * ROWS
    pad[off:off + L] = s
    Y, hits = {}, {}
    todo, whole, f = tiles(L, N, start)
    for jA, cnt in todo:
        nb, qa = (cnt + P - 1) // P, jA // P
        rmin, rmax = -((jA + P - 1) // P), (L - 1 - jA) // P
        acc = np.zeros((nb, P), dtype=np.int64)
        for tau in range(rmin - (nb - 1), rmax + 1):
            b = np.arange(nb)
            inside = (b + tau >= rmin) & (b + tau <= rmax)
            is_b = (b >= tau - qa) & (b <= tau + rmax)
            assert kinds((jA, nb, qa, rmin, rmax), tau) == int((inside & is_b).any()) | 2 * int((inside & ~is_b).any())
            S = np.stack([pad[off + jA + P * (r + tau):off + jA + P * (r + tau) + P] for r in range(nb)])
            u = np.abs(P * tau + np.arange(P)[:, None] - np.arange(P)[None, :])
            ok = (u >= 1) & (u < L)
            for c, rows in ((B, is_b), (D, ~is_b)):
                acc += (S * rows[:, None]) @ np.where(ok, c[np.minimum(u, L - 1)], 0)
        lo, hi = min(jA, L - 1 - jA) + 1, max(jA, L - 1 - jA)
        e = int(E[lo:hi + 1].sum()) if hi >= lo else 0
        for x in range(cnt):
            j = jA + x
            e += e_step(E, j, L) if x else 0
            Y[j], hits[j] = int(s[j]) * int(acc[x // P, x % P]) + e, hits.get(j, 0) + 1
    for i in range(1, N + 1):
        j = (start + i) % L
        kin, kout = min(j, L - 1 - j), max(j, L - 1 - j)
        want = sum(int(B[k]) * int(s[j]) * int(s[j + k] + s[j - k]) for k in range(1, kin + 1))
        want += sum(int(E[k]) + int(D[k]) * int(s[j]) * int(s[j + k] if j + k < L else s[j - k]) for k in range(kin + 1, kout + 1))
        o = j if whole or j < f else j - f
        j0 = j - o % P
        hi_t, hi_r = min(2 * j, L - 1), min(j0 + P * (j0 // P) + P - 1, L - 1)
        lo_t, lo_r = max(2 * j - (L - 1), 0), max(j0 - P * ((L - 1 - j0) // P), 0)
        band = lambda a, b: sum(int(B[abs(p - j)] - D[abs(p - j)]) * int(s[p]) for p in range(a, b))
        fix = band(hi_r + 1, hi_t + 1) if hi_t > hi_r else -band(hi_t + 1, hi_r + 1)
        fix += band(lo_t, lo_r) if lo_t < lo_r else -band(lo_r, lo_t)
        assert hits[j] == 1 and Y[j] + int(s[j]) * fix == want, (i, j)


def test_digits_are_exact_in_half_precision():
    """Three balanced base-4096 digits of a difference of two 24-bit values below 2^35, in FP32 arithmetic:
    within one unit, and at most 2048 in magnitude (a half holds those integers exactly)."""
    rng = np.random.Generator(np.random.PCG64(5))
    f = np.float32
    scale = 2.0 ** rng.uniform(0, 34, 200000)
    a = (rng.uniform(-0.5, 0.5, scale.size) * scale).astype(f)
    b = (rng.uniform(-0.5, 0.5, scale.size) * scale).astype(f)
    edge = np.array([2.0**34 * (1 - 2.0**-24), -(2.0**34), 2.0**34 - 2.0**10, 2047.5, 2048, 2**23 - 0.5, 2**23, 0], dtype=f)
    a, b = np.concatenate([a, edge, edge]), np.concatenate([b, -edge, f(0) * edge])
    magic = f(12582912.0)
    hi = a - b
    bb = hi - a
    e = (a - (hi - bb)) - (b + bb)
    rnd = lambda x: (x.astype(f) + magic) - magic
    d2 = rnd((hi * f(2.0**-24)).astype(f))
    r = (hi.astype(np.float64) - d2.astype(np.float64) * 2.0**24).astype(f) + e
    d1 = rnd(r * f(2.0**-12))
    d0 = rnd((r.astype(np.float64) - d1.astype(np.float64) * 4096).astype(f))
    got = d0.astype(np.float64) + 4096 * d1.astype(np.float64) + 2.0**24 * d2.astype(np.float64)
    assert np.abs(got - (a.astype(np.float64) - b.astype(np.float64))).max() <= 1.0
    for d in (d0, d1, d2):
        assert np.abs(d).max() <= 2048 and np.array_equal(d.astype(np.float16).astype(f), d)
