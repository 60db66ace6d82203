"""psl_autocorr packs its sequences on the device, guard words included: lengths around word and block edges,
several sequences, on memory that earlier calls have filled."""
import numpy as np
import pytest

from helpers import fft_autocorr, have_gpu

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not have_gpu(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("L", [1, 2, 31, 32, 33, 127, 128, 129, 191, 192, 193, 255, 256, 257, 8191])
@pytest.mark.parametrize("nseq", [1, 5])
def test_autocorr_at_word_and_block_edges(L, nseq):
    import paper_2107_09801_gb300 as P
    gen = np.random.Generator(np.random.PCG64(L * 10 + nseq))
    with P.Context(arena_bytes=1 << 24, max_walks=1) as ctx:
        ctx.autocorr(-np.ones((nseq + 3, 8192), dtype=np.int8))  # every bit set
        s = (1 - 2 * gen.integers(0, 2, size=(nseq, L))).astype(np.int8)
        C = ctx.autocorr(s)
    for q in range(nseq):
        assert np.array_equal(C[q].astype(np.int64), fft_autocorr(s[q]))
