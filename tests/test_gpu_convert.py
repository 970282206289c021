"""The fused conversion at its edges, bit for bit against the oracle.

Digit widths w on both sides of a 32-bit word boundary, X in 8 and in 12 words
(large guard settings), one and four elements per thread (few and many
positions), moduli split over the grid, K next to the padding step, and
entries whose digits are all ones, all zeros or a lone top bit.  Outputs are
single-valued, so the comparison is exact.
"""
import numpy as np
import pytest

from oracle import oz2
from synth import random_expansions

from gpu_util import gpu_gemm, ozlu

pytestmark = pytest.mark.gpu


def _special(M):
    """Entries with extreme digit patterns: +-1, one unit below, a lone low bit."""
    nc = M.shape[2]
    for i, lead in enumerate([1.0, -1.0, 1.0, -1.0, 0.0, 2.0 ** -50]):
        M[i % M.shape[0], i % M.shape[1]] = 0.0
        M[i % M.shape[0], i % M.shape[1], 0] = lead
        if i in (2, 3):   # 1 - tiny: every digit below the top all ones (or its negative)
            M[i % M.shape[0], i % M.shape[1], nc - 1] = -lead * 2.0 ** (-53 * nc + 2)
    return M


def _w(nc, k, S, g_ex, be):
    return ozlu.ozlu_plan(53 * nc, k, ozlu.make_opts(be, S, 0, g_ex)).w


@pytest.mark.parametrize("be", ["int8", "fp16", "fp8"])
@pytest.mark.parametrize("nc,S,wmod", [(4, 2, 0), (4, 2, 31), (4, 3, 1), (3, 2, 0), (2, 1, 31), (4, 0, 0)])
@pytest.mark.parametrize("shape", [(9, 65, 5), (650, 250, 600)])
def test_digit_word_boundaries(be, nc, S, wmod, shape):
    m, k, n = shape
    g_ex = 0
    if S:  # the guard bits that put w on the wanted side of a word boundary
        while _w(nc, k, S, g_ex, be) % 32 != wmod:
            g_ex += 1
    _check(be, nc, S, g_ex, m, k, n)


@pytest.mark.parametrize("be", ["int8", "fp16"])
@pytest.mark.parametrize("shape", [(9, 64, 5), (650, 255, 600)])
def test_wide_inputs(be, shape):
    # 90 guard bits: X takes more than 8 words
    m, k, n = shape
    opts = ozlu.make_opts(be, 3, 0, 90)
    info = ozlu.ozlu_plan(212, k, opts)
    assert info.Q + 1 > 8 * 32
    _check(be, 4, 3, 90, m, k, n)


def _check(be, nc, S, g_ex, m, k, n):
    A = _special(random_expansions(m, k, nc, 7 + m + k, -6, 0))
    B = _special(random_expansions(k, n, nc, 8 + n + k, -6, 0))
    out = gpu_gemm(A, B, opts=ozlu.make_opts(be, S, 0, g_ex))
    rows = np.unique(np.concatenate([np.arange(min(m, 6)), [m - 1]]))
    cols = np.unique(np.concatenate([np.arange(min(n, 4)), [n - 1]]))
    ref = oz2.oz2_gemm(A[rows], B[:, cols], 53 * nc, backend=be, S=S or None, g_ex=g_ex)
    np.testing.assert_array_equal(out[np.ix_(rows, cols)], ref)
