"""The packed t values (a 32-bit word per triple of moduli) at ragged sizes.

Products with enough 128 x 128 tiles leave the tensor-core epilogue packed by
triples of moduli; smaller ones as bytes.  Ragged rows and columns, every
remainder of the number of moduli by three, and old values of C below, inside
and far above the product's window (the wide path of the CRT) are compared
bit for bit with the oracle on sampled rows and columns, and the t values that
ozlu_debug_fetch recovers from the words with the oracle's.
"""
import numpy as np
import pytest

from oracle import oz2
from synth import random_expansions

from gpu_util import gpu_gemm, handle, ozlu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("be,nc,S,g_ex,m,n,k", [("fp16", 4, 2, 0, 1000, 1157, 70), ("fp16", 4, 3, 0, 1001, 1153, 65),
                                                ("fp16", 3, 2, 4, 1155, 1025, 33), ("fp8", 4, 2, 0, 1000, 1157, 130),
                                                ("fp8", 2, 1, 0, 1920, 1281, 70), ("fp8", 4, 2, 8, 1025, 1153, 1)])
def test_packed_ragged(be, nc, S, g_ex, m, n, k):
    A = random_expansions(m, k, nc, 11 + m, -8, 8)
    B = random_expansions(k, n, nc, 12 + n, -8, 8)
    C = random_expansions(m, n, nc, 13 + k, -10, 10)
    C[1::7] = np.ldexp(C[1::7], 300)      # far above the product: the grid is raised
    C[2::7] = np.ldexp(C[2::7], 90)       # above the narrow window or inside it
    C[3::7] = np.ldexp(C[3::7], -400)     # below the grid
    C[4::7] = 0.0
    opts = ozlu.make_opts(be, S, 0, g_ex)
    out = gpu_gemm(A, B, alpha=-1, beta=1, C=C, opts=opts)
    rows = np.unique(np.concatenate([np.arange(8), [127, 128, m - 1]]))
    cols = np.array([0, 31, 32, 128, n - 1])
    ref, dbg = oz2.oz2_gemm(A[rows], B[:, cols], 53 * nc, alpha=-1, beta=1, C=C[np.ix_(rows, cols)], backend=be,
                            S=S, g_ex=g_ex, debug=True)
    np.testing.assert_array_equal(out[np.ix_(rows, cols)], ref)
    pl = dbg.plan
    t = ozlu.ozlu_debug_fetch(handle(), 5, np.zeros((len(pl.groups), pl.N, n, m), np.uint8))
    for l in range(pl.N):
        for gi, g in enumerate(pl.groups):
            np.testing.assert_array_equal(t[gi, l][np.ix_(cols, rows)].T, dbg.t[(l, g)])
