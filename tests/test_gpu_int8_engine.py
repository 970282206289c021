"""INT8 plans, whose residue products run as binary16 ones on the tensor cores.

The binary32 accumulators take 1024 products of residues at a time and are folded
into each other: inner dimensions at and just past the edges of one, two and
three accumulators (for S = 2 also with an edge inside a pair term), bytes and
packed t values, the residues that ozlu_debug_fetch reads back from their
binary16 form.  Constant matrices, so that every term of an accumulation has one
sign; an output depends on its row and column only, so the oracle replays one
1 x K by K x 1 product, and every t value and output must equal it bit for bit.
"""
import numpy as np
import pytest

from oracle import oz2

from gpu_util import gpu_gemm, handle, ozlu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc,S,k,m,n", [(2, 1, 1024, 130, 129), (2, 1, 1025, 130, 129), (3, 2, 512, 40, 130),
                                        (3, 2, 513, 129, 33), (4, 2, 1024, 5, 7), (4, 2, 1100, 130, 1),
                                        (4, 3, 700, 1, 130), (2, 1, 3137, 64, 64), (4, 2, 1536, 1025, 1153)])
def test_accumulators_of_an_int8_plan(nc, S, k, m, n):
    rng = np.random.default_rng(k + nc)
    a, b = ([rng.uniform(0.5, 1.0)] + [rng.uniform(-1, 1) * 2.0 ** (-55 * (c + 1)) for c in range(nc - 1)]
            for _ in range(2))
    A, B = np.zeros((m, k, nc)), np.zeros((k, n, nc))
    A[:], B[:] = a, b
    out = gpu_gemm(A, B, opts=ozlu.make_opts("int8", S))
    assert ozlu.ozlu_debug_fetch(handle(), 6, np.zeros(1, np.int32))[0] == 0
    ref_out, ref = oz2.oz2_gemm(A[:1], B[:, :1], 53 * nc, backend="int8", S=S, debug=True)
    pl = ref.plan
    t = ozlu.ozlu_debug_fetch(handle(), 5, np.zeros((len(pl.groups), pl.N, n, m), np.uint8))
    ra = ozlu.ozlu_debug_fetch(handle(), 3, np.zeros((pl.N, pl.S, m, k), np.int8))
    rb = ozlu.ozlu_debug_fetch(handle(), 4, np.zeros((pl.N, pl.S, n, k), np.int8))
    for l in range(pl.N):
        for gi, g in enumerate(pl.groups):
            assert (t[gi, l] == ref.t[(l, g)][0, 0]).all()
        for s in range(pl.S):
            assert (ra[l, s] == ref.res_A[(l, s)][0, 0]).all()
            assert (rb[l, s] == ref.res_B[(l, s)][0, 0]).all()
    assert (out == ref_out[0, 0]).all()
