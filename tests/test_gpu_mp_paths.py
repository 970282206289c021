"""The forms of the p-bit conversion and CRT at their edges, bit for bit.

Four elements a thread against one; digits of every word count; elements whose
digits are exact halves, all ones or zeros, of both signs; elements far below
their row's largest; a warp per output against a thread per output; windows of
more than 32 words; an old C far above and below the product.  The oracle replays
sampled rows and columns (an output depends on its row and column only).  And
the LU of a singular matrix, whose zero pivot only the device knows.
"""
import random

import pytest

from oracle.mp import oz2_gemm_mp

from gpu_util import handle, ozlu, torch

pytestmark = pytest.mark.gpu


def _elem(rng, p, spread):
    kind = rng.randrange(8)
    N = (1 << (p - 1)) if kind == 0 else (1 << p) - 1 if kind == 1 else \
        ((1 << (p - 1)) | (1 << rng.randrange(p))) if kind == 2 else rng.getrandbits(p) | (1 << (p - 1))
    if kind == 3:
        return (0, 0)
    e = rng.randint(-3, 3) - (rng.randint(0, spread) if kind == 4 else 0)
    return (-N if rng.random() < 0.5 else N, e - p)


def _matrix(rng, rows, cols, p, spread):
    return [[_elem(rng, p, spread) for _ in range(cols)] for _ in range(rows)]


def _norm(pair, L):
    N, E = pair
    if N == 0:
        return (0, 0)
    s = 32 * L - abs(N).bit_length()
    return (N << s, E - s)


@pytest.mark.parametrize("m,n,k,p,beta", [
    (160, 161, 1000, 100, 0), (161, 160, 1021, 200, 1),     # four elements a thread
    (5, 6, 33, 31, 1), (4, 3, 9, 320, 1), (3, 4, 8, 700, 1), (2, 3, 7, 1216, 1), (1, 2, 1, 2000, 0),
    (20, 17, 300, 700, 1), (3, 18, 65, 1216, 0),            # wide: accumulators folded
    (128, 128, 4, 150, 1), (127, 129, 4, 150, 1)])          # a thread and a warp per output
def test_conversion_and_crt_forms(m, n, k, p, beta):
    rng = random.Random(m * 1000 + p)
    L = (p + 31) // 32
    A, B = _matrix(rng, m, k, p, 2 * p), _matrix(rng, k, n, p, 2 * p)
    C = [[_elem(rng, p, 0) for _ in range(n)] for _ in range(m)]
    for i in range(m):
        C[i] = [(N, E + (3 * p + 500, -3 * p, 0)[(i + j) % 3]) if N else (0, 0) for j, (N, E) in enumerate(C[i])]
    dA, dB, dC = (ozlu.MPMatrix.from_pairs(X, L) for X in (A, B, C))
    ozlu.ozlu_mp_gemm(handle(), p, m, n, k, -1, dA.desc(), dB.desc(), beta, dC.desc())
    torch.cuda.synchronize()
    got = dC.to_pairs()
    rows = sorted({0, 1 % m, 31 % m, 32 % m, m - 1})
    cols = sorted({0, 1 % n, 2 % n, 33 % n, n - 1})
    ref = oz2_gemm_mp([A[i] for i in rows], [[B[h][j] for j in cols] for h in range(k)], p, alpha=-1, beta=beta,
                      C=[[C[i][j] for j in cols] for i in rows] if beta else None)
    for a, i in enumerate(rows):
        for b, j in enumerate(cols):
            assert got[i][j] == _norm(ref[a][b], L), (i, j)


@pytest.mark.parametrize("n,z", [(1, 0), (9, 4), (33, 32)])
def test_zero_pivot_goes_on(n, z):
    # a zero column: info names it, its multipliers are left alone, the others are as usual
    rng = random.Random(n)
    p, L = 130, 5
    A = [[(0, 0) if j == z else (rng.getrandbits(p) | (1 << (p - 1)), -p + (4 if i == j else -4)) for j in range(n)]
         for i in range(n)]
    dA = ozlu.MPMatrix.from_pairs(A, L)
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ozlu.ozlu_mp_getrf(handle(), p, n, dA.desc(), ipiv, 8, info)
    torch.cuda.synchronize()
    assert int(info.item()) == z + 1
    LU = [[N * 2.0 ** E for N, E in row] for row in dA.to_pairs()]
    want = [[N * 2.0 ** E for N, E in row] for row in A]
    for k, q in enumerate(ipiv.cpu().tolist()):
        want[k], want[q - 1] = want[q - 1], want[k]
    for i in range(n):
        for j in range(n):
            # L's diagonal is 1
            v = sum(LU[i][h] * LU[h][j] for h in range(min(i, j + 1))) + (LU[i][j] if i <= j else 0.0)
            assert abs(v - want[i][j]) <= 1e-13 * 32
