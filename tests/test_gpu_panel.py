"""The cooperative panel kernel at its edges.

Ties of the pivot search inside a block, between the lanes' two rows and
between blocks (the lowest row must win), zero pivots in
the middle of a base block, blocks of one row, base blocks of odd width, and
panels tall enough for two and for more rows per lane of the pivot warp.
"""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import dev, handle, host, ozlu, torch

pytestmark = pytest.mark.gpu


def _getrf(M, nb, panel_width=0):
    h = handle()
    n, nc = M.shape[0], M.shape[2]
    dA = dev(M)
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    ozlu.ozlu_getrf(h, nc, 0, n, dA, n, ipiv, nb, info, ozlu.make_opts("int8", panel_width=panel_width))
    torch.cuda.synchronize()
    return host(dA, n), ipiv.cpu().numpy(), int(info.item())


def _exact_pivots(lead):
    """Interchanges (1-based) of the LU in exact rationals, the lowest row on ties."""
    n = lead.shape[0]
    A = [[Fraction(int(v)) for v in row] for row in lead]
    out = []
    for k in range(n):
        p = max(range(k, n), key=lambda i: (abs(A[i][k]), -i))
        out.append(p + 1)
        A[k], A[p] = A[p], A[k]
        for i in range(k + 1, n):
            f = A[i][k] / A[k][k]
            assert f.denominator & (f.denominator - 1) == 0
            if f:
                for j in range(k + 1, n):
                    A[i][j] -= f * A[k][j]
    return out


@pytest.mark.parametrize("nc,n,nb", [(2, 32, 32), (4, 64, 48), (3, 128, 128)])
def test_ties_take_the_lowest_row(nc, n, nb):
    # a Sylvester Hadamard matrix, rows shuffled, rows and columns negated: every
    # multiplier is a small dyadic number (asserted below), so that every step is
    # exact, and most columns have many rows of one magnitude
    rng = np.random.default_rng(n)
    lead = np.array([[(-1.0) ** bin(i & j).count("1") for j in range(n)] for i in range(n)])
    lead = lead[rng.permutation(n)] * rng.choice([-1.0, 1.0], (n, 1)) * rng.choice([-1.0, 1.0], (1, n))
    ref = _exact_pivots(lead)
    M = np.zeros((n, n, nc))
    M[..., 0] = lead
    LU, piv, info = _getrf(M, nb)
    assert info == 0
    assert [int(p) for p in piv] == ref


@pytest.mark.parametrize("n,nb,width", [(50, 50, 0), (33, 33, 0), (17, 5, 0), (1, 1, 0), (96, 96, 64)])
def test_odd_widths_and_zero_columns(n, nb, width):
    # a zero column in the middle: its pivot is exactly zero, the rest goes on
    rng = np.random.default_rng(n)
    M = np.zeros((n, n, 4))
    M[..., 0] = rng.integers(-9, 10, (n, n)) + 0.0
    M[np.arange(n), np.arange(n), 0] += 40.0
    z = n // 2
    if n > 1:
        M[:, z, 0] = 0.0
    LU, piv, info = _getrf(M, nb, width)
    assert info == (z + 1 if n > 1 else 0)
    L = np.tril(LU[..., 0], -1) + np.eye(n)
    U = np.triu(LU[..., 0])
    PA = M[..., 0].copy()
    for k in range(n):
        PA[[k, piv[k] - 1]] = PA[[piv[k] - 1, k]]
    assert np.max(np.abs(PA - L @ U)) < 1e-11 * np.max(np.abs(PA)) * n


@pytest.mark.parametrize("n,nb", [(5100, 128), (9800, 64)])
def test_tall_panels(n, nb):
    # 34 rows per block (two per lane), 65 rows per block (more than two)
    h = handle()
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    A = torch.zeros((n, n, 2), dtype=torch.float64, device="cuda")
    A[..., 0] = torch.rand((n, n), dtype=torch.float64, device="cuda", generator=g) - 0.5
    LU = A.clone()
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.ones(1, dtype=torch.int32, device="cuda")
    opts = ozlu.make_opts("fp16")
    ozlu.ozlu_getrf(h, 2, 0, n, LU, n, ipiv, nb, info, opts)
    b = A[..., 0].sum(0)                     # column-major: sum over columns, x = 1
    X = torch.zeros((1, n, 2), dtype=torch.float64, device="cuda")
    X[0, :, 0] = b
    ozlu.ozlu_getrs(h, 2, 0, n, 1, LU, n, ipiv, X, n, opts)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert float(torch.tril(LU[..., 0].T, -1).abs().max()) <= 1.0
    # the residual of the solve in the leading components
    r = (X[0, :, 0] @ A[..., 0]) - b
    assert float(r.abs().max()) < 1e-10 * n
