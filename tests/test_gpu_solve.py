"""ozlu_getrs at the edges of its two forms: blocks of 32 rows, the split of the
warps over right-hand sides, interchanges beyond one list, pivots that point
backwards, zero pivots, and the first number of right-hand sides of the blocked
form.  The reference is the substitution in 480-bit fixed point.
"""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import handle, ozlu, torch

pytestmark = pytest.mark.gpu

FX = 480  # fractional bits of the reference


def _fixed(limbs):
    v = sum((Fraction(float(c)) for c in limbs), Fraction(0))
    return int(v * (1 << FX))  # exact: the inputs have their last bit above 2^-480


def _expand(rng, shape, nc, scale):
    x = np.zeros(shape + (nc,))
    for c in range(nc):
        x[..., c] = rng.uniform(-1, 1, shape) * scale * 2.0 ** (-54 * c)
    return x


def _factors(rng, n, nc):
    """Random triangles with |l|, |u| below 1 / n off a diagonal in [1, 2]:
    both inverses have entries below e."""
    M = _expand(rng, (n, n), nc, 1.0 / n)
    d = np.arange(n)
    M[d, d, 0] = rng.uniform(1, 2, n) * rng.choice([-1.0, 1.0], n)
    return M


def _solve(M, B, ipiv):
    n, nrhs = M.shape[0], B.shape[1]
    F = [[_fixed(M[i, j]) for j in range(n)] for i in range(n)]
    out = []
    for r in range(nrhs):
        x = [_fixed(B[i, r]) for i in range(n)]
        for k in range(n):
            p = int(ipiv[k]) - 1
            x[k], x[p] = x[p], x[k]
        for i in range(n):
            x[i] -= sum(F[i][k] * x[k] for k in range(i)) >> FX
        for i in range(n - 1, -1, -1):
            s = x[i] - (sum(F[i][k] * x[k] for k in range(i + 1, n)) >> FX)
            x[i] = (s << FX) // F[i][i] if F[i][i] else 0
        out.append(x)
    return out


def _run(M, B, ipiv, opts=None):
    n, nrhs, nc = B.shape
    LU = torch.from_numpy(np.ascontiguousarray(M.transpose(1, 0, 2))).cuda()
    X = torch.from_numpy(np.ascontiguousarray(B.transpose(1, 0, 2))).cuda()
    ozlu.ozlu_getrs(handle(), nc, 0, n, nrhs, LU, n, torch.from_numpy(ipiv).cuda(), X, n, opts)
    torch.cuda.synchronize()
    return X.cpu().numpy()


def _check(M, B, ipiv, got):
    n, nrhs, nc = B.shape
    ref = _solve(M, B, ipiv)
    # |inverse entries| < e each way, so a relative error u of every operation
    # and of the stored halfway result is below 2 e^2 (n + 3) u of the largest x;
    # u = 2^(1 - 53 nc) bounds a rounding to nc components and, with room, one
    # update of the blocked form (p = 53 nc bits of the row and column maxima)
    bound = 2.0 * 2.72 ** 2 * (n + 3) * 2.0 ** (1 - 53 * nc)
    for r in range(nrhs):
        top = max(abs(v) for v in ref[r])
        err = max(abs(_fixed_any(got[r, i]) - ref[r][i]) for i in range(n))
        assert Fraction(err, max(top, 1)) <= Fraction(bound), (r, float(Fraction(err, max(top, 1))))


def _fixed_any(limbs):
    return int(sum((Fraction(float(c)) for c in limbs), Fraction(0)) * (1 << FX))


@pytest.mark.parametrize("nc,n,nrhs", [(2, 1, 1), (2, 32, 2), (3, 33, 3), (4, 31, 4), (4, 65, 5), (3, 100, 8),
                                       (2, 96, 9), (4, 64, 16), (4, 70, 17), (2, 200, 1)])
def test_solve_against_fixed_point(nc, n, nrhs):
    rng = np.random.default_rng(1000 * n + nrhs)
    M, B = _factors(rng, n, nc), _expand(rng, (n, nrhs), nc, 1.0)
    ipiv = np.array([rng.integers(k, n) + 1 for k in range(n)], dtype=np.int32)
    _check(M, B, ipiv, _run(M, B, ipiv))


@pytest.mark.parametrize("n", [40, 600, 1100])
def test_interchanges_in_any_direction(n):
    # the triangles are the identity: the result is the permuted right-hand side,
    # with pivots that point backwards as well
    rng = np.random.default_rng(n)
    M = np.zeros((n, n, 2))
    M[np.arange(n), np.arange(n), 0] = 1.0
    B = _expand(rng, (n, 3), 2, 1.0)
    ipiv = rng.integers(1, n + 1, n).astype(np.int32)
    want = B.copy()
    for k in range(n):
        p = ipiv[k] - 1
        want[[k, p]] = want[[p, k]]
    got = _run(M, B, ipiv).transpose(1, 0, 2)
    # equal values (the random pairs are not normalised, the results are)
    assert [[_fixed_any(v) for v in row] for row in got] == [[_fixed_any(v) for v in row] for row in want]


@pytest.mark.parametrize("nrhs", [2, 17])
def test_zero_pivots_give_zeros(nrhs):
    rng = np.random.default_rng(nrhs)
    n, nc = 70, 3
    M, B = _factors(rng, n, nc), _expand(rng, (n, nrhs), nc, 1.0)
    for z in (3, 40, 69):
        M[z, z] = 0.0
    ipiv = np.arange(1, n + 1, dtype=np.int32)
    got = _run(M, B, ipiv)
    assert not got[:, [3, 40, 69]].any()
    _check(M, B, ipiv, got)


def test_options_without_a_plan_are_refused():
    rng = np.random.default_rng(5)
    M, B = _factors(rng, 40, 4), _expand(rng, (40, 1), 4, 1.0)
    with pytest.raises(ozlu.OzluError):
        _run(M, B, np.arange(1, 41, dtype=np.int32), ozlu.make_opts("int8", nslice=1))
