"""Panels of several rows a lane: ties and near-ties of the pivot search between the
rows of one lane, and the factors themselves against exact sums.

A block of the panel kernel holds ceil(n / SMs) rows; the lanes of its pivot warp
hold the rows r, r + 32, r + 64 ... of it.  n = 5100 gives 34 rows a block on 152
SMs (two a lane), n = 9800 65 (three, the kernel for more than two).
"""
import numpy as np
import pytest

from gpu_util import handle, ozlu, torch

pytestmark = pytest.mark.gpu


def _rows_a_block(n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = -(-n // sms)
    if rows <= 32:
        pytest.skip("one row a lane on this device")
    return rows


@pytest.mark.parametrize("n", [5100, 9800])
def test_ties_between_the_rows_of_a_lane(n):
    # Column j < nb has entries of one magnitude (or of magnitudes that differ in
    # bit 45 only, the same order key) in rows 32 apart of one block, zeros
    # elsewhere; every other row has one entry, 2, in a column of its own.  No
    # elimination changes an entry, so the interchanges follow from the matrix.
    h = handle()
    nb, rows = 64, _rows_a_block(n)
    rng = np.random.default_rng(n)
    groups = []                                       # rows of one lane of one block
    for g in range(-(-nb // rows) + 1, n // rows):    # (rows below nb stay out)
        for r in range(rows - 32):
            groups.append([g * rows + r + 32 * q for q in range((rows - r + 31) // 32)])
    groups = [groups[i] for i in rng.permutation(len(groups))[:nb]]
    assert len(groups) == nb and all(len(x) >= 2 for x in groups)
    content = [None] * n                              # of the row: its column past nb
    entry = {}
    winner = []
    for j, rws in enumerate(groups):
        vals = np.ones(len(rws))
        kind = j % 4
        if kind == 1:
            vals[-1] += 2.0 ** -45                    # the last row wins by a low bit
        elif kind == 2:
            vals[:] += 2.0 ** -45
            vals[0] += 2.0 ** -45                     # the first one does
        elif kind == 3 and len(rws) > 2:
            vals[1] += 2.0 ** -45
        win = int(np.argmax(vals))                    # the lowest row among equal ones
        winner.append(rws[win])
        for r, v in zip(rws, vals * rng.choice([-1.0, 1.0], len(rws))):
            entry[r, j] = v
    cols = iter(rng.permutation(np.arange(nb, n)))
    for r in range(n):
        if r not in set(winner):
            content[r] = int(next(cols))
            entry[r, content[r]] = 2.0
    A = torch.zeros((n, n, 2), dtype=torch.float64, device="cuda")   # (column, row, component)
    rc = np.array(list(entry.keys()))
    A[torch.from_numpy(rc[:, 1]).cuda(), torch.from_numpy(rc[:, 0]).cuda(), 0] = \
        torch.tensor(list(entry.values()), dtype=torch.float64, device="cuda")
    # the interchanges: rows by what they hold
    where = list(range(n))                            # original row -> position
    at = list(range(n))                               # position -> original row
    holds = {content[r]: r for r in range(n) if content[r] is not None}
    holds.update({j: winner[j] for j in range(nb)})
    want = []
    for c in range(n):
        p = where[holds[c]]
        assert p >= c
        want.append(p + 1)
        a, b = at[c], at[p]
        at[c], at[p] = b, a
        where[b], where[a] = c, p
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.ones(1, dtype=torch.int32, device="cuda")
    ozlu.ozlu_getrf(h, 2, 0, n, A, n, ipiv, nb, info, ozlu.make_opts("fp16"))
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    np.testing.assert_array_equal(ipiv.cpu().numpy(), np.array(want))


def _ints(x, bits):
    """Components (..., nc) -> the value in units of 2^-bits, as Python integers."""
    out = np.zeros(x.shape[:-1], dtype=object)
    for c in range(x.shape[-1]):
        m, e = np.frexp(x[..., c])
        sh = e.astype(np.int64) - 53 + bits
        assert (sh[m != 0] >= 0).all()
        out = out + np.frompyfunc(lambda q, s: int(q) << max(int(s), 0), 2, 1)((m * 2.0 ** 53).astype(np.int64), sh)
    return out


@pytest.mark.parametrize("n,nb", [(5100, 128), (9800, 64)])
def test_factors_of_tall_panels(n, nb):
    # |P A - L U| at sampled entries, exactly.  Each entry takes an update per
    # panel and per level of the panel's recursion, fewer than n in all; each is
    # rounded to 106 bits of a value of at most max |U| (and cut off below that).
    h = handle()
    g = torch.Generator(device="cuda")
    g.manual_seed(n + 1)
    A = torch.zeros((n, n, 2), dtype=torch.float64, device="cuda")
    A[..., 0] = torch.rand((n, n), dtype=torch.float64, device="cuda", generator=g) - 0.5
    A[..., 1] = A[..., 0] * (torch.rand((n, n), dtype=torch.float64, device="cuda", generator=g) - 0.5) * 2.0 ** -55
    s = A[..., 0] + A[..., 1]
    A[..., 1] -= s - A[..., 0]
    A[..., 0] = s
    LU = A.clone()
    ipiv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.ones(1, dtype=torch.int32, device="cuda")
    ozlu.ozlu_getrf(h, 2, 0, n, LU, n, ipiv, nb, info, ozlu.make_opts("fp16"))
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    perm = np.arange(n)
    for k, p in enumerate(ipiv.cpu().numpy()):
        perm[[k, p - 1]] = perm[[p - 1, k]]
    umax = float(torch.triu(LU[..., 0].T).abs().max())
    rng = np.random.default_rng(n)
    pairs = [(n - 1, n - 1), (nb, nb - 1), (n - 1, nb - 1), (n - 1, 0), (0, n - 1)]
    pairs += [(int(i), int(j)) for i, j in rng.integers(0, n, (20, 2))]
    bits = 240
    for i, j in pairs:
        k = min(i, j + 1)
        row, col = _ints(LU[:k, i].cpu().numpy(), bits), _ints(LU[j, :k].cpu().numpy(), bits)
        acc = sum(a * b for a, b in zip(row, col))
        if i <= j:
            acc += int(_ints(LU[j, i].cpu().numpy()[None], bits)[0]) << bits
        d = (int(_ints(A[j, int(perm[i])].cpu().numpy()[None], bits)[0]) << bits) - acc
        assert abs(d) < n * umax * 2.0 ** (2 * bits - 105), (i, j, abs(d) / 2 ** (2 * bits))
