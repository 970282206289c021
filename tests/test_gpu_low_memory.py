"""INT8 products where the binary16 residues do not fit in memory and the int8
ones do: the same results, also from CUDA graphs that are replayed.  The shortage
is made on the host (allocations from a given size on fail)."""
import numpy as np
import pytest

from synth import random_expansions

from gpu_util import dev, handle, host, ozlu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def limit():
    handle()
    yield ozlu.ozlu_debug_limit_alloc
    ozlu.ozlu_debug_limit_alloc(0)


def _between(N, S, G, m, n, k):
    """A size that workspaces of the binary16 planes of an m x n x k product exceed
    and those of its int8 planes do not, t values packed or not."""
    up = lambda v, q: (v + q - 1) // q * q
    planes = N * S * (up(m, 128) + up(n, 128)) * up(k, 64)
    t = G * N * m * n
    assert planes > t
    return planes * 3 // 2 + t


def test_product(limit):
    m, n, k = 200, 150, 500
    A, B = random_expansions(m, k, 4, 1, -3, 3), random_expansions(k, n, 4, 2, -3, 3)
    info = ozlu.ozlu_plan(212, k, ozlu.make_opts("int8"))
    out = []
    for size in (0, _between(info.n_mod, info.S, info.n_groups, m, n, k)):
        h = ozlu.ozlu_create(None)
        try:
            C = torch.zeros((n, m, 4), dtype=torch.float64, device="cuda")
            limit(size)
            for _ in range(2):
                ozlu.ozlu_gemm(h, 4, 0, m, n, k, 1, dev(A), m, dev(B), k, 0, C, m, ozlu.make_opts("int8"))
                torch.cuda.synchronize()
                out.append(host(C, m))
            # the residues of the int8 form and of the binary16 form are the same
            out.append(ozlu.ozlu_debug_fetch(h, 3, np.zeros((info.n_mod, info.S, m, k), np.int8)))
        finally:
            limit(0)
            ozlu.ozlu_destroy(h)
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[3])
    np.testing.assert_array_equal(out[0], out[4])
    np.testing.assert_array_equal(out[2], out[5])


def test_one_failure_is_enough(limit):
    # the allocation of the larger residues fails for any reason: the call goes on
    h = ozlu.ozlu_create(None)
    try:
        A, B = random_expansions(130, 70, 3, 3, -2, 2), random_expansions(70, 140, 3, 4, -2, 2)
        C = torch.zeros((140, 130, 3), dtype=torch.float64, device="cuda")
        ozlu.ozlu_debug_fetch(h, 6, np.zeros(1, np.int32))
        ozlu.ozlu_gemm(h, 3, 0, 1, 1, 1, 1, dev(A), 130, dev(B), 70, 0, C, 130, ozlu.make_opts("fp16"))
        first = []
        for fails in (2, 0):  # the padded and the exact size of the binary16 layout
            ozlu.ozlu_debug_fail_alloc(fails)
            ozlu.ozlu_gemm(h, 3, 0, 130, 140, 70, 1, dev(A), 130, dev(B), 70, 0, C, 130, ozlu.make_opts("int8"))
            torch.cuda.synchronize()
            first.append(host(C, 130))
        np.testing.assert_array_equal(first[0], first[1])
    finally:
        ozlu.ozlu_debug_fail_alloc(0)
        ozlu.ozlu_destroy(h)


def test_captured_factorisation(limit):
    n, nc, nb = 300, 2, 128
    A0 = dev(random_expansions(n, n, nc, 5, -1, 1))
    info = ozlu.ozlu_plan(106, nb, ozlu.make_opts("int8"))
    size = _between(info.n_mod, info.S, info.n_groups, n - nb, n - nb, nb)
    opts = ozlu.make_opts("int8", graph=1)
    out = []
    for lim in (0, size):
        h = ozlu.ozlu_create(None)
        try:
            small = dev(random_expansions(8, 8, nc, 6, -1, 1))
            piv = torch.zeros(n, dtype=torch.int32, device="cuda")
            inf = torch.zeros(1, dtype=torch.int32, device="cuda")
            ozlu.ozlu_getrf(h, nc, 0, 8, small, 8, piv, 8, inf, opts)  # the scratch that does not depend on n
            torch.cuda.synchronize()
            limit(lim)
            A = torch.empty_like(A0)
            for call in range(5):
                A.copy_(A0)
                ozlu.ozlu_getrf(h, nc, 0, n, A, n, piv, nb, inf, opts)
                torch.cuda.synchronize()
                assert int(inf.item()) == 0
                # eager, captured, then replayed: the workspace has not moved since
                assert ozlu.ozlu_get_stats(h).graph_status == min(call, 2)
                out.append((host(A, n), piv.cpu().numpy()))
        finally:
            limit(0)
            ozlu.ozlu_destroy(h)
    for lu, p in out[1:]:
        np.testing.assert_array_equal(lu, out[0][0])
        np.testing.assert_array_equal(p, out[0][1])


def test_p_bit_product(limit):
    h = handle()
    m, n, k, p = 150, 140, 300, 320
    info = ozlu.ozlu_mp_plan(p, k)
    size = _between(info.n_mod, info.S, info.n_groups, m, n, k)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)

    def rand(r, c):
        M = ozlu.MPMatrix(r, c, 10)
        lim = torch.randint(0, 1 << 32, (10, r * c), device="cuda", generator=g)
        lim[9] |= 1 << 31
        M.limbs.copy_(torch.where(lim >= 1 << 31, lim - (1 << 32), lim).to(torch.int32))
        M.signs.copy_(torch.randint(0, 2, (r * c,), device="cuda", generator=g))
        return M

    A, B = rand(m, k), rand(k, n)
    got = []
    for lim in (0, size):
        h = ozlu.ozlu_create(None)
        try:
            o = ozlu.make_opts("int8")
            ozlu.ozlu_mp_set_opts(h, o)
            C = ozlu.MPMatrix(m, n, 10)
            limit(lim)
            for _ in range(2):
                ozlu.ozlu_mp_gemm(h, p, m, n, k, 1, A.desc(), B.desc(), 0, C.desc())
            torch.cuda.synchronize()
            got.append((C.limbs.cpu().numpy(), C.exps.cpu().numpy(), C.signs.cpu().numpy()))
        finally:
            limit(0)
            ozlu.ozlu_destroy(h)
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)
