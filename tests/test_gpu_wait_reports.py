"""A bounded device wait that runs out inside a call reaches the caller: as the
return value where the call waits for the GPU anyway, else as the handle's error
word, also where the handle's sub-streams ran it.  The wait is one of the library's
own routines on a word or barrier that nothing sets, with a short limit."""
import numpy as np
import pytest

from synth import random_expansions

from gpu_util import dev, handle, ozlu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def h():
    handle()
    h = ozlu.ozlu_create(None)
    yield h
    ozlu.ozlu_destroy(h)


def _word(h):
    return int(ozlu.ozlu_debug_fetch(h, 6, np.zeros(1, np.int32))[0])


def _system(n, nrhs, nc=2):
    M = random_expansions(n, n, nc, 1, -1, 1)
    M[np.arange(n), np.arange(n), 0] += 40.0
    return M, random_expansions(n, nrhs, nc, 2, -1, 1), np.arange(1, n + 1, dtype=np.int32)


@pytest.mark.parametrize("nrhs", [1, 20])
def test_solve_with_host_arrays(h, nrhs):
    n = 70
    M, B, piv = _system(n, nrhs)
    LU, X = ozlu.to_colmajor(M), ozlu.to_colmajor(B)
    ozlu.ozlu_debug_wait_limit(h, 5000)
    with pytest.raises(ozlu.OzluError) as e:
        ozlu.ozlu_getrs(h, 2, 0, n, nrhs, LU, n, piv, X, n)
    assert e.value.code == ozlu.OZLU_ERR_TIMEOUT
    ozlu.ozlu_debug_wait_limit(h, 0)
    ozlu.ozlu_getrs(h, 2, 0, n, nrhs, LU, n, piv, ozlu.to_colmajor(B), n)
    assert _word(h) == 0


@pytest.mark.parametrize("graph", [0, 1])
def test_solve_on_the_device(h, graph):
    n = 70
    M, B, piv = _system(n, 2)
    LU, X, p = dev(M), dev(B), torch.from_numpy(piv).cuda()
    opts = ozlu.make_opts("int8", graph=graph)
    for limit in (5000, 0):
        ozlu.ozlu_debug_wait_limit(h, limit)
        ozlu.ozlu_getrs(h, 2, 0, n, 2, LU, n, p, X, n, opts)
        assert _word(h) == (ozlu.OZLU_ERR_TIMEOUT if limit else 0)


def test_batch_keeps_the_word_of_every_instance(h):
    # 40 instances on 32 streams: the last one of a stream does not wipe the first's
    ns = [40] * 40
    M, B, piv = _system(40, 1)
    lus, xs, ps = [dev(M) for _ in ns], [dev(B) for _ in ns], [torch.from_numpy(piv).cuda() for _ in ns]
    for limit in (5000, 0):
        ozlu.ozlu_debug_wait_limit(h, limit)
        ozlu.ozlu_getrs_batched(h, 2, 0, ns, 1, lus, ns, ps, xs, ns)
        assert _word(h) == (ozlu.OZLU_ERR_TIMEOUT if limit else 0)
    # a later product on the handle itself has a word of its own
    ozlu.ozlu_debug_wait_limit(h, 5000)
    ozlu.ozlu_getrs_batched(h, 2, 0, ns, 1, lus, ns, ps, xs, ns)
    ozlu.ozlu_debug_wait_limit(h, 0)
    C = torch.zeros((40, 40, 2), dtype=torch.float64, device="cuda")
    ozlu.ozlu_gemm(h, 2, 0, 40, 40, 40, 1, lus[0], 40, lus[1], 40, 0, C, 40)
    assert _word(h) == 0


def test_p_bit_calls(h):
    n, L, p = 48, 4, 128
    A, X, C = ozlu.MPMatrix(n, n, L), ozlu.MPMatrix(n, 20, L), ozlu.MPMatrix(n, n, L)
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    for Z in (A, X):
        v = torch.randint(0, 1 << 31, Z.limbs.shape, device="cuda", generator=g)
        v[L - 1] -= 1 << 31
        Z.limbs.copy_(v.to(torch.int32))
    piv = torch.zeros(n, dtype=torch.int32, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    for limit in (1000, 0):
        ozlu.ozlu_debug_wait_limit(h, limit)
        calls = (lambda: ozlu.ozlu_mp_getrf(h, p, n, A.desc(), piv, 0, info),
                 lambda: ozlu.ozlu_mp_getrs(h, p, n, 20, A.desc(), piv, X.desc()))
        for call in calls:
            if limit:
                with pytest.raises(ozlu.OzluError) as e:
                    call()
                assert e.value.code == ozlu.OZLU_ERR_TIMEOUT
            else:
                call()
            assert _word(h) == (ozlu.OZLU_ERR_TIMEOUT if limit else 0)
        ozlu.ozlu_mp_gemm(h, p, n, n, n, 1, A.desc(), A.desc(), 0, C.desc())
        assert _word(h) == (ozlu.OZLU_ERR_TIMEOUT if limit else 0)
