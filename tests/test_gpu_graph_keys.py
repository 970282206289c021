"""Captured solves of the same matrices and right-hand sides with other leading
dimensions: each is a call of its own, not a replay of the first one's graph."""
import numpy as np
import pytest

from synth import random_expansions

from gpu_util import handle, ozlu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 20])
@pytest.mark.parametrize("lda,ldb", [(100, 110), (108, 100)])
def test_leading_dimensions_are_part_of_the_graph(nrhs, lda, ldb):
    handle()
    n, nc = 100, 2
    M = random_expansions(108, n, nc, 1, -1, 1)
    M[np.arange(n), np.arange(n), 0] += 40.0
    LU = torch.from_numpy(ozlu.to_colmajor(M)).cuda()       # (n, 108, nc): room for either lda
    B = torch.from_numpy(ozlu.to_colmajor(random_expansions(110, nrhs, nc, 2, -1, 1))).cuda()
    X = torch.empty_like(B)
    piv = torch.arange(1, n + 1, dtype=torch.int32, device="cuda")
    h = ozlu.ozlu_create(None)
    try:
        got = {}
        for graph in (0, 1):
            opts = ozlu.make_opts("int8", graph=graph)
            for la, lb in ((n, n), (lda, ldb), (n, n)):
                for _ in range(3):
                    X.copy_(B)
                    ozlu.ozlu_getrs(h, nc, 0, n, nrhs, LU, la, piv, X, lb, opts)
                    torch.cuda.synchronize()
                    got.setdefault((la, lb), []).append(X.cpu().numpy())
        for runs in got.values():
            for x in runs[1:]:
                np.testing.assert_array_equal(x, runs[0])
        assert not np.array_equal(got[n, n][0], got[lda, ldb][0])
    finally:
        ozlu.ozlu_destroy(h)
