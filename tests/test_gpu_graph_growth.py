"""A captured call after a larger one on the same handle: the larger call replaces
the workspace whose addresses the graph holds, so the graph is captured again and
the call gives the same bits as before."""
import numpy as np
import pytest

from synth import random_expansions

from gpu_util import dev, host, ozlu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("backend", ["fp16", "int8"])
def test_graph_after_the_workspace_has_grown(backend):
    h = ozlu.ozlu_create(None)
    opts = ozlu.make_opts(backend, graph=1)
    try:
        def case(n, nrhs, seed):
            A0 = dev(random_expansions(n, n, 2, seed, -1, 1))
            X0 = torch.rand((nrhs, n, 2), dtype=torch.float64, device="cuda",
                            generator=torch.Generator("cuda").manual_seed(seed))
            X0[..., 1] = 0
            A, X = torch.empty_like(A0), torch.empty_like(X0)
            piv = torch.zeros(n, dtype=torch.int32, device="cuda")
            info = torch.zeros(1, dtype=torch.int32, device="cuda")

            def run():
                A.copy_(A0)
                X.copy_(X0)
                ozlu.ozlu_getrf(h, 2, 0, n, A, n, piv, 64, info, opts)
                ozlu.ozlu_getrs(h, 2, 0, n, nrhs, A, n, piv, X, n, opts)
                torch.cuda.synchronize()
                assert int(info.item()) == 0
                return host(A, n), X.cpu().numpy(), ozlu.ozlu_get_stats(h).graph_status
            return run

        small = case(150, 1, 1)
        first = [small() for _ in range(3)]
        assert first[-1][2] == 2
        large = case(400, 3, 2)
        again = case(150, 1, 1)
        for _ in range(3):
            large()
        status = []
        for run in (small, small, again):
            got = run()
            status.append(got[2])
            np.testing.assert_array_equal(got[0], first[0][0])
            np.testing.assert_array_equal(got[1], first[0][1])
        assert status[:2] == [1, 2]
    finally:
        ozlu.ozlu_destroy(h)
