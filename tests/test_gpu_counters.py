"""The byte counters of ozlu_stats name what a product's phases move: the residues
as they are stored (two bytes in binary16, three planes of base-17 digits) and the t
values (a byte each, or a 32-bit word per three moduli)."""
import pytest

from synth import random_expansions

from gpu_util import dev, handle, ozlu, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("backend,per,kstep", [("int8", 2, 64), ("fp16", 2, 64), ("fp8", 3, 128)])
@pytest.mark.parametrize("m,n,k", [(130, 70, 100), (1500, 1400, 40)])
def test_bytes_of_a_product(backend, per, kstep, m, n, k):
    handle()
    up = lambda v, q: -(-v // q) * q
    h = ozlu.ozlu_create(None)
    try:
        A, B = dev(random_expansions(m, k, 2, 1, -1, 1)), dev(random_expansions(k, n, 2, 2, -1, 1))
        C = torch.zeros((n, m, 2), dtype=torch.float64, device="cuda")
        ozlu.ozlu_set_timing(h, 0)
        opts = ozlu.make_opts(backend)
        ozlu.ozlu_gemm(h, 2, 0, m, n, k, 1, A, m, B, k, 0, C, m, opts)
        torch.cuda.synchronize()
        st, i = ozlu.ozlu_get_stats(h), ozlu.ozlu_plan(106, k, opts)
        planes = i.n_mod * i.S * (up(m, 128) + up(n, 128)) * up(k, kstep) * per
        assert st.convert_bytes == 16 * (m * k + k * n) + planes
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        words = -(-i.n_mod // 3)
        packed = up(m, 128) // 128 * (up(n, 128) // 128) * words * i.n_groups >= 4 * sms
        assert st.crt_bytes == m * n * (i.n_groups * (4 * words if packed else i.n_mod) + 16)
    finally:
        ozlu.ozlu_destroy(h)
