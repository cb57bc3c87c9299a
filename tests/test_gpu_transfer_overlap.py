"""Restriction and prolongation of FP32 vectors that share memory: the coarse vectors
inside the fine ones, across their end, and directly behind them.  The result is the one
of separate vectors, bit for bit (both routes take every sum in the same order)."""
import pytest

import lqcd_inputs as li
from gpu_util import Field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 3])
def test_overlapping_transfer_vectors(nrhs):
    import torch
    dims, nvec = (8, 8, 8, 8), 6
    f = Field(dims, 0.5, 11, 0.126, 1.0)
    c = f.c
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = 2
    p.nvec[0] = nvec
    h = c.amg_setup_from_vectors(f.d, p, [li.to_interleaved(li.test_vectors(dims, 11, nvec))])
    try:
        n, m = nrhs * f.V * 24, nrhs * (f.V // 16) * 2 * nvec * 2
        gen = torch.Generator(device="cuda").manual_seed(4)
        src_f = torch.randn(n, device="cuda", generator=gen)
        src_c = torch.randn(m, device="cuda", generator=gen)
        ref_c, ref_f = torch.empty_like(src_c), torch.empty_like(src_f)
        c.amg_restrict(h, 0, src_f, ref_c, nrhs, c.AMG_F32)
        c.amg_prolong(h, 0, src_c, ref_f, nrhs, c.AMG_F32)
        # start of the fine vector and of the coarse one in a shared buffer (multiples of two floats)
        for at_f, at_c in ((0, 0), (0, 2), (0, n // 2), (0, n - 2), (m, 0), (m - 4, 0), (0, n)):
            buf = torch.empty(n + m + 4, device="cuda")
            fine, coarse = buf[at_f:at_f + n], buf[at_c:at_c + m]
            fine.copy_(src_f)
            c.amg_restrict(h, 0, fine, coarse, nrhs, c.AMG_F32)
            assert torch.equal(coarse, ref_c)
            coarse.copy_(src_c)
            c.amg_prolong(h, 0, coarse, fine, nrhs, c.AMG_F32)
            assert torch.equal(fine, ref_f)
    finally:
        c.amg_hierarchy_destroy(h)
        f.close()
