"""Restriction and prolongation have finished when the call returns, on every path: the
stream they ran on, busy with earlier stencil applications until then, is idle."""
import pytest

import lqcd_inputs as li
from gpu_util import Field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,offset", [(1, 0), (1, 1), (0, 0)])   # direct; through the scratch field; FP64
def test_transfers_return_with_the_result(prec, offset):
    import torch
    dims, nvec = (8, 8, 8, 8), 6
    f = Field(dims, 0.5, 11, 0.126, 1.0)
    c = f.c
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = 4
    p.nvec[0] = nvec
    h = c.amg_setup_from_vectors(f.d, p, [li.to_interleaved(li.test_vectors(dims, 11, nvec))])
    try:
        dt = torch.float64 if prec == 0 else torch.float32
        n, m = f.V * 24, 16 * 2 * nvec * 2
        fine = torch.randn(n + 4, device="cuda", dtype=dt)[offset:offset + n]
        coarse = torch.randn(m, device="cuda", dtype=dt)
        x = torch.randn(f.V * 24, device="cuda", dtype=torch.float64)
        y = torch.empty_like(x)
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        for call in (lambda: c.amg_restrict(h, 0, fine, coarse, 1, prec, st.cuda_stream),
                     lambda: c.amg_prolong(h, 0, coarse, fine, 1, prec, st.cuda_stream)):
            for _ in range(200):   # about 30 us each: milliseconds of work ahead of the call
                c.amg_apply_D(f.d, x, y, 1, c.AMG_F64, st.cuda_stream)
            call()
            assert st.query()
    finally:
        torch.cuda.synchronize()
        c.amg_hierarchy_destroy(h)
        f.close()
