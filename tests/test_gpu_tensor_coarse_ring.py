"""Tensor-core coarse stencil with many sites per CTA: the ring of shared-memory stages
wraps (more than eight sites per CTA, the most stages there are), both accumulators are
handed back and refilled, and the last lap is ragged.  One piece per site (Nc 16, 48) and
three (Nc 64); accumulator columns for up to 8 and for up to 16 right-hand sides.

Against the SIMT stencil of the same bfloat16 operator on the same bfloat16-rounded
vectors: both accumulate in FP32, relative L2 <= 1e-5 as in the oracle's comparison."""
import pytest

import lqcd_inputs as li
from gpu_util import capi

pytestmark = pytest.mark.gpu

CDIMS = (6, 8, 4, 8)   # 1536 coarse sites of 2^4


@pytest.mark.parametrize("nvec", [8, 24, 32])
def test_ring_of_stages_wraps(nvec):
    import torch
    c = capi()
    dims = tuple(2 * n for n in CDIMS)
    assert 1536 > 8 * torch.cuda.get_device_properties(0).multi_processor_count
    n = 12 * dims[0] * dims[1] * dims[2] * dims[3]
    lat = c.amg_lattice_create(dims, True)
    g = c.amg_gauge_random(lat, 0.5, 3)
    d = c.amg_dirac_create(g, 0.128, 1.0)
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = 2
    p.nvec[0] = nvec
    p.prec_coarsest = c.AMG_BF16
    v = torch.empty(nvec * n * 2, dtype=torch.float64, device="cuda")
    c.amg_random_normal(7, li.STREAM_TESTVEC, 0, nvec * n, v)
    torch.cuda.synchronize()
    h = c.amg_setup_from_vectors(d, p, [v])
    try:
        m = 1536 * 2 * nvec * 2
        gen = torch.Generator(device="cuda").manual_seed(nvec)
        for nrhs in (5, 16):
            x = torch.randn(nrhs, m, device="cuda", generator=gen).bfloat16().float()
            y, ref = torch.empty_like(x), torch.empty_like(x)
            c.amg_apply_coarse(h, 1, x, y, nrhs, c.AMG_BF16)
            c.amg_apply_coarse(h, 1, x, ref, nrhs, c.AMG_F32)
            torch.cuda.synchronize()
            for r in range(nrhs):
                assert float((y[r] - ref[r]).norm() / ref[r].norm()) < 1e-5
    finally:
        c.amg_hierarchy_destroy(h)
        c.amg_dirac_destroy(d)
        c.amg_gauge_destroy(g)
        c.amg_lattice_destroy(lat)
