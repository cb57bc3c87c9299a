"""The stencil on canonical vectors with more sites than one launch has threads for
(65,535 CTAs of 128), so that CTAs take a second stretch: bitwise equal to the general
path, which unaligned vectors take."""
import pytest

from gpu_util import capi

pytestmark = pytest.mark.gpu


def test_more_sites_than_threads():
    import torch
    c = capi()
    dims = (64, 64, 64, 33)
    V = 64 ** 3 * 33
    assert V > 65535 * 128
    lat = c.amg_lattice_create(dims, True)
    g = c.amg_gauge_random(lat, 0.5, 3)
    d = c.amg_dirac_create(g, 0.128, 1.0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(3)
        x = torch.randn(V * 24, device="cuda", generator=gen)
        pad = torch.empty(V * 24 + 4, device="cuda")
        u = pad[1:1 + V * 24]
        u.copy_(x)
        y, ref = torch.empty_like(x), torch.empty_like(x)
        c.amg_apply_D(d, x, y, 1, c.AMG_F32)
        c.amg_apply_D(d, u, ref, 1, c.AMG_F32)
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
    finally:
        torch.cuda.synchronize()
        c.amg_dirac_destroy(d)
        c.amg_gauge_destroy(g)
        c.amg_lattice_destroy(lat)
