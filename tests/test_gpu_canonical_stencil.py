"""The stencil on canonical vectors (amg_apply_D, amg_apply_Dsap on aligned
vectors) against the general path through the internal layout, which overlapping
or unaligned vectors take: the same arithmetic per site, so bitwise equal in FP32
and FP16; FP64 to 1e-14 (another kernel body may contract multiply-adds
differently: a few roundings of 1e-16 in a sum of about 200 terms).

Lattices: fewer sites than a warp, a ragged last warp, extents of two and three,
more sites than one launch has threads for in one stretch."""
import numpy as np
import pytest

import lqcd_inputs as li
from gpu_util import Field

pytestmark = pytest.mark.gpu

DIMS = [(2, 2, 2, 2), (3, 3, 5, 7), (4, 4, 4, 4), (8, 6, 10, 12)]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_canonical_stencil_equals_the_general_path(dims, prec, nrhs):
    import torch
    f = Field(dims, 0.6, 9, 0.127, 1.0)
    try:
        dt = torch.float64 if prec == 0 else torch.float32
        n = nrhs * f.V * 24
        gen = torch.Generator(device="cuda").manual_seed(3)
        x = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen).to(dt)
        pad = torch.zeros(n + 4, dtype=dt, device="cuda")
        unaligned = pad[1:1 + n]
        unaligned.copy_(x)
        blocks = [None]
        if all(d % 2 == 0 and d > 2 for d in dims):
            blocks.append((2, 2, 2, 2))
        for block in blocks:
            def apply(inp, out):
                if block is None:
                    f.c.amg_apply_D(f.d, inp, out, nrhs, prec)
                else:
                    f.c.amg_apply_Dsap(f.d, block, inp, out, nrhs, prec)
            y = torch.empty_like(x)
            ref = torch.empty_like(x)
            same = x.clone()
            apply(x, y)
            apply(unaligned, ref)
            apply(same, same)                 # overlapping: through the work fields
            if prec == 0:
                assert float((y - ref).norm() / ref.norm()) < 1e-14
                assert float((same - ref).norm() / ref.norm()) < 1e-14
            else:
                assert torch.equal(y, ref)
                assert torch.equal(same, ref)
    finally:
        f.close()
