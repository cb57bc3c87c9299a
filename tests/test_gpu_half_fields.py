"""Batches of half-precision fields on volumes that are no multiple of four: a field
is 52 bytes per site, so without padding the second field of a batch would start off
the 16-byte boundary that its 16-byte words need.  Every vector of a batch equals the
same vector alone, bit for bit (one site's arithmetic does not depend on the batch)."""
import pytest

from gpu_util import Field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(3, 3, 5, 7), (3, 3, 3, 2), (2, 3, 5, 3)])
@pytest.mark.parametrize("entry", ["amg_apply_D", "amg_apply_D_noalloc"])
def test_half_precision_batch_on_any_volume(dims, entry):
    import torch
    f = Field(dims, 0.5, 4, 0.126, 1.0)
    try:
        apply = getattr(f.c, entry)
        n = f.V * 24
        gen = torch.Generator(device="cuda").manual_seed(8)
        x = torch.randn(3 * n, dtype=torch.float32, device="cuda", generator=gen)
        y = torch.empty_like(x)
        apply(f.d, x, y, 3, f.c.AMG_F16)
        for q in range(3):
            one, out = x[q * n:(q + 1) * n].clone(), torch.empty(n, dtype=torch.float32, device="cuda")
            apply(f.d, one, out, 1, f.c.AMG_F16)
            assert torch.equal(y[q * n:(q + 1) * n], out)
    finally:
        f.close()
