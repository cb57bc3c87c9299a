"""Restriction and prolongation of batches (several right-hand sides per CTA, on the
caller's canonical FP32 vectors) against the same calls one vector at a time and
against the general path through the internal layout, which unaligned vectors take.
Every right-hand side goes through the same sums in the same order, so all of them are
bitwise equal.  Batches that fill a group of four, leave a rest, and split unevenly;
blocks of 16, 81, 256 and 320 sites (the last beyond the batched kernel's range);
vector counts that are no multiple of the vectors in flight."""
import pytest

import lqcd_inputs as li
from gpu_util import Field

pytestmark = pytest.mark.gpu

CASES = [((4, 4, 4, 4), (2, 2, 2, 2), 5), ((6, 6, 6, 6), (3, 3, 3, 3), 7), ((8, 8, 8, 8), (4, 4, 4, 4), 6),
         ((8, 8, 8, 10), (4, 4, 4, 5), 3)]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("half", [False, True])
def test_batches_equal_single_calls(case, half):
    import torch
    dims, block, nvec = CASES[case]
    f = Field(dims, 0.5, 11, 0.126, 1.0)
    c = f.c
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = block[mu]
    p.nvec[0] = nvec
    if half:
        p.prec_vectors = c.AMG_F16
    h = c.amg_setup_from_vectors(f.d, p, [li.to_interleaved(li.test_vectors(dims, 11, nvec))])
    try:
        n, m = f.V * 24, 1
        for mu in range(4):
            m *= dims[mu] // block[mu]
        m *= 2 * nvec * 2
        gen = torch.Generator(device="cuda").manual_seed(2)
        for nrhs in (1, 2, 3, 4, 5, 6, 9):
            fine = torch.randn(nrhs * n, device="cuda", generator=gen)
            coarse = torch.randn(nrhs * m, device="cuda", generator=gen)
            oc, of = torch.empty_like(coarse), torch.empty_like(fine)
            c.amg_restrict(h, 0, fine, oc, nrhs, c.AMG_F32)
            c.amg_prolong(h, 0, coarse, of, nrhs, c.AMG_F32)
            for q in range(nrhs):
                a, b = torch.empty(m, device="cuda"), torch.empty(n, device="cuda")
                c.amg_restrict(h, 0, fine[q * n:(q + 1) * n].clone(), a, 1, c.AMG_F32)
                c.amg_prolong(h, 0, coarse[q * m:(q + 1) * m].clone(), b, 1, c.AMG_F32)
                assert torch.equal(oc[q * m:(q + 1) * m], a)
                assert torch.equal(of[q * n:(q + 1) * n], b)
            pad = torch.empty(nrhs * n + 4, device="cuda")
            u = pad[1:1 + nrhs * n]
            u.copy_(fine)
            gc = torch.empty_like(oc)
            c.amg_restrict(h, 0, u, gc, nrhs, c.AMG_F32)
            assert torch.equal(gc, oc)
            c.amg_prolong(h, 0, coarse, u, nrhs, c.AMG_F32)
            assert torch.equal(u, of)
    finally:
        c.amg_hierarchy_destroy(h)
        f.close()
