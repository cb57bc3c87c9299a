"""A ragged batch of more problems than a quarter of the SMs: its coarse solves run as one
thread-block cluster per problem until the easy half of the problems has converged, then
on shares of all SMs, on the same barrier words and partial sums.  Every problem reaches
the FP64 tolerance (re-checked with the oracle's D) and agrees with its own solve to 1e-8,
the bound of the other ragged batches; for both storages of the coarse operator."""
import numpy as np
import pytest

import lqcd_inputs as li
from oracle import dirac as odirac
from gpu_util import Field, to_dev, from_dev, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coarse", ["AMG_F32", "AMG_BF16"])
def test_batch_of_more_problems_than_a_quarter_of_the_sms(coarse):
    import torch
    dims, nvec = (4, 4, 4, 4), 8
    limit = torch.cuda.get_device_properties(0).multi_processor_count // 4
    n = limit + 4
    easy, hard = Field(dims, 0.3, 1, 0.06, 1.0), Field(dims, 0.6, 2, 0.130, 1.0)
    c = easy.c
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = 2
    p.nvec[0] = nvec
    p.prec_coarsest = getattr(c, coarse)
    fs, hs = [easy if i % 2 else hard for i in range(n)], []
    ops = {f: odirac.WilsonClover(f.U, f.kappa, 1.0, True) for f in (easy, hard)}
    try:
        for i, f in enumerate(fs):
            hs.append(c.amg_setup_from_vectors(f.d, p, [li.to_interleaved(li.test_vectors(dims, 20 + i, nvec))]))
        bs = [li.rhs(dims, 200 + i) for i in range(n)]
        bd = [to_dev(b) for b in bs]
        xs = [torch.zeros_like(b) for b in bd]
        st, infos = c.amg_solve_ragged(hs, bd, xs, 1e-10, 300)
        shape = easy.shape4 + (12,)
        for f, h, b, d, x, info in zip(fs, hs, bs, bd, xs, infos):
            assert info.converged == 1 and info.true_rel_residual <= 1e-10
            r = b.reshape(shape) - ops[f].apply(from_dev(x, shape))
            assert np.linalg.norm(r) / np.linalg.norm(b) <= 1.05e-10
            x1 = torch.zeros_like(x)
            c.amg_solve(h, d, x1, 1, 1e-10, 300)
            assert rel(from_dev(x, shape), from_dev(x1, shape)) < 1e-8
        # the problems left when the easy ones are done are few enough for the other form
        assert max(infos[i].iters for i in range(1, n, 2)) < min(infos[i].iters for i in range(0, n, 2))
    finally:
        for h in hs:
            c.amg_hierarchy_destroy(h)
        easy.close()
        hard.close()
