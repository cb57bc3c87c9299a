"""Inputs far from unit scale: the sums that are kept as pairs of floats scale
their operands by powers of two, which is exact, so vectors of any FP32 scale give
the same results as unit ones.

FP32 test vectors times 2^60 and 2^-60 orthonormalise to the same bits (the scale
drops out exactly)."""
import numpy as np
import pytest

import lqcd_inputs as li
from gpu_util import Field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,block", [((4, 4, 4, 8), (2, 2, 2, 4)), ((6, 6, 6, 6), (3, 3, 3, 3))])
@pytest.mark.parametrize("exponent", [60, -60])
def test_orthonormal_vectors_do_not_depend_on_the_scale(dims, block, exponent):
    f = Field(dims, 0.6, 5, 0.130, 1.0)
    c = f.c
    nvec = 5   # odd: the last projection of a pair of vectors has one
    try:
        p = c.amg_params_default()
        for mu in range(4):
            p.block[0][mu] = block[mu]
        p.nvec[0] = nvec
        p.nlevels, p.prec_smoother, p.prec_coarsest = 2, 1, 1
        v0 = np.asarray(li.to_interleaved(li.test_vectors(dims, 5, nvec)))
        got = []
        for scale in (1.0, 2.0 ** exponent):
            h = c.amg_setup_from_vectors(f.d, p, [v0 * scale])
            got.append(c.amg_get_vectors(h, 0, nvec, f.V))
            c.amg_hierarchy_destroy(h)
        assert np.array_equal(got[0], got[1])
    finally:
        f.close()
