"""Inputs far from unit scale: the sums that are kept as pairs of floats scale
their operands by powers of two, which is exact, so vectors of any FP32 scale give
the same results as unit ones.

FP32 test vectors times 2^60 and 2^-60 orthonormalise to the same bits (the scale
drops out exactly).  A training step on (r, e) times 2^60 and 2^-70 has the same
relative loss: the squares are then summed in FP64 instead of pairs of 48 bits,
1e-12; the second step's loss depends on the first's gradient, which would be zero
if its products had left the range."""
import numpy as np
import pytest

import lqcd_inputs as li
from gpu_util import Field, to_dev

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


@pytest.mark.parametrize("channels", [[1, 1], [1, 4, 1]])
@pytest.mark.parametrize("exponent", [60, -70])
def test_training_step_does_not_depend_on_the_scale(channels, exponent):
    dims = (3, 2, 5, 7)
    f = Field(dims, 0.5, 6, 0.126, 1.0)
    c = f.c
    rng = np.random.default_rng(7)
    w = (0.1 * rng.normal(size=sum(c.nn_weight_sizes(channels)))).astype(np.float32)
    r = np.stack([li.rhs(dims, 30 + k) for k in range(2)])
    e = np.stack([li.rhs(dims, 40 + k) for k in range(2)])
    losses = []
    try:
        for scale in (1.0, 2.0 ** exponent):
            nn = c.amg_nn_create(f.d, channels, w)
            rd, ed = to_dev(r * scale, "float32"), to_dev(e * scale, "float32")
            losses.append([c.amg_nn_train_step(nn, rd, ed, 2, 1e-2) for _ in range(2)])
            c.amg_nn_destroy(nn)
        assert losses[0][0] != losses[0][1]
        assert np.allclose(losses[0], losses[1], rtol=1e-12, atol=0)
    finally:
        f.close()
