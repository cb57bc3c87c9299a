"""Layers of every channel pair of the learned preconditioner (1..4 in, 1..4 out: the
layer transports whichever side has fewer channels, forwards and in the weight
gradient) against the oracle with the same bfloat16 weights.  Volumes below one warp,
with a ragged last warp, and beyond one flush of the gradient's running sums.

Bounds: FP32 arithmetic on sums of at most 9 x 4 x 4 spin terms per value, 1e-5 as in
the other learned-layer tests; the weight gradient sums those over the lattice with
the partial sums kept to 48 bits, so the same bound relative to the whole gradient."""
import numpy as np
import pytest

import lqcd_inputs as li
from oracle import ptconv as opt
from gpu_util import Field, bf16_round, from_dev, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 2, 5, 7), (4, 4, 6, 8)])
@pytest.mark.parametrize("cin", [1, 2, 3, 4])
@pytest.mark.parametrize("cout", [1, 2, 3, 4])
def test_layer_forward_and_backward_on_every_channel_pair(dims, cin, cout):
    import torch
    f = Field(dims, 0.5, 6, 0.126, 1.0)
    c = f.c
    # the layer under test between two that make it a network from one field to one field
    channels = [1, cin, cout, 1]
    rng = np.random.default_rng(100 * cin + cout)
    w = rng.normal(size=sum(c.nn_weight_sizes(channels))).astype(np.float32)
    sizes = c.nn_weight_sizes(channels)
    nn = c.amg_nn_create(f.d, channels, w)
    try:
        W = bf16_round(w[sizes[0]:sizes[0] + sizes[1]]).reshape(cout, cin, 9, 4, 4, 2)
        W = W[..., 0] + 1j * W[..., 1]
        shp = f.shape4 + (4, 3)
        psi = np.stack([li.rhs(f.dims, 30 + k).reshape(shp) for k in range(cin)])
        g = np.stack([li.rhs(f.dims, 40 + k).reshape(shp) for k in range(cout)])
        x, gd = to_dev(psi, "float32"), to_dev(g, "float32")
        out = torch.empty(cout * f.V * 24, dtype=torch.float32, device="cuda")
        gin = torch.empty(cin * f.V * 24, dtype=torch.float32, device="cuda")
        c.amg_nn_layer_forward(nn, 1, x, out)
        assert rel(from_dev(out, (cout,) + shp), opt.layer(f.U, W, psi)) < 1e-5
        gw = c.amg_nn_layer_backward(nn, 1, x, gd, gin, True, sizes[1])
        assert rel(from_dev(gin, (cin,) + shp), opt.layer_adjoint(f.U, W, g)) < 1e-5
        got = gw.reshape(cout, cin, 9, 4, 4, 2)
        assert rel(got[..., 0] + 1j * got[..., 1], opt.weight_grad(f.U, psi, g)) < 1e-5
    finally:
        c.amg_nn_destroy(nn)
        f.close()
