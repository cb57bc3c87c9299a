"""Weight gradient of a learned layer on enough sites that every warp moves its running
sums on more than once (eight stretches of 32 sites per warp on about 140 CTAs: from
35,000 sites on), prefetches across stretches and ends in a ragged one; with the input
transported (1 -> 4 channels) and with the output gradient transported (4 -> 1).  Against
the oracle to 1e-5 of the whole gradient, as on the small volumes."""
import numpy as np
import pytest

import lqcd_inputs as li
from oracle import ptconv as opt
from gpu_util import Field, rel, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout", [(1, 4), (4, 1)])
def test_weight_gradient_beyond_one_flush(cin, cout):
    dims = (13, 14, 15, 17)   # 46,410 sites, 10 more than whole stretches
    f = Field(dims, 0.5, 6, 0.126, 1.0)
    c = f.c
    channels = [1, 4, 1]
    sizes = c.nn_weight_sizes(channels)
    nn = c.amg_nn_create(f.d, channels, np.zeros(sum(sizes), np.float32))
    try:
        shp = f.shape4 + (4, 3)
        psi = np.stack([li.rhs(dims, 30 + k).reshape(shp) for k in range(cin)])
        g = np.stack([li.rhs(dims, 40 + k).reshape(shp) for k in range(cout)])
        layer = 0 if cin == 1 else 1
        gw = c.amg_nn_layer_backward(nn, layer, to_dev(psi, "float32"), to_dev(g, "float32"), None, True, sizes[layer])
        got = gw.reshape(cout, cin, 9, 4, 4, 2)
        assert rel(got[..., 0] + 1j * got[..., 1], opt.weight_grad(f.U, psi, g)) < 1e-5
    finally:
        c.amg_nn_destroy(nn)
        f.close()
