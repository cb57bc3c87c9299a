"""The sums of squares behind the loss of a training step carry FP64.

The network is the identity (spin matrix 1 on the site itself), the residual lives on the
odd components and the error on the even ones, so y - e is formed without rounding and
|y - e|^2 = |r|^2 + |e|^2.  One site of the lattice is not zero.  Its values are integers
below 2^24 times one power of two: FP64 holds every partial sum of the 24 squares (48
bits and at most 2^4.6 of them), so the loss is the exact ratio, rounded once; sums kept
to 48 bits lose the last bits of it.  With values on all sites the sums round in FP64:
at most 60 roundings of 2^-53 on each side of the ratio and one in it, 1.4e-14."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_util import Field

pytestmark = pytest.mark.gpu

# values of unit scale; of the ranges that are scaled before they are squared; across their edge
EXPONENTS = [-24, -68, -61, 44]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 2, 5, 7), (6, 6, 6, 20)])   # half a warp .. several CTAs
@pytest.mark.parametrize("exponent", EXPONENTS)
def test_loss_is_the_exact_ratio(dims, exponent):
    import torch
    f = Field(dims, 0.5, 6, 0.126, 1.0)
    c = f.c
    w = np.zeros((9, 4, 4, 2), np.float32)
    w[0, :, :, 0] = np.eye(4)
    try:
        for seed in range(8):
            rng = np.random.default_rng(seed)
            for one in (True, False):
                ir, ie = rng.integers(-2 ** 24 + 1, 2 ** 24, size=(2, f.V, 24))
                ir[:, ::2] = 0
                ie[:, 1::2] = 0
                if one:
                    at = rng.integers(f.V)
                    ir[np.arange(f.V) != at] = 0
                    ie[np.arange(f.V) != at] = 0
                nn = c.amg_nn_create(f.d, [1, 1], w.reshape(-1))
                r, e = (torch.from_numpy((v * 2.0 ** exponent).astype(np.float32).reshape(-1)).cuda()
                        for v in (ir, ie))
                loss = c.amg_nn_train_step(nn, r, e, 1, 1e-3)
                c.amg_nn_destroy(nn)
                rr, ee = (sum(int(v) ** 2 for v in t.reshape(-1)) for t in (ir, ie))
                exact = float(Fraction(rr + ee, ee))
                assert loss == exact if one else abs(loss - exact) <= 1.4e-14 * exact
    finally:
        f.close()
