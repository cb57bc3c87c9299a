"""A training step on targets that do not start on a 16-byte boundary: the loss and the
weights of the aligned step, bit for bit, and no device memory for a copy of the batch."""
import numpy as np
import pytest

from gpu_util import Field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_unaligned_targets(offset):
    import torch
    dims, npairs, channels = (8, 8, 8, 8), 64, [1, 2, 1]
    f = Field(dims, 0.5, 6, 0.126, 1.0)
    c = f.c
    w = (0.1 * np.random.default_rng(3).normal(size=sum(c.nn_weight_sizes(channels)))).astype(np.float32)
    n = npairs * f.V * 24   # 25 MB
    gen = torch.Generator(device="cuda").manual_seed(5)
    r, e = torch.randn(n, device="cuda", generator=gen), torch.randn(n, device="cuda", generator=gen)
    u = torch.empty(n + 4, device="cuda")[offset:offset + n]
    u.copy_(e)
    got = []
    try:
        for target in (e, u):
            nn = c.amg_nn_create(f.d, channels, w)
            c.amg_nn_train_step(nn, r, e, 1, 1e-3)
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            loss = c.amg_nn_train_step(nn, r, target, npairs, 1e-3)
            assert free - torch.cuda.mem_get_info()[0] < 2 * n   # half of the batch's bytes
            got.append((loss, c.amg_nn_get_weights(nn, channels, effective=False)))
            c.amg_nn_destroy(nn)
        assert got[0][0] == got[1][0]
        assert np.array_equal(got[0][1], got[1][1])
    finally:
        f.close()
