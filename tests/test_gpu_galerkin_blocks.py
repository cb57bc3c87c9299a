"""The coarse operator (Eq. 7) on blocks whose face tile and partial sums do not fit the
48 KB of shared memory that a launch gets unasked: an extent of two (half of the block
is one face), and FP64 blocks of many vectors.  Each hierarchy is built from given
vectors; its operator, applied to random coarse vectors, is P^dag D P for the vectors it
holds.

Bounds, relative L2: FP64 1e-12 and FP32 2e-6, those of the same comparison on other
blocks (the sums are over at most 512 sites here)."""
import numpy as np
import pytest

import lqcd_inputs as li
from oracle import dirac as odirac, multigrid as omg
from gpu_util import Field, rel

pytestmark = pytest.mark.gpu

CASES = [
    # precision of the vectors, block, vectors; shared memory of the launch
    (0, (2, 4, 4, 8), 3),     # 50 KB: the face tile alone fills 48 KB
    (0, (8, 4, 4, 2), 4),     # 50 KB, the face in the slowest direction
    (0, (4, 4, 4, 4), 49),    # 48.5 KB: the partial sums go past it
    (1, (8, 8, 4, 2), 3),     # 49.5 KB
    (1, (2, 6, 6, 6), 15),    # 54.7 KB, 216 face sites in 224 threads
    (1, (2, 2, 2, 2), 3),     # smallest block: one group of threads, no face tile
]


@pytest.mark.parametrize("prec,block,nvec", CASES)
def test_galerkin_operator_on_any_block(prec, block, nvec):
    dims = tuple(2 * b for b in block)
    f = Field(dims, 0.6, 3, 0.130, 1.0)
    c = f.c
    p = c.amg_params_default()
    for mu in range(4):
        p.block[0][mu] = block[mu]
    p.nvec[0] = nvec
    p.prec_smoother = p.prec_coarsest = prec
    h = None
    try:
        h = c.amg_setup_from_vectors(f.d, p, [li.to_interleaved(li.test_vectors(dims, 3, nvec))])
        got = c.amg_get_vectors(h, 0, nvec, f.V)
        v = (got[..., 0] + 1j * got[..., 1]).reshape((nvec,) + f.shape4 + (12,))
        B = c.amg_get_coarse_op(h, 1)
        B = B[..., 0] + 1j * B[..., 1]
        op = odirac.WilsonClover(f.U, 0.130, 1.0, True)
        got = omg.CoarseStencil(B.reshape((2, 2, 2, 2, 9, 2 * nvec, 2 * nvec)), nvec)
        for k in range(2):
            x = li.complex_normal(60 + k, li.STREAM_MISC, (2, 2, 2, 2, 2 * nvec))
            ref = omg.restrict(v, op.apply(omg.prolong(v, x, block)), block)
            assert rel(got.apply(x), ref) < (1e-12 if prec == 0 else 2e-6)
    finally:
        if h is not None:
            c.amg_hierarchy_destroy(h)
        f.close()
