"""The Householder panels of the refresh (bf16 weights at r = 4 and 8, and panels shorter than 4r)
at the edges of warps, of a block's rows and of the column groups a step passes over."""

import numpy as np
import pytest
import torch

from gpu_util import snapshot
from oracle import haar
from parity import UV_ABS

pytestmark = pytest.mark.gpu

SHAPES = {
    4: [(4, 31), (33, 255), (257, 4095), (4096, 4097)],
    8: [(8, 31), (33, 255), (257, 2047), (2048, 2049)],
    16: [(16, 31), (32, 33), (62, 63)],
    32: [(32, 63), (64, 65), (97, 127)],
    64: [(64, 127), (128, 129), (160, 255)],
    128: [(128, 255), (256, 257), (288, 511)],
}


@pytest.mark.parametrize("r", sorted(SHAPES))
def test_householder_panels_match_oracle(lib, gpu, r):
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    seed, base, j = 290 + r, 2, 1
    weights = [torch.zeros(m, (n + 7) // 8 * 8, dtype=torch.bfloat16, device=gpu)[:, :n]
               for m, n in SHAPES[r]]
    z = SubZeroPlus(weights, r, 2, seed, matrix_index_base=base)
    z.refresh(j)
    z.sync()
    s = snapshot(z)
    for i, (m, n) in enumerate(SHAPES[r]):
        U, V = haar.haar_proj(seed, base + i, j, m, n, r)
        for got, want, rows in ((s["U"][i], U, m), (s["V"][i], V, n)):
            assert np.max(np.abs(got.T @ got - np.eye(r))) <= 1e-5, (r, rows)
            # fp32's error grows with the panel's condition number: about 6 at 2r rows; nearly
            # square panels (where it is unbounded) are held to their span below
            if rows >= 2 * r - 2:
                assert np.max(np.abs(got - want)) <= UV_ABS, (r, rows)
            # the same span and signs: Q^T Q_oracle is the identity up to error x condition
            # number, which for a square Gaussian panel is below about 100 r
            assert np.max(np.abs(got.T @ want - np.eye(r))) <= 100 * r * 2.0 ** -22, (r, rows)
    z.close()
