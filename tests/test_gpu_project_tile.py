"""The FMA path's projection P = C V^T at r = 16 ... 128 at the edges of its 128-column tiles and
of a warp's 32 columns, through a perturbation of a zero fp32 weight: W = U (C V^T)."""

import numpy as np
import pytest
import torch

from gpu_util import f32, snapshot
from oracle import subzero

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [16, 32, 64, 128])
def test_projection_tile_edges(lib, gpu, r):
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    widths = [n for n in (16, 31, 33, 95, 97, 127, 128, 129, 160, 257) if n >= r]
    seed, t, eps = 31, 4, f32(0.5)
    weights = [torch.zeros(r + 1, (n + 3) // 4 * 4, device=gpu)[:, :n] for n in widths]
    z = SubZeroPlus(weights, r, 2, seed)
    zb.zo_set_option(z.ctx, zb.ZO_OPTION_WPASS_PATH, 1)
    z.init_subspace(0)
    z.perturb(t, 1, 1.0, -1, 0.0, eps)
    z.sync()
    s = snapshot(z)
    for i, n in enumerate(widths):
        U, V = s["U"][i].astype(np.float64), s["V"][i].astype(np.float64)
        C = subzero.perturb_coeff(seed, i, t, r, [(1, 1.0)], eps)
        want = U @ C @ V.T
        # two chains of r multiply-adds, C's own rounding and its draws' (a few 2^-22 of |Z| + 1)
        scale = np.abs(U) @ (np.abs(C) + eps) @ np.abs(V).T
        assert np.all(np.abs(s["W"][i] - want) <= (2 * r + 16) * 2.0 ** -24 * scale), (r, n)
    z.close()
