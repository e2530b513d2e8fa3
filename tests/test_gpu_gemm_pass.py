"""The 64 x 128-tile FMA pass at the edges of its tiles: widths and heights one short of, at
and one past a tile (widths not a multiple of 4 copy P word by word), padded rows, the
smallest matrix of each rank, and sets of more matrices than one probe of the tile table."""

import numpy as np
import pytest

from gpu_util import dtype_of, f32, make_weight, oracle_step, snapshot
from parity import assert_weights

pytestmark = pytest.mark.gpu


def _shapes(r):
    edges = [(63, 127), (64, 128), (65, 129), (64, 130), (129, 257), (192, 256)]
    return [(r, r)] + [(m, n) for m, n in edges if min(m, n) >= r]


@pytest.mark.parametrize("r", [4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_tile_edges_match_oracle(lib, gpu, dtype, r):
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    per = 4 if dtype == "f32" else 8
    shapes = _shapes(r) + [(r + 1, r + 3)] * 40          # more than 32 matrices
    weights = [make_weight(m, n, dtype, k, gpu, ldw=(n + per - 1) // per * per + per * (k % 2))
               for k, (m, n) in enumerate(shapes)]
    z = SubZeroPlus(weights, r, 2, 77)
    zb.zo_set_option(z.ctx, zb.ZO_OPTION_WPASS_PATH, 1)
    z.init_subspace(0)
    before = snapshot(z)
    eps, lr = 1e-1, 1e-2
    z.step(1, 1, np.asarray([0.5, -1.5], np.float32), "direct", eps, lr, 0.9, 0.95, 1e-8, 1, 1.0)
    z.sync()
    after = snapshot(z)
    for i, (m, n) in enumerate(shapes[:10] + shapes[-1:]):
        i = i if i < 10 else len(shapes) - 1
        W, M, Vm, G, terms = oracle_step(before, i, dtype_of(weights[i]), 77, i, 1, r, 2,
                                         [0.5, -1.5], "direct", eps, lr, 0.9, 0.95, 1e-8, 1,
                                         [(1, 1.0)])
        assert_weights(after["W"][i], W, dtype_of(weights[i]), f"{m}x{n} r={r}",
                       before=before["W"][i], terms=terms)
    z.close()


def test_tiles_find_their_matrix(lib, gpu):
    """1100 matrices (three probes of the tile table): the set's pass gives the bits of passes
    over its halves."""
    import torch
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    W0 = torch.randn(1100, 20, 24, device=gpu) * 0.02
    whole, halves = W0.clone(), W0.clone()
    for W, parts in ((whole, [(0, 1100)]), (halves, [(0, 500), (500, 1100)])):
        for a, b in parts:
            z = SubZeroPlus(list(W[a:b]), 16, 2, 5, matrix_index_base=a)
            z.init_subspace(0)
            z.perturb(0, 1, 1.0, -1, 0.0, f32(1e-1))
            assert zb.zo_wpass_path(z.ctx) == 1
            z.sync()
            z.close()
    assert torch.equal(whole, halves)
    assert not torch.any(torch.all((whole - W0).flatten(1) == 0, dim=1))
