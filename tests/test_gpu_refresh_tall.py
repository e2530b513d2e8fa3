"""The refresh of tall panels (r = 16 ... 128) at the edges of its chunks and stages: the
shortest tall panel, one row less and more than a stage, a chunk and two chunks, and several
panels of different lengths in one context; bit-equal when a panel is refreshed alone."""

import numpy as np
import pytest
import torch

from gpu_util import snapshot
from oracle import haar
from parity import UV_ABS

pytestmark = pytest.mark.gpu

SHAPES = {
    16: [(64, 65), (127, 129), (1023, 1025), (2047, 2049)],
    32: [(128, 129), (255, 257), (1023, 1025), (2047, 2049)],
    64: [(256, 257), (1023, 1025), (2047, 2049)],
    128: [(512, 513), (1023, 1025), (2047, 2049)],
}


@pytest.mark.parametrize("r", [16, 32, 64, 128])
def test_tall_panels_match_oracle(lib, gpu, r):
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    seed, base, j = 190 + r, 5, 2
    weights = [torch.zeros(m, (n + 7) // 8 * 8, dtype=torch.bfloat16, device=gpu)[:, :n]
               for m, n in SHAPES[r]]
    z = SubZeroPlus(weights, r, 2, seed, matrix_index_base=base)
    z.refresh(j)
    z.sync()
    s = snapshot(z)
    for i, (m, n) in enumerate(SHAPES[r]):
        U, V = haar.haar_proj(seed, base + i, j, m, n, r)
        for got, want in ((s["U"][i], U), (s["V"][i], V)):
            # panels of at least 4r rows: the condition number is at most about 3
            assert np.max(np.abs(got - want)) <= UV_ABS, (r, got.shape)
            assert np.max(np.abs(got.T @ got - np.eye(r))) <= 1e-5
    z.close()
    one = SubZeroPlus(weights[1:2], r, 2, seed, matrix_index_base=base + 1)
    one.refresh(j)
    one.sync()
    s1 = snapshot(one)
    assert np.array_equal(s1["U"][0], s["U"][1]) and np.array_equal(s1["V"][0], s["V"][1])
    one.close()


@pytest.mark.parametrize("r", [16, 32, 64, 128])
def test_many_chunks_have_the_bits_of_few(lib, gpu, r):
    """More than 608 chunks (at r < 128 several per CTA, the last CTA's incomplete; panels of one and
    of two chunks, the second of 16 rows, so that most of the CTAs its slices are dealt to have
    none): each panel has the bits it has in a context of its own."""
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    n = [(4 * r + 1, 4 * r + 37)] * 306 + [(1040, 4 * r)]
    weights = [torch.zeros(a, (b + 7) // 8 * 8, dtype=torch.bfloat16, device=gpu)[:, :b] for a, b in n]
    z = SubZeroPlus(weights, r, 2, 8)
    z.refresh(1)
    z.sync()
    for i in (0, 1, 7, 8, 150, 304, 305, 306):
        one = SubZeroPlus(weights[i:i + 1], r, 2, 8, matrix_index_base=i)
        one.refresh(1)
        one.sync()
        assert torch.equal(one.U[0], z.U[i]) and torch.equal(one.V[0], z.V[i]), i
        one.close()
    z.close()
