"""The refresh at r = 4 and 8 with panels in registers, at its edges: short panels up to the
last Householder one and the first tall one, panels of one row less and more than a CTA's and
a cluster's, and one that falls back to the TSQR; the set in one context, refreshed twice."""

import numpy as np
import pytest
import torch

from gpu_util import make_weight, snapshot
from oracle import haar
from parity import UV_ABS

pytestmark = pytest.mark.gpu

CASES = {
    4: [(4, 5), (15, 16), (17, 31), (5119, 5120), (5121, 10241), (20480, 20481), (40960, 40961)],
    8: [(8, 9), (31, 32), (33, 2047), (2048, 2049), (4096, 4097), (8192, 8193), (16384, 16385)],
}


@pytest.mark.parametrize("r", [4, 8])
def test_panels_in_registers_match_oracle(lib, gpu, r):
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    seed, base = 90 + r, 3
    # only U and V matter: one row of W per panel pair is enough for a wide matrix's memory
    weights = [make_weight(m, n, "f32", k, gpu, ldw=(n + 3) // 4 * 4) if m * n < 1 << 22
               else torch.zeros(m, (n + 3) // 4 * 4, device=gpu)[:, :n]
               for k, (m, n) in enumerate(CASES[r])]
    z = SubZeroPlus(weights, r, 2, seed, matrix_index_base=base)
    for j in (1, 2):
        z.refresh(j)
        z.sync()
        s = snapshot(z)
        for i, (m, n) in enumerate(CASES[r]):
            U, V = haar.haar_proj(seed, base + i, j, m, n, r)
            for got, want, rows in ((s["U"][i], U, m), (s["V"][i], V, n)):
                # nearly square Gaussian panels: fp32's error grows with the condition number
                # (up to ~100 here), 1e-5 elsewhere as in the other refresh tests
                tol = UV_ABS if rows >= 2 * r else 10 * UV_ABS
                assert np.max(np.abs(got - want)) <= tol, (r, rows)
                assert np.max(np.abs(got.T @ got - np.eye(r))) <= 1e-5
    a = [t.clone() for t in z.U + z.V]
    z.refresh(1)
    z.refresh(2)
    z.sync()
    assert all(torch.equal(x, y) for x, y in zip(a, z.U + z.V))
    z.close()


@pytest.mark.parametrize("r", [4, 8])
def test_short_panels_have_the_householder_panels_bits(lib, gpu, r):
    """fp32 and bf16 weights of one index: panels shorter than 4r, whose condition number can be
    large, are the same whichever kernel forms them."""
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    shapes = [(r, r + 1), (2 * r - 1, 2 * r), (2 * r + 1, 4 * r - 1)]
    sets = [[torch.zeros(m, (n + 7) // 8 * 8, dtype=dt, device=gpu)[:, :n] for m, n in shapes]
            for dt in (torch.float32, torch.bfloat16)]
    got = []
    for weights in sets:
        z = SubZeroPlus(weights, r, 2, 17, matrix_index_base=4)
        z.refresh(2)
        z.sync()
        got.append([t.clone() for t in z.U + z.V])
        z.close()
    assert all(torch.equal(a, b) for a, b in zip(*got))
