"""The few-token linear layer (tiling 9: all the tokens x a few columns of Y per CTA,
S from the first CTAs) at the sizes where it can go wrong: one token, a token more or
less than the boxes' steps, the 32 tokens of a CTA of S and the most it takes, K
of one stage up to many with a ragged last panel, columns of Y that do not fill the last CTA,
padded rows of X, W and Y; the flags of calls in turn with the SM-pair kernel's."""

import pytest
import torch

from gpu_util import f32, make_weight, snapshot
from oracle import subzero
from test_gpu_linear import _check, _tokens

pytestmark = pytest.mark.gpu

SHAPES = [(8 * 17, 136, 144), (128, 520, None), (136, 2056, None), (520, 4104, 4112), (264, 128, None)]


@pytest.mark.parametrize("r", [16, 32, 64])
def test_few_tokens_match_oracle(lib, gpu, r):
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    spec = [s for s in SHAPES if min(s[0], s[1]) >= r]
    z = SubZeroPlus([make_weight(m, n, "bf16", 30 + k, gpu, ldw) for k, (m, n, ldw) in enumerate(spec)],
                    r, 2, 321, matrix_index_base=7)
    z.init_subspace(0)
    eps = 1e-1
    zb.zo_linear_prepare(z.ctx, 3, 1, 1.0, 0, -1.0, eps)
    before = snapshot(z)
    took = 0
    for i, (m, n, _) in enumerate(spec):
        C = subzero.perturb_coeff(321, 7 + i, 3, r, [(1, 1.0), (0, -1.0)], f32(eps))
        for T in (1, 15, 16, 17, 31, 32, 33, 97, 128, 129, 300, 64):
            Xb = torch.zeros(T, n + 8, dtype=torch.bfloat16, device=gpu)
            Xb[:, :n] = _tokens(T, n, 5 * T + i, gpu)
            Xb[:, n:] = float("nan")                    # past X's columns: not read
            Y = torch.full((T, m + 8), float("nan"), dtype=torch.bfloat16, device=gpu)
            zb.zo_linear_perturbed(z.ctx, i, Xb[:, :n], Y[:, :m])
            tiling = zb.zo_linear_tiling(z.ctx)
            z.sync()
            took += tiling == 9
            if tiling == 9:
                # the SM-pair kernel's K steps and products, in its order: its bits
                Yp = torch.empty(T, m, dtype=torch.bfloat16, device=gpu)
                zb.zo_set_option(z.ctx, zb.ZO_OPTION_LINEAR_TILE, 8)
                zb.zo_linear_perturbed(z.ctx, i, Xb[:, :n], Yp)
                zb.zo_set_option(z.ctx, zb.ZO_OPTION_LINEAR_TILE, 0)
                z.sync()
                assert torch.equal(Y[:, :m], Yp), (m, n, T)
            assert torch.isnan(Y[:, m:].float()).all()
            _check(Y[:, :m], Xb[:, :n], before["W"][i], before["U"][i], before["V"][i], C,
                   2.0 * f32(eps), f"r={r} {m}x{n} T={T}")
    assert took >= 5 * len(spec)
    z.close()


def test_few_token_wait_reports_timeout_and_the_context_recovers(lib, gpu):
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    z = SubZeroPlus([make_weight(264, 2056, "bf16", 4, gpu)], 32, 2, 9)
    z.init_subspace(0)
    zb.zo_linear_prepare(z.ctx, 3, 0, 1.0, -1, 0.0, 1e-2)
    X = _tokens(40, 2056, 12, gpu)
    Y = torch.empty((40, 264), dtype=torch.bfloat16, device=gpu)
    zb.zo_linear_perturbed(z.ctx, 0, X, Y)
    z.sync()
    want = Y.clone()
    zb.zo_set_option(z.ctx, zb.ZO_OPTION_TEST_WAIT_TIMEOUT, 1)
    zb.zo_linear_perturbed(z.ctx, 0, X, Y)
    assert zb.zo_linear_tiling(z.ctx) == 9
    with pytest.raises(zb.ZoError) as e:
        z.sync()
    assert e.value.status == zb.ZO_ERR_TIMEOUT
    z.sync()
    Y.fill_(float("nan"))
    zb.zo_linear_perturbed(z.ctx, 0, X, Y)
    z.sync()
    assert torch.equal(Y, want)
    z.close()
