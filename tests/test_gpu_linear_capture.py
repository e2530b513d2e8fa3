"""zo_linear_perturbed under stream capture: what a call may allocate, and replays."""

import pytest
import torch

from gpu_util import make_weight
from test_gpu_linear import _tokens

pytestmark = pytest.mark.gpu


def _layer(gpu, stream, r, m, n):
    from paper_2608_15665_gb300 import binding as zb
    from paper_2608_15665_gb300.schedule import SubZeroPlus
    z = SubZeroPlus([make_weight(m, n, "bf16", 6, gpu)], r, 2, 11, stream=stream)
    z.init_subspace(0)
    zb.zo_linear_prepare(z.ctx, 3, 0, 1.0, -1, 0.0, 1e-1)
    return z


def test_few_token_call_within_the_token_capacity_allocates_nothing(lib, gpu):
    """100 tokens leave a workspace for 128: a captured call of 120, the largest so far, neither
    synchronises the stream nor allocates."""
    from paper_2608_15665_gb300 import binding as zb
    s = torch.cuda.Stream()
    z = _layer(gpu, s, 32, 264, 2056)
    X = _tokens(120, 2056, 3, gpu)
    Y = torch.empty(120, 264, dtype=torch.bfloat16, device=gpu)
    torch.cuda.synchronize()
    zb.zo_linear_perturbed(z.ctx, 0, X[:100], Y[:100])
    z.sync()
    Y.fill_(float("nan"))
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        zb.zo_linear_perturbed(z.ctx, 0, X, Y)
    g.replay()
    torch.cuda.synchronize()
    want = torch.empty_like(Y)
    torch.cuda.synchronize()
    zb.zo_linear_perturbed(z.ctx, 0, X, want)
    assert zb.zo_linear_tiling(z.ctx) == 9
    z.sync()
    assert torch.equal(Y, want)
    z.close()


@pytest.mark.parametrize("T", [97, 300])
def test_replays_read_the_rows_of_their_own_s(lib, gpu, T):
    """A captured call (few tokens; SM pairs) replayed on other inputs in turn: the tiles of Y wait
    for this replay's S, not for the flags that the one before has left.  S = X P^T carries a
    large part of Y here, so that another replay's S shows."""
    from paper_2608_15665_gb300 import binding as zb
    s = torch.cuda.Stream()
    z = _layer(gpu, s, 32, 1024, 4104)
    zb.zo_linear_prepare(z.ctx, 3, 0, 1.0, -1, 0.0, 10.0)
    inputs = [_tokens(T, 4104, 100 + k, gpu) for k in range(4)]
    wants = [torch.empty(T, 1024, dtype=torch.bfloat16, device=gpu) for _ in inputs]
    X, Y = torch.empty_like(inputs[0]), torch.empty_like(wants[0])
    torch.cuda.synchronize()
    for x, want in zip(inputs, wants):
        zb.zo_linear_perturbed(z.ctx, 0, x, want)
        assert (zb.zo_linear_tiling(z.ctx) == 9) == (T <= 128)
    z.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        zb.zo_linear_perturbed(z.ctx, 0, X, Y)
    for k in [0, 1, 2, 3] * 5:
        X.copy_(inputs[k])
        Y.fill_(float("nan"))
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(Y, wants[k]), k
    # a live call after the replays, and a replay after it
    zb.zo_linear_perturbed(z.ctx, 0, inputs[2], Y)
    z.sync()
    assert torch.equal(Y, wants[2])
    X.copy_(inputs[1])
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        g.replay()
    z.sync()
    assert torch.equal(Y, wants[1])
    z.close()
