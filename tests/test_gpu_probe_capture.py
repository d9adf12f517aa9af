"""A probe call inside a stream capture: replays score the queries as they are then, and the budget and the commit that follow use
the replays' scores.  Both selection rules."""
import numpy as np
import pytest
import torch

from paper_2607_06519_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule,T", [(0, 700), (0, 3000), (1, 700)])
def test_captured_probe(rule, T):
    L, H, G, d, W = 4, 2, 2, 128, 16
    g = torch.Generator(device="cuda")
    g.manual_seed(3)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda").bfloat16()

    k, v = ([rand(T, H, d) for _ in range(L)] for _ in range(2))
    q = [rand(W, G * H, d) for _ in range(L)]
    other = [3 * rand(W, G * H, d) for _ in range(L)]
    pos = np.arange(T - W, T, dtype=np.int32)
    budget = int(0.75 * 2 * L * H * T * d * 2)

    def staged():
        ctx = B.Context(B.Config(L, G * H, H, d, 1, T, 1, B.BF16, 1, 16, rule))
        ctx.compress_prefill(0, 0, L // 2, T, k, v)
        return ctx

    want = []
    for x in (q, other):
        ctx = staged()
        _, scores = ctx.probe(0, 0, L // 2, x, pos, 0.0)
        want.append((scores.clone(), ctx.route_budget(0, budget)))
        ctx.close()
    ctx = staged()
    ctx.probe(0, 0, L // 2, other, pos, 0.0)  # (an earlier call on another stream than the capture's)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        _, scores = ctx.probe(0, 0, L // 2, q, pos, 0.0)
    pos[:] = 0
    for x, (want_scores, want_route) in zip((q, other), want):
        for a, b in zip(q, x):
            a.copy_(b)
        graph.replay()
        assert torch.equal(scores, want_scores)
        fits, lam, modes = ctx.route_budget(0, budget)
        assert fits == want_route[0] and lam == want_route[1] and torch.equal(modes, want_route[2])
    ctx.commit(0)
    out = ctx.decode_attn(0, rand(1, G * H, d))
    assert bool(torch.isfinite(out.float()).all())
    assert ctx.device_status() == 0
    del graph
    ctx.close()
