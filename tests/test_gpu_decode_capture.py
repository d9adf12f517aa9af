"""Captured decode calls of short contexts: a replay reads the descriptors that the device holds then, so it serves a later prompt of the
same length with other modes too; few units and more."""
import pytest
import torch

from paper_2607_06519_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv", [2, 8, 9])
def test_replay_after_another_commit(hkv):
    L, G, d, T = 2, 2, 128, 700
    g = torch.Generator(device="cuda")
    g.manual_seed(4)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda").bfloat16()

    ctx = B.Context(B.Config(L, G * hkv, hkv, d, 1, T, 1, B.BF16, 1, 16))
    q, out, want = rand(1, G * hkv, d), torch.empty((1, G * hkv, d), dtype=torch.bfloat16, device="cuda"), []
    graph = torch.cuda.CUDAGraph()
    for prompt in range(2):
        if prompt:
            ctx.reset()
        k, v = ([rand(T, hkv, d) for _ in range(L)] for _ in range(2))
        ctx.compress_prefill(0, 0, 1, T, k, v)
        ctx.set_modes(0, [(h + prompt) % 3 for h in range(hkv)])
        ctx.commit(0)
        want.append(ctx.decode_attn(1, q).clone())
        if not prompt:
            with torch.cuda.graph(graph):
                ctx.decode_attn(1, q, out=out)
        graph.replay()
        assert torch.equal(out, want[prompt])
    assert not torch.equal(want[0], want[1])
    assert ctx.device_status() == 0
    del graph
    ctx.close()
