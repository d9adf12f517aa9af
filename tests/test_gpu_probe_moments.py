"""Probe errors by second moments (keys every probe query sees) and by products (the keys after): both block sizes, lengths
and probe positions around the 128- and 256-key tiles, more and fewer probe rows than a 128-row tile, units shared by
several thread blocks and thread blocks that share units."""
import numpy as np
import pytest
import torch

from oracle import fdkv_ref as R
from oracle import fdkv_ref_b4 as R4
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [2, 4])
@pytest.mark.parametrize("hkv,group,T,pos", [
    (1, 1, 257, [254]), (1, 1, 257, [255]), (1, 2, 300, [256, 299]), (2, 4, 1000, range(990, 1000)), (1, 1, 20000, [19999]),
    (3, 4, 700, range(600, 700)), (8, 4, 2049, range(1985, 2049)), (2, 8, 5000, [10, 3000, 4999]), (2, 1, 1100, [511, 512, 1023, 1024]),
])
def test_probe_errors(block, hkv, group, T, pos):
    pos = np.array(list(pos), dtype=np.int32)
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2 * block, n_kv_heads=hkv, n_q_heads=hkv * group, T=T, W=len(pos), n_needles=4, keep_den=7,
                                            block_size=block, name="moments")
    pf = runner.Prefilled(w)
    pf.compress(0)
    _, scores = pf.ctx.probe(0, 0, w.n_blocks, pf.upload_probe_q(0), pos, 0.0)
    scores = scores.cpu().numpy()
    for p in range(w.n_blocks):
        pq = [synth.probe_q(w, 0, block * p + l) for l in range(block)]
        for h in sorted({0, hkv - 1}):
            if block == 4:
                u = R4.Unit4(synth.block_tensor(w, 0, p, h, False), synth.block_tensor(w, 0, p, h, True), True, w.keep_num, w.keep_den)
                want = R4.probe_error4(u.dev["k"], u.kept["k"], pq, group, h, pos)
            else:
                u = R.Unit(*synth.unit_tensor(w, 0, p, h, False), *synth.unit_tensor(w, 0, p, h, True), True, w.keep_num, w.keep_den)
                want = R.probe_error(u.z1["k"], u.kept["k"], pq[0], pq[1], group, h, pos)
            np.testing.assert_allclose(scores[p, h], want, rtol=2e-5)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("hkv,T,pos", [(1, 1300, [1278, 1299]), (1, 1300, [1279, 1299]), (150, 2048, [5, 2047]), (150, 2049, [5, 2048])])
def test_products_of_short_prompts_and_items(hkv, T, pos):
    """The most keys that go to the products although every query sees them, and one tile more; items of eight tiles and of nine."""
    test_probe_errors(2, hkv, 1, T, pos)


@pytest.mark.parametrize("block,group,W", [(2, 4, 64), (2, 8, 128), (4, 2, 16)])
@pytest.mark.parametrize("eps", [1.0, 0.2, 0.03, 0.0])
def test_queries_nearly_orthogonal_to_the_deviations(block, group, W, eps):
    """Deviations in a random half of the directions, queries in the other half up to a share eps (and the rounding to bf16): the
    second moments' sum cancels, the products do not.  A product is 8 steps of float32 rounded towards zero and its square, second
    moments are 16 and 8: 2e-6 covers either and the float32 scores."""
    from paper_2607_06519_b200 import binding as B

    hkv, T, d = 2, 3100, 128
    g = torch.Generator(device="cuda")
    g.manual_seed(5)

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    u, _ = torch.linalg.qr(rand(d, d))
    x = [(rand(T, hkv, 64) @ u[:64]).bfloat16() for _ in range(block)]
    q = [(rand(W, hkv * group, 64) @ u[64:] + eps * rand(W, hkv * group, 64) @ u[:64]).bfloat16() for _ in range(block)]
    ctx = B.Context(B.Config(block, hkv * group, hkv, d, 1, T, 1, B.BF16, 1, 16, block_size=block))
    ctx.compress_prefill(0, 0, 1, T, x, x)
    pos = np.arange(T - W, T, dtype=np.int32)
    _, scores = ctx.probe(0, 0, 1, q, pos, 0.0)
    for h in range(hkv):
        xs = [a[:, h].float().cpu().numpy() for a in x]
        qs = [a.float().cpu().numpy() for a in q]
        if block == 4:
            u4 = R4.Unit4(xs, xs, True, 1, 16)
            want = R4.probe_error4(u4.dev["k"], u4.kept["k"], qs, group, h, pos)
        else:
            u2 = R.Unit(*xs, *xs, True, 1, 16)
            want = R.probe_error(u2.z1["k"], u2.kept["k"], qs[0], qs[1], group, h, pos)
        np.testing.assert_allclose(scores[0, h].cpu().numpy(), want, rtol=2e-6)
    assert ctx.device_status() == 0
    ctx.close()


@pytest.fixture
def moments(monkeypatch):
    """Every probe call takes second moments for all keys that every query sees, however few."""
    from paper_2607_06519_b200 import binding as B

    probe = B.Context.probe

    def always(self, *args, **kw):
        assert B._lib.fdkv_test_probe_moments(self.h, 1) == 0
        return probe(self, *args, **kw)

    monkeypatch.setattr(B.Context, "probe", always)


@pytest.mark.parametrize("block", [2, 4])
@pytest.mark.parametrize("hkv,group,T,pos", [
    (1, 1, 257, [254]), (1, 1, 257, [255]), (1, 2, 300, [256, 299]), (2, 4, 1000, range(990, 1000)), (1, 1, 20000, [19999]),
    (3, 4, 700, range(600, 700)), (8, 4, 2049, range(1985, 2049)), (2, 8, 5000, range(4900, 5000)), (2, 1, 1100, [511, 512, 1023, 1024]),
])
def test_probe_errors_by_moments(block, hkv, group, T, pos, moments):
    test_probe_errors(block, hkv, group, T, pos)


@pytest.mark.parametrize("block,group,W", [(2, 4, 64), (2, 8, 128), (4, 2, 16)])
@pytest.mark.parametrize("eps", [1.0, 0.2, 0.03, 0.0])
def test_queries_nearly_orthogonal_by_moments(block, group, W, eps, moments):
    test_queries_nearly_orthogonal_to_the_deviations(block, group, W, eps)


@pytest.mark.parametrize("layers,hkv,group,W,T", [(32, 8, 4, 64, 1400), (32, 8, 4, 64, 2300), (8, 8, 1, 4, 2100), (8, 8, 1, 4, 4200)])
def test_either_side_of_the_rule(layers, hkv, group, W, T):
    """Where the rule turns from products to moments: both forms of the same call, and the rule's."""
    from paper_2607_06519_b200 import binding as B

    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    k = [torch.randn((T, hkv, 128), generator=g, device="cuda").bfloat16() for _ in range(layers)]
    q = [torch.randn((W, hkv * group, 128), generator=g, device="cuda").bfloat16() for _ in range(layers)]
    ctx = B.Context(B.Config(layers, hkv * group, hkv, 128, 1, T, 1, B.BF16, 1, 16))
    ctx.compress_prefill(0, 0, layers // 2, T, k, k)
    got = []
    for form in (2, 1, 0):
        assert B._lib.fdkv_test_probe_moments(ctx.h, form) == 0
        got.append(ctx.probe(0, 0, layers // 2, q, np.arange(T - W, T, dtype=np.int32), 0.0)[1].double().cpu().numpy())
    np.testing.assert_allclose(got[1], got[0], rtol=2e-6)
    assert np.array_equal(got[2], got[0]) or np.array_equal(got[2], got[1])
    assert ctx.device_status() == 0
    ctx.close()
