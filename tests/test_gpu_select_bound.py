"""The selection's bound is a guess from a sample of the tokens: inputs that mislead it must give the same lists.  Also the edges
of the candidate chunks (16 to 64 tokens), for both block sizes, storage types and head dimensions."""
import numpy as np
import pytest
import torch

from gpu_util import check_compression
from oracle import fdkv_ref as R
from oracle import fdkv_ref_b4 as R4
from paper_2607_06519_b200 import synth

pytestmark = pytest.mark.gpu


def _sampled_tokens(T, d):
    """Tokens the bound is taken from: one in each of n equal parts, at a hashed place."""
    n = min(T, 65536 // d)
    r = np.arange(n, dtype=np.uint64)
    jitter = ((r * np.uint64(2654435761)) & np.uint64(0xFFFFFFFF)) >> np.uint64(16)
    return ((((r << np.uint64(16)) | jitter) * np.uint64(T)) // np.uint64(n << 16)).astype(np.int64)


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("factor", [100.0, 0.01])
@pytest.mark.parametrize("keep", [(1, 4), (1, 64)])
def test_a_sample_that_misleads(dtype, d, factor, keep):
    """The sampled tokens' deviations a hundred times larger (too few candidates: everything runs again with bound 0) or
    smaller (far too many)."""
    from paper_2607_06519_b200 import binding as B

    T = 5003
    rng = np.random.default_rng(7)
    scale = np.ones((T, 1, 1), np.float32)
    scale[_sampled_tokens(T, d)] = factor
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    base = rng.standard_normal((T, 2, d)).astype(np.float32)
    x = [torch.from_numpy(a).to(tdt).cuda() for a in (base, base + scale * rng.standard_normal((T, 2, d)).astype(np.float32))]
    ctx = B.Context(B.Config(2, 2, 2, d, 1, T, 1, B.BF16 if dtype == "bf16" else B.F32, *keep))
    ctx.compress_prefill(0, 0, 1, T, x, x)
    for h in range(2):
        _, z1 = R.depth_split(x[0][:, h].float().cpu().numpy(), x[1][:, h].float().cpu().numpy(), dtype == "bf16")
        want = R.select_entries(z1, T * d * keep[0] // keep[1])
        for is_v in (0, 1):
            idx, val = ctx.get_residual(0, 0, h, is_v)
            assert np.array_equal(idx.cpu().numpy(), want)
            assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])
    assert ctx.device_status() == 0


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("T", [1, 31, 32, 33, 63, 64, 65, 127, 128, 129, 1024, 1025, 2049])
def test_chunk_edges(dtype, d, T):
    from paper_2607_06519_b200 import runner

    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=1, n_q_heads=2, head_dim=d, T=T, dtype=dtype, n_needles=min(T, 2), W=1,
                                            keep_num=1, keep_den=5, name="edges")
    pf = runner.Prefilled(w)
    pf.compress(0)
    check_compression(pf.ctx, w, 0, 0, 0)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("hkv", [4, 8])
def test_a_sample_that_misleads_for_one_head(hkv):
    """Only one head's K runs again with bound 0: a block then works on items that lie one, three, ... others apart."""
    from paper_2607_06519_b200 import binding as B

    T, d, L = 5003, 128, 8
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    scale = torch.ones((T, 1, 1), device="cuda")
    scale[torch.from_numpy(_sampled_tokens(T, d)).cuda()] = 100.0
    k, v = [], []
    for layer in range(L):
        if layer % 2 == 0:
            base = [torch.randn((T, hkv, d), generator=g, device="cuda") for _ in range(2)]
            k.append(base[0].bfloat16())
            v.append(base[1].bfloat16())
        else:
            dk, dv = (torch.randn((T, hkv, d), generator=g, device="cuda") for _ in range(2))
            dk[:, 1:2] *= scale
            k.append((base[0] + dk).bfloat16())
            v.append((base[1] + dv).bfloat16())
    ctx = B.Context(B.Config(L, hkv, hkv, d, 1, T, 1, B.BF16, 1, 16))
    ctx.compress_prefill(0, 0, L // 2, T, k, v)
    for p in range(L // 2):
        for h in range(hkv):
            for is_v, x in ((0, k), (1, v)):
                _, z1 = R.depth_split(x[2 * p][:, h].float().cpu().numpy(), x[2 * p + 1][:, h].float().cpu().numpy(), True)
                want = R.select_entries(z1, T * d // 16)
                idx, val = ctx.get_residual(0, p, h, is_v)
                assert np.array_equal(idx.cpu().numpy(), want), (p, h, is_v)
                assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want]), (p, h, is_v)
    assert ctx.device_status() == 0


@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
@pytest.mark.parametrize("T,keep", [(4099, (3, 10)), (4099, (6, 10)), (4099, (61, 100)), (4099, (99, 100)), (4099, (1, 1)), (1030, (3, 4)), (9000, (2, 5))])
@pytest.mark.parametrize("block", [2, 4])
def test_lists_of_many_entries(dtype, d, T, keep, block):
    """Either side of the shares from which every position is listed as a candidate, up to all of them."""
    from paper_2607_06519_b200 import runner

    if T == 9000 and (dtype, block, d) != ("bf16", 2, 128):
        pytest.skip("one long case")
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=block, n_kv_heads=2, n_q_heads=2, head_dim=d, T=T, dtype=dtype, n_needles=2, W=1, keep_num=keep[0],
                                            keep_den=keep[1], block_size=block, name="many")
    pf = runner.Prefilled(w)
    pf.compress(0)
    for h in range(2):
        if block == 2:
            check_compression(pf.ctx, w, 0, 0, h)
            continue
        u = R4.Unit4(synth.block_tensor(w, 0, 0, h, False), synth.block_tensor(w, 0, 0, h, True), dtype == "bf16", *keep)
        for is_v, name in ((0, "k"), (1, "v")):
            idx, val = pf.ctx.get_residual(0, 0, h, is_v)
            got = idx.cpu().numpy()
            assert np.array_equal(got, u.kept[name])
            want = np.stack([u.dev[name][l].ravel()[got] for l in range(4)])
            assert np.array_equal(val.float().cpu().numpy().reshape(4, -1), want)
    assert pf.ctx.device_status() == 0
    pf.ctx.close()


@pytest.mark.parametrize("keep", [(1, 3), (7, 10)])
@pytest.mark.parametrize("factor", [100.0, 0.01])
def test_a_sample_that_misleads_many(keep, factor):
    """The same with many entries: a list of candidates, and every position one (whose threshold starts from the sample's bound too)."""
    test_a_sample_that_misleads("bf16", 128, factor, keep)
    test_a_sample_that_misleads("f32", 64, factor, keep)



@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("dtype,T,keep", [("bf16", 5003, (1, 64)), ("f32", 5003, (1, 16)), ("bf16", 509, (1, 16)), ("bf16", 8192, (1, 2))])
def test_shared_coefficients_in_a_layers_place(dtype, T, keep, which):
    """One tensor pair whose shared coefficients replace a layer's rows, with a sample that misleads: no row is read twice."""
    from paper_2607_06519_b200 import binding as B

    d = 128
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    rng = np.random.default_rng(7)
    scale = np.ones((T, 1), np.float32)
    scale[_sampled_tokens(T, d)] = 100.0
    base = rng.standard_normal((T, d)).astype(np.float32)
    x = [torch.from_numpy(a).to(tdt).cuda() for a in (base, base + scale * rng.standard_normal((T, d)).astype(np.float32))]
    want_z0, z1 = R.depth_split(x[0].float().cpu().numpy(), x[1].float().cpu().numpy(), dtype == "bf16")
    k = T * d * keep[0] // keep[1]
    want = R.select_entries(z1, k)
    idx, val = torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, dtype=tdt, device="cuda")
    assert B.compress_unit_noalloc(x[0], x[1], *keep, x[which], idx, val) == k
    assert np.array_equal(x[which].float().cpu().numpy(), want_z0)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("values", ["normal", "few", "wide"])
@pytest.mark.parametrize("hkv,T", [(12, 1501), (10, 4099)])
@pytest.mark.parametrize("den", [9, 2])
def test_threshold_of_many_tensors(den, hkv, T, values, dtype):
    """A block per tensor: the k-th key among the 63 above the bound and far from it (values over forty octaves), and more keys that share
    the first digit than are gathered (integers); with half of them kept the sample expects it far away more often."""
    from paper_2607_06519_b200 import binding as B

    d, tdt = 128, torch.bfloat16 if dtype == "bf16" else torch.float32
    rng = np.random.default_rng(12)
    base = rng.integers(-8, 9, (T, hkv, d)).astype(np.float32)
    diff = rng.standard_normal((T, hkv, d)).astype(np.float32)
    if values == "few":
        diff = np.rint(diff)
    elif values == "wide":
        base, diff = 0 * base, np.ldexp(diff, rng.integers(-20, 20, diff.shape)).astype(np.float32)
    x = [torch.from_numpy(a).to(tdt).cuda() for a in (base, base + diff)]
    ctx = B.Context(B.Config(2, hkv, hkv, d, 1, T, 1, B.BF16 if dtype == "bf16" else B.F32, 1, den))
    ctx.compress_prefill(0, 0, 1, T, x, x)
    for h in (0, hkv - 1):
        _, z1 = R.depth_split(x[0][:, h].float().cpu().numpy(), x[1][:, h].float().cpu().numpy(), dtype == "bf16")
        want = R.select_entries(z1, T * d // den)
        idx, val = ctx.get_residual(0, 0, h, 1)
        assert np.array_equal(idx.cpu().numpy(), want)
        assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])
    assert ctx.device_status() == 0
