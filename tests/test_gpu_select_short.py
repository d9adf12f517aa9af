"""Few short unit-tensors, one cluster each: the edges of its tiles, blocks and 32-position words, every key equal, everything and
nothing kept; and as many of the same lengths that the four kernels of longer ones take them."""
import numpy as np
import pytest
import torch

from gpu_util import check_compression
from oracle import fdkv_ref as R
from oracle import fdkv_ref_b4 as R4
from paper_2607_06519_b200 import binding as B
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu


LENGTHS = [(1, 2), (15, 3), (16, 16), (17, 5), (113, 8), (128, 8), (129, 8), (1008, 16), (1024, 16), (1025, 16), (2048, 16), (2049, 16)]


@pytest.mark.parametrize("hkv,T,den", [(1, *x) for x in LENGTHS] + [(40, *x) for x in LENGTHS if x[0] < 200])
@pytest.mark.parametrize("dtype,d", [("bf16", 128), ("bf16", 64), ("f32", 128), ("f32", 64)])
def test_lengths(dtype, d, hkv, T, den):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv, head_dim=d, T=T, dtype=dtype, n_needles=min(T, 2), W=1,
                                            keep_num=1, keep_den=den, name="short")
    pf = runner.Prefilled(w)
    pf.compress(0)
    for h in {0, hkv - 1}:
        check_compression(pf.ctx, w, 0, 0, h)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("keep", [(0, 1), (1, 1), (1, 3), (2, 3)])
@pytest.mark.parametrize("equal", [True, False])
def test_ties_and_extremes(dtype, keep, equal):
    """Keys of one or of three values, so that ties go on over blocks and words."""
    T, d = 500, 128
    rng = np.random.default_rng(3)
    diff = np.ones((T, d), np.float32) if equal else rng.integers(-1, 2, (T, d)).astype(np.float32)
    base = rng.integers(-4, 5, (T, d)).astype(np.float32)
    x0, x1 = (torch.from_numpy(a).cuda().to(dtype) for a in (base + diff, base - diff))
    k = T * d * keep[0] // keep[1]
    z0, idx, val = torch.empty((T, d), dtype=dtype, device="cuda"), torch.full((max(k, 4),), -1, dtype=torch.int32, device="cuda"), torch.empty(max(k, 4), dtype=dtype, device="cuda")
    assert B.compress_unit_noalloc(x0, x1, *keep, z0, idx[:k] if k else idx, val[:k] if k else val) == k
    torch.cuda.synchronize()
    want_z0, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), dtype == torch.bfloat16)
    want = R.select_entries(z1, k)
    assert np.array_equal(z0.float().cpu().numpy(), want_z0)
    assert np.array_equal(idx[:k].cpu().numpy(), want)
    assert np.array_equal(val[:k].float().cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("T", [16, 100, 509, 512, 513])
def test_blocks_of_four(T):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=4, n_kv_heads=2, n_q_heads=4, T=T, n_needles=2, W=1, keep_num=1, keep_den=9, block_size=4,
                                            name="short4")
    pf = runner.Prefilled(w)
    pf.compress(0)
    for h in range(2):
        for is_v, name in ((0, "k"), (1, "v")):
            u = R4.Unit4(synth.block_tensor(w, 0, 0, h, False), synth.block_tensor(w, 0, 0, h, True), True, 1, 9)
            idx, val = pf.ctx.get_residual(0, 0, h, is_v)
            assert np.array_equal(idx.cpu().numpy(), u.kept[name])
            want = np.stack([u.dev[name][l].ravel()[u.kept[name]] for l in range(4)])
            assert np.array_equal(val.float().cpu().numpy(), want)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("T", [30, 509, 1000])
@pytest.mark.parametrize("scale", [0.0, 2.0**-40, 2.0**-24, 2.0**9, 2.0**60, 2.0**120])
@pytest.mark.parametrize("den", [2, 16])
def test_any_scale(scale, den, T):
    """The k-th key below the first window of octaves, at its edges, above it, and with positions on both sides of it."""
    d = 128
    rng = np.random.default_rng(5)
    x = rng.standard_normal((2, T, d)).astype(np.float32)
    x[:, ::3] *= scale
    if scale > 1:
        x[:, 1::3] *= 2.0**-80
    x0, x1 = (torch.from_numpy(a).cuda().bfloat16() for a in x)
    k = T * d // den
    z0, idx, val = torch.empty_like(x0), torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, dtype=torch.bfloat16, device="cuda")
    assert B.compress_unit_noalloc(x0, x1, 1, den, z0, idx, val) == k
    _, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), True)
    want = R.select_entries(z1, k)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("dtype,d,T", [("bf16", 128, 2064), ("bf16", 64, 4111), ("bf16", 128, 4096), ("bf16", 128, 4097), ("bf16", 128, 8064), ("bf16", 128, 8065),
                                       ("f32", 128, 4096), ("f32", 128, 4097), ("f32", 64, 4099), ("f32", 64, 8191)])
@pytest.mark.parametrize("den", [3, 16])
def test_clusters_of_sixteen(dtype, d, T, den):
    """Two and four words of positions per thread, at and beside the most that two of them hold, and lengths that four no longer hold."""
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=1, n_q_heads=1, head_dim=d, T=T, dtype=dtype, n_needles=2, W=1, keep_num=1, keep_den=den,
                                            name="sixteen")
    pf = runner.Prefilled(w)
    pf.compress(0)
    check_compression(pf.ctx, w, 0, 0, 0)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("T", [600, 1500, 1600])
def test_blocks_of_four_in_clusters_of_sixteen(T):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=4, n_kv_heads=1, n_q_heads=1, T=T, n_needles=2, W=1, keep_num=1, keep_den=9, block_size=4, name="sixteen4")
    pf = runner.Prefilled(w)
    pf.compress(0)
    for is_v, name in ((0, "k"), (1, "v")):
        u = R4.Unit4(synth.block_tensor(w, 0, 0, 0, False), synth.block_tensor(w, 0, 0, 0, True), True, 1, 9)
        idx, val = pf.ctx.get_residual(0, 0, 0, is_v)
        assert np.array_equal(idx.cpu().numpy(), u.kept[name])
        assert np.array_equal(val.float().cpu().numpy(), np.stack([u.dev[name][l].ravel()[u.kept[name]] for l in range(4)]))
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("keep", [(0, 1), (1, 1), (1, 3), (2, 3)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_ties_over_sixteen_blocks(dtype, keep):
    T, d = 4099, 64
    rng = np.random.default_rng(6)
    diff, base = rng.integers(-1, 2, (T, d)).astype(np.float32), rng.integers(-4, 5, (T, d)).astype(np.float32)
    x0, x1 = (torch.from_numpy(a).cuda().to(dtype) for a in (base + diff, base - diff))
    k = T * d * keep[0] // keep[1]
    z0, idx, val = torch.empty((T, d), dtype=dtype, device="cuda"), torch.full((max(k, 4),), -1, dtype=torch.int32, device="cuda"), torch.empty(max(k, 4), dtype=dtype, device="cuda")
    assert B.compress_unit_noalloc(x0, x1, *keep, z0, idx[:k] if k else idx, val[:k] if k else val) == k
    _, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), dtype == torch.bfloat16)
    want = R.select_entries(z1, k)
    assert np.array_equal(idx[:k].cpu().numpy(), want)
    assert np.array_equal(val[:k].float().cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("T,near", [(T, near) for T in (40, 500, 2100) for near in (1, 127, 128, 129, 1023, 1024, 1025, 4000)] +
                         [(8000, near) for near in (1, 4095, 4096, 4097, 20000)])
@pytest.mark.parametrize("copies", [1, 3])
def test_keys_that_share_the_top_half(copies, T, near):
    """float32 keys of which exactly `near` share the threshold's upper 16 bits, each value `copies` times: ranked one by one, by digits
    among those gathered, or by digits over the cluster, and (8000 tokens) gathered or counted over the chunks; the threshold at the
    first, in the middle and at the last of them."""
    d = 128
    rng = np.random.default_rng(near)
    x = (1 + rng.random(200_000) * 2.0**-7).astype(np.float32)
    key = R.depth_split(x, np.zeros_like(x), False)[1].view(np.uint32)
    x = np.unique(x[key >> 16 == key[0] >> 16])
    band = np.tile(x[:-(-near // copies)], copies)[:near] * rng.choice([-1, 1], near).astype(np.float32)
    x0 = np.where(rng.random(T * d) < 0.5, rng.uniform(2, 3, T * d), rng.uniform(0.1, 0.5, T * d)).astype(np.float32)
    x0[rng.choice(T * d, near, replace=False)] = band
    x0 = x0.reshape(T, d)
    _, z1 = R.depth_split(x0, np.zeros_like(x0), False)
    above = int((np.abs(x0) > 1.5).sum())
    dev = torch.from_numpy(x0).cuda()
    for k in sorted({above + 1, above + (near + 1) // 2, above + near}):
        z0, idx, val = torch.empty_like(dev), torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, device="cuda")
        assert B.compress_unit_noalloc(dev, torch.zeros_like(dev), k, T * d, z0, idx, val) == k
        want = R.select_entries(z1, k)
        assert np.array_equal(idx.cpu().numpy(), want)
        assert np.array_equal(val.cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("T", [300, 2100])
@pytest.mark.parametrize("tiny", [0.0, 2.0**-70, 2.0**-30])
@pytest.mark.parametrize("keep", [(3, 10), (13, 20), (17, 20), (19, 20), (1, 1)])
def test_threshold_at_zero(keep, tiny, T, dtype):
    """A third of the keys normal, a third zero and a third zero or tiny, below the first window: the k-th among each of them, and zero
    with keys between it and the window and without."""
    d = 128
    rng = np.random.default_rng(9)
    diff = rng.standard_normal((T, d)).astype(np.float32)
    part = rng.integers(0, 3, (T, d))
    diff[part == 1] = 0
    diff[part == 2] *= tiny
    x0 = torch.from_numpy(diff).cuda().to(dtype)
    x1 = torch.zeros_like(x0)
    k = T * d * keep[0] // keep[1]
    z0, idx, val = torch.empty_like(x0), torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, dtype=dtype, device="cuda")
    assert B.compress_unit_noalloc(x0, x1, *keep, z0, idx, val) == k
    _, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), dtype == torch.bfloat16)
    want = R.select_entries(z1, k)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("T,kernels", [(17, 1), (500, 1), (1100, 1), (3072, 1), (3073, 4), (7936, 4)])
def test_everything_kept(T, kernels, dtype):
    """Zero keys among them; either side of the length up to which one kernel writes all of them."""
    d = 128
    x0, x1 = (torch.randint(-3, 4, (T, d), device="cuda", generator=torch.Generator("cuda").manual_seed(s)).to(dtype) for s in (1, 2))
    z0, idx, val = torch.empty_like(x0), torch.empty(T * d, dtype=torch.int32, device="cuda"), torch.empty(T * d, dtype=dtype, device="cuda")
    before = B.launch_count()
    assert B.compress_unit_noalloc(x0, x1, 1, 1, z0, idx, val) == T * d
    assert B.launch_count() - before == kernels
    want_z0, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), dtype == torch.bfloat16)
    assert np.array_equal(z0.float().cpu().numpy(), want_z0)
    assert np.array_equal(idx.cpu().numpy(), np.arange(T * d))
    assert np.array_equal(val.float().cpu().numpy(), z1.ravel())


@pytest.mark.parametrize("d,T,kernels", [(128, 4096, 1), (128, 4097, 1), (128, 7936, 1), (128, 7937, 6), (64, 16128, 1), (64, 16129, 6)])
@pytest.mark.parametrize("values,keep", [("normal", (1, 16)), ("normal", (3, 5)), ("three", (1, 3)), ("three", (3, 5)), ("equal", (1, 3)), ("equal", (3, 5))])
def test_four_words_per_thread(values, keep, d, T, kernels):
    """bf16 pairs in clusters of sixteen up to the most that a block's counts of 16 bits hold (31 tiles of 2 048, 63 of 1 024 positions), among them keys that
    are all equal or of three values; one tile more a block takes the separate kernels."""
    rng = np.random.default_rng(8)
    diff = {"normal": rng.standard_normal((T, d)), "three": rng.integers(-1, 2, (T, d)), "equal": np.ones((T, d))}[values].astype(np.float32)
    x0 = torch.from_numpy(diff).cuda().bfloat16()
    x1 = torch.zeros_like(x0)
    k = T * d * keep[0] // keep[1]
    z0, idx, val = torch.empty_like(x0), torch.empty(k, dtype=torch.int32, device="cuda"), torch.empty(k, dtype=torch.bfloat16, device="cuda")
    before = B.launch_count()
    assert B.compress_unit_noalloc(x0, x1, *keep, z0, idx, val) == k
    assert B.launch_count() - before == kernels
    _, z1 = R.depth_split(x0.float().cpu().numpy(), x1.float().cpu().numpy(), True)
    want = R.select_entries(z1, k)
    assert np.array_equal(idx.cpu().numpy(), want)
    assert np.array_equal(val.float().cpu().numpy(), z1.ravel()[want])
