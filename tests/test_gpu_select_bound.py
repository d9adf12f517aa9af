"""The selection's bound is a guess from a sample of the tokens: inputs that mislead it must give the same lists.  Also the edges
of the candidate chunks (16 to 64 tokens), for both block sizes, storage types and head dimensions."""
import numpy as np
import pytest
import torch

from gpu_util import check_compression
from oracle import fdkv_ref as R
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
