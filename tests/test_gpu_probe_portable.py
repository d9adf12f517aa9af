"""The portable probe kernel at the edges of its tiles (64 tokens) and turns (32 probe rows), both storage types it serves, both
head dimensions and block sizes."""
import numpy as np
import pytest

from oracle import fdkv_ref as R
from oracle import fdkv_ref_b4 as R4
from paper_2607_06519_b200 import runner, synth

import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [2, 4])
@pytest.mark.parametrize("dtype,d", [("f32", 64), ("f32", 128), ("bf16", 64)])
@pytest.mark.parametrize("group,T,W", [(1, 1, 1), (2, 63, 8), (1, 64, 16), (1, 65, 17), (2, 129, 16), (4, 200, 33), (8, 1000, 64)])
def test_probe_errors(block, dtype, d, group, T, W):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=block, n_kv_heads=2, n_q_heads=2 * group, head_dim=d, T=T, W=W, n_needles=min(T, 2), keep_num=1,
                                            keep_den=7, dtype=dtype, block_size=block, name="portable")
    pf = runner.Prefilled(w)
    pf.compress(0)
    _, scores = pf.ctx.probe(0, 0, 1, pf.upload_probe_q(0), synth.probe_positions(w), 0.0)
    scores = scores.cpu().numpy()
    pq = [synth.probe_q(w, 0, l) for l in range(block)]
    bf16 = dtype == "bf16"
    for h in range(2):
        if block == 4:
            u = R4.Unit4(synth.block_tensor(w, 0, 0, h, False), synth.block_tensor(w, 0, 0, h, True), bf16, 1, 7)
            want = R4.probe_error4(u.dev["k"], u.kept["k"], pq, group, h, synth.probe_positions(w))
        else:
            u = R.Unit(*synth.unit_tensor(w, 0, 0, h, False), *synth.unit_tensor(w, 0, 0, h, True), bf16, 1, 7)
            want = R.probe_error(u.z1["k"], u.kept["k"], pq[0], pq[1], group, h, synth.probe_positions(w))
        # float32 dot products of up to 128 terms, squared and summed: 2 x 128 x 2^-24, with room for the sums
        np.testing.assert_allclose(scores[0, h], want, rtol=3e-5, atol=1e-12)
    assert pf.ctx.device_status() == 0
