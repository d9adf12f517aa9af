"""Decode over 8-bit rows at the edges of its tiles (256 tokens, two 16-token slices per warp) and of its list windows (12 entries
per lane and list in registers, more loaded when used): shorter than a tile, a tile and its neighbours, ranges that start
inside a unit, both walking directions, sparse to dense lists."""
import numpy as np
import pytest
import torch

from gpu_util import TOL, f32, vector_errors
from oracle import fdkv_ref_fp8 as R8
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,T,den", [(1, 15, 2), (2, 255, 8), (1, 256, 2), (2, 257, 4), (3, 287, 16), (150, 300, 8), (2, 9001, 8), (1, 40000, 32)])
def test_fp8_tile_edges(hkv, T, den):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv * 4, T=T, n_needles=1, W=1, n_steps=1, row_format=1,
                                            keep_num=1, keep_den=den, name="fp8_tiles")
    pf = runner.Prefilled(w, max_tail=1)
    modes = np.array([[(1 + 2 * h) % 3 for h in range(hkv)]])
    pf.prefill(0, modes)
    for layer in range(2):
        q = pf.decode_q(layer, 0)
        out = f32(pf.ctx.decode_attn(layer, q, out_dtype=0))[0]
        torch.cuda.synchronize()
        for h in {0, hkv // 2, hkv - 1}:
            u = R8.UnitFp8(*synth.unit_tensor(w, 0, 0, h, False), *synth.unit_tensor(w, 0, 0, h, True), True, 1, den)
            ref = u.attend(int(modes[0, h]), layer, f32(q)[0][h * 4:(h + 1) * 4])
            assert vector_errors(out[h * 4:(h + 1) * 4], ref).max() <= TOL["bf16"], (layer, h)
    assert pf.ctx.device_status() == 0
    pf.ctx.close()
