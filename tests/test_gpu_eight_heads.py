"""Eight query heads per KV head (bf16, head_dim 128): the weights of the second product carry as many bits as with four.

A weight acts as its bf16 rounding plus the bf16 rounding of the remainder, off by at most 2^-18; the errors of a vector's
tokens are independent, so the vector is off by about that much of its largest element, three or four times it where the
channels' maximum falls on a small element, and float32 logits add as much again: 3e-5.  (With the rounding alone, 2^-9 a
weight: up to 2e-2, and different with every cut of the tokens.)"""
import numpy as np
import pytest

from gpu_util import f32, oracle_unit, vector_errors
from oracle import fdkv_ref_b4 as R4
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu
BOUND = 3e-5


# clusters (the first three), a unit's blocks whole, ranges that straddle units, one block; more sequences than the short list of tails holds
@pytest.mark.parametrize("group", [4, 8])
@pytest.mark.parametrize("hkv,T,batch,tail", [(8, 1000, 1, 0), (2, 1024, 1, 130), (1, 37, 1, 1), (3, 4099, 1, 2), (8, 4096, 1, 0), (8, 1500, 6, 0), (2, 32768, 1, 0), (2, 65, 70, 0)])
def test_entries(hkv, group, T, batch, tail):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv * group, T=T, batch=batch, n_needles=2, W=1, n_steps=max(tail, 1),
                                            name="eight")
    pf = runner.Prefilled(w, max_tail=max(tail, 1))
    modes = np.array([[(1 + h) % 3 for h in range(hkv)]])
    for b in range(batch):
        pf.prefill(b, modes)
    worst = 0.0
    for layer in range(2):
        for step in range(max(tail, 1)):
            q = pf.decode_q(layer, step)
            out = pf.ctx.decode_attn(layer, q, *(pf.new_rows(layer, step) if tail else (None, None)), out_dtype=0)
        for b in {0, batch - 1}:
            for h in range(min(3, hkv)):
                u = oracle_unit(w, b, 0, h)
                for step in range(tail):
                    kn, vn = pf.new_rows(layer, step)
                    u.append(layer, f32(kn)[b, h], f32(vn)[b, h])
                ref = u.attend(int(modes[0, h]), layer, f32(q)[b][h * group:(h + 1) * group])
                worst = max(worst, float(vector_errors(f32(out)[b][h * group:(h + 1) * group], ref).max()))
    print("worst", worst)
    assert worst <= BOUND, worst
    assert pf.ctx.device_status() == 0
    pf.ctx.close()


@pytest.mark.parametrize("T", [700, 5000])
def test_blocks_of_four(T):
    hkv, group = 3, 8
    w = synth.WORKLOADS["decode32k_b4"].scaled(n_layers=4, n_kv_heads=hkv, n_q_heads=hkv * group, T=T, n_needles=2, W=1, n_steps=1, name="eight4")
    pf = runner.Prefilled(w)
    modes = np.array([[0, 1, 2]])
    pf.prefill(0, modes)
    for layer in (0, 3):
        q = pf.decode_q(layer, 0)
        out = f32(pf.ctx.decode_attn(layer, q, out_dtype=0))[0]
        for h in range(hkv):
            u = R4.Unit4(synth.block_tensor(w, 0, 0, h, False), synth.block_tensor(w, 0, 0, h, True), True, w.keep_num, w.keep_den)
            ref = u.attend(int(modes[0, h]), layer, f32(q)[0][h * group:(h + 1) * group])
            assert vector_errors(out[h * group:(h + 1) * group], ref).max() <= BOUND, (layer, h)
    assert pf.ctx.device_status() == 0
    pf.ctx.close()
