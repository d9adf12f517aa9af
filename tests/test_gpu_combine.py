"""The kernel that joins a query head's split-K parts: one part, a part per thread block of the whole device (more than one
round of 32), every group size, and the form for many heads."""
import numpy as np
import pytest
import torch

from gpu_util import TOL, f32, oracle_layer_out, oracle_unit, vector_errors
from paper_2607_06519_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hkv,group,T,batch", [(1, 1, 19001, 1), (1, 8, 33, 1), (2, 4, 4700, 1), (8, 4, 130, 6), (8, 8, 129, 3)])
def test_parts_join(hkv, group, T, batch):
    from paper_2607_06519_b200 import runner

    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv * group, T=T, batch=batch, n_needles=4, W=8, name="combine")
    pf = runner.Prefilled(w)
    modes = np.array([[(1 + h) % 3 for h in range(hkv)]])
    for b in range(batch):
        pf.prefill(b, modes)
    for layer in range(2):
        q = pf.decode_q(layer, 0)
        for od in (0, 1):
            out = f32(pf.ctx.decode_attn(layer, q, out_dtype=od))
            for b in {0, batch - 1}:
                units = {h: oracle_unit(w, b, 0, h) for h in range(hkv)}
                err = vector_errors(out[b], oracle_layer_out(units, modes[0], w, layer, f32(q)[b]))
                assert err.max() <= TOL["bf16"], (layer, od, b, float(err.max()))
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("hkv,T", [(8, 5003), (7, 6007), (5, 4801)])
def test_parts_beside_the_rounds(hkv, T):
    """About 18, 21 and 29 parts per head: below, beside and above the 20 that are joined in one round."""
    from paper_2607_06519_b200 import runner

    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv, T=T, n_needles=4, W=8, name="combine_rounds")
    pf = runner.Prefilled(w)
    modes = np.array([[h % 3 for h in range(hkv)]])
    pf.prefill(0, modes)
    q = pf.decode_q(1, 0)
    out = f32(pf.ctx.decode_attn(1, q))
    for h in (0, hkv - 1):
        ref = oracle_unit(w, 0, 0, h).attend(int(modes[0, h]), 1, f32(q)[0][h:h + 1])
        assert vector_errors(out[0][h:h + 1], ref).max() <= TOL["bf16"], h
    assert pf.ctx.device_status() == 0
