"""Short contexts: a unit's thread blocks as one cluster, from one block to eight, with and without appended rows (the appended
row of a call is not read back from the tail), first and last row of a 16-row slice and of a 128-row box, both row formats."""
import numpy as np
import pytest
import torch

from gpu_util import TOL, f32, oracle_unit, vector_errors
from oracle import fdkv_ref_fp8 as R8
from paper_2607_06519_b200 import binding as B
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("hkv,group,T,n", [(1, 4, 1, 2), (2, 1, 17, 18), (1, 2, 130, 3), (8, 4, 513, 129), (3, 4, 1000, 2), (16, 2, 300, 2)])
def test_generated_rows(hkv, group, T, n, rows):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv * group, T=T, n_needles=1, W=1, n_steps=n, row_format=rows,
                                            name="clusters")
    pf = runner.Prefilled(w, max_tail=n)
    modes = np.array([[(1 + h) % 3 for h in range(hkv)]])
    pf.prefill(0, modes)
    units = {}
    for h in {0, hkv - 1}:
        if rows:
            units[h] = R8.UnitFp8(*synth.unit_tensor(w, 0, 0, h, False), *synth.unit_tensor(w, 0, 0, h, True), True, w.keep_num, w.keep_den)
        else:
            units[h] = oracle_unit(w, 0, 0, h)
    for step in range(n):
        for layer in range(2):
            q = pf.decode_q(layer, step)
            kn, vn = pf.new_rows(layer, step)
            out = pf.ctx.decode_attn(layer, q, kn, vn)
            for h, u in units.items():
                u.append(layer, f32(kn)[0, h], f32(vn)[0, h])
                if step in (0, 1, 15, 16, 17, 127, 128) or step == n - 1:
                    ref = u.attend(int(modes[0, h]), layer, f32(q)[0][h * group:(h + 1) * group])
                    assert vector_errors(f32(out)[0][h * group:(h + 1) * group], ref).max() <= TOL["bf16"], (step, layer, h)
    assert pf.ctx.device_status() == 0


@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("hkv,T,tail", [(8, 1024, 0), (8, 1024, 3), (8, 1040, 129), (8, 1025, 1), (8, 1536, 0), (4, 2047, 0), (8, 127, 40), (2, 4096, 0)])
def test_whole_tiles(hkv, T, tail, rows):
    """Blocks that take whole tiles, the last one with the remainder and the tail: at and beside whole tiles for eight blocks."""
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv * 2, T=T, n_needles=1, W=1, n_steps=max(tail, 1), row_format=rows,
                                            name="clusters_cut")
    pf = runner.Prefilled(w, max_tail=max(tail, 1))
    modes = np.array([[(1 + h) % 3 for h in range(hkv)]])
    pf.prefill(0, modes)
    for layer in range(2):
        for step in range(max(tail, 1)):
            q = pf.decode_q(layer, step)
            rows_new = pf.new_rows(layer, step) if tail else (None, None)
            out = pf.ctx.decode_attn(layer, q, *rows_new)
        for h in (0, hkv - 1):
            if rows:
                u = R8.UnitFp8(*synth.unit_tensor(w, 0, 0, h, False), *synth.unit_tensor(w, 0, 0, h, True), True, w.keep_num, w.keep_den)
            else:
                u = oracle_unit(w, 0, 0, h)
            for step in range(tail):
                kn, vn = pf.new_rows(layer, step)
                u.append(layer, f32(kn)[0, h], f32(vn)[0, h])
            ref = u.attend(int(modes[0, h]), layer, f32(q)[0][h * 2:(h + 1) * 2])
            assert vector_errors(f32(out)[0][h * 2:(h + 1) * 2], ref).max() <= TOL["bf16"], (layer, h)
    assert pf.ctx.device_status() == 0
    pf.ctx.close()


@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("rule", [0, 1])
@pytest.mark.parametrize("hkv,T,tail", [(2, 256, 0), (2, 2048, 0), (2, 2048, 2), (32, 2000, 0), (32, 2000, 2), (30, 2800, 0)])
def test_full_scratch_behind_the_last_tiles(hkv, T, tail, rule, rows):
    """Every position kept, one to three tiles a block: the last ones fill all of the scratch that the next tile's entries, the state put
    aside before a tail and the merge are written over.  The same bits from every call, within the tolerance of the oracle's."""
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=2, n_kv_heads=hkv, n_q_heads=hkv, T=T, n_needles=1, W=1, n_steps=max(tail, 1), row_format=rows,
                                            residual_rule=rule, keep_num=1, keep_den=1, name="full_scratch")
    pf = runner.Prefilled(w, max_tail=max(tail, 1))
    pf.prefill(0, np.ones((1, hkv), np.int64))
    for layer in range(2):
        for step in range(tail):
            pf.ctx.decode_attn(layer, pf.decode_q(layer, step), *pf.new_rows(layer, step))
        q = pf.decode_q(layer, 0)
        launches = B.launch_count()
        first = pf.ctx.decode_attn(layer, q).clone()
        assert B.launch_count() == launches + 1  # (clusters: no kernel that joins)
        for _ in range(10):
            assert torch.equal(pf.ctx.decode_attn(layer, q), first)
        for h in (0, hkv - 1):
            if rows:
                u = R8.UnitFp8(*synth.unit_tensor(w, 0, 0, h, False), *synth.unit_tensor(w, 0, 0, h, True), True, 1, 1)
            else:
                u = oracle_unit(w, 0, 0, h)
            if rule:
                u.use_tokens(np.arange(T))
            for step in range(tail):
                kn, vn = pf.new_rows(layer, step)
                u.append(layer, f32(kn)[0, h], f32(vn)[0, h])
            ref = u.attend(1, layer, f32(q)[0][h:h + 1])
            assert vector_errors(f32(first)[0][h:h + 1], ref).max() <= TOL["bf16"], (layer, h)
    assert pf.ctx.device_status() == 0
    pf.ctx.close()
