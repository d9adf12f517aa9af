"""Shared coefficients staged where commit leaves them: readable before and after the commit in every mode, for both block
sizes and a length that is no whole box, and in the workspace when the arena has no room for them."""
import numpy as np
import pytest
import torch

from paper_2607_06519_b200 import synth

pytestmark = pytest.mark.gpu


def _all_z0(ctx, w):
    return [ctx.get_shared(0, p, h, v, w.T).view(torch.int16) for p in range(w.n_blocks) for h in range(w.n_kv_heads) for v in (0, 1)]


@pytest.mark.parametrize("block,rule", [(2, 0), (4, 0), (2, 1), (4, 1)])
def test_z0_is_readable_before_and_after_commit(block, rule):
    from paper_2607_06519_b200 import binding as B, runner

    w = synth.WORKLOADS["decode32k"].scaled(n_layers=8, n_kv_heads=4, n_q_heads=8, T=1101, n_needles=8, W=8, block_size=block, residual_rule=rule,
                                            name="in_place")
    pf = runner.Prefilled(w)
    small = runner.Prefilled(w, arena_bytes=4 << 20)  # the tails fit, the coefficients do not
    modes = np.array([[(p + h) % 3 for h in range(w.n_kv_heads)] for p in range(w.n_blocks)])
    for f in (small, pf):
        f.compress(0)
        f.probe(0, 0.0)
        f.ctx.set_modes(0, modes)
    before = _all_z0(pf.ctx, w)
    assert all(torch.equal(a, b) for a, b in zip(before, _all_z0(small.ctx, w)))
    with pytest.raises(B.FdkvError) as e:
        small.commit(0)
    assert e.value.code == 3  # arena full, and nothing was changed
    assert all(torch.equal(a, b) for a, b in zip(before, _all_z0(small.ctx, w)))
    pf.commit(0)
    assert all(torch.equal(a, b) for a, b in zip(before, _all_z0(pf.ctx, w)))
    assert pf.ctx.device_status() == 0
