"""Page-locked tables and scores of a context: contexts of several sizes opened, used and closed from two threads on streams of
their own (blocks of closed contexts serve the next ones), one closed with its scores still on their way, and the smallest
lambda that fits."""
import threading

import numpy as np
import pytest
import torch

from oracle import fdkv_ref as R
from paper_2607_06519_b200 import runner, synth

pytestmark = pytest.mark.gpu


def _once(T, hkv, share, leave_early=False):
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=4, n_kv_heads=hkv, n_q_heads=hkv * 2, T=T, n_needles=2, W=8, n_steps=1, name="host_tables")
    pf = runner.Prefilled(w, max_tail=1)
    pf.compress(0)
    if leave_early:
        pf.ctx.probe(0, 0, 2, pf.upload_probe_q(0), synth.probe_positions(w), 0.0)
        pf.ctx.close()
        return None
    _, scores = pf.probe(0, 0.0)
    one = 4 * T * 128 * 2
    n = 2 * hkv
    _, lam, modes = pf.ctx.route_budget(0, int(share * n * one))
    pf.commit(0)
    out = pf.ctx.decode_attn(3, pf.decode_q(3, 0))
    res = (scores, lam, modes.numpy().copy(), out.float().cpu().numpy())
    assert pf.ctx.device_status() == 0
    pf.ctx.close()
    return res


def test_contexts_of_two_threads():
    cases = [(300, 1, 0.55), (700, 4, 0.62), (257, 2, 0.7), (1200, 8, 0.6)]
    want = [_once(*c) for c in cases]
    got, failed = {}, []

    def work(who):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for r in range(3):
                    for i in range(len(cases)):
                        j = (i + 2 * who + r) % len(cases)
                        if r == 1:
                            _once(*cases[j], leave_early=True)
                        got[who, r, j] = _once(*cases[j])
        except BaseException as e:  # (reported by the test's own thread)
            failed.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for (_, _, j), res in got.items():
        for a, b in zip(res, want[j]):
            assert np.array_equal(a, b), j


@pytest.mark.parametrize("hkv", [1, 4])
def test_smallest_lambda(hkv):
    """Below the lambda that is returned (by a relative 1e-6, above the float32 rounding of the scores that the caller gets) the
    routing does not fit; above it it is the returned one and fits."""
    w = synth.WORKLOADS["decode32k"].scaled(n_layers=8, n_kv_heads=hkv, n_q_heads=hkv * 2, T=500, n_needles=2, W=8, n_steps=1, name="scan")
    pf = runner.Prefilled(w, max_tail=1)
    pf.compress(0)
    _, scores = pf.probe(0, 0.0)
    e = scores.reshape(-1, 2)
    n, one = 4 * hkv, 4 * 500 * 128 * 2
    om = R.omega(500, 128, 2, w.k_keep)

    def route(lam):
        return np.argmin(np.stack([e[:, 0] + lam * om[0], e[:, 1] + lam * om[1], np.full(n, lam * om[2])]), axis=0)

    def size(m):
        return sum(om[i] for i in m) * one

    seen = set()
    for share in np.linspace(0.45, 1.05, 61):
        budget = int(share * n * one)
        fits, lam, modes = pf.ctx.route_budget(0, budget)
        assert fits == (size([0] * n) <= budget)
        if not fits:
            continue
        got = modes.numpy().reshape(-1)
        seen.add(tuple(got))
        assert size(got) <= budget and np.array_equal(got, route(lam * (1 + 1e-6)))
        if lam > 0:
            assert size(route(lam * (1 - 1e-6))) > budget, share
    assert len(seen) > n
    pf.ctx.close()
