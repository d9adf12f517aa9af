"""What this library is measured on: the calls a serving program makes, from one short tensor pair to a 128k context.

A case is a plain dict.  Its "path" says which calls one pass makes:

  unit      binding.compress_unit_noalloc on one [T, head_dim] tensor pair (a caller without a context)
  decode    one attention step: Context.decode_attn of every layer over committed sequences (or, with io = "host", one
            Context.decode_step_host on pinned host buffers)
  generate  `new` tokens: the tails go back to their length before the pass (Context.set_tail_len), then `new` steps of
            Context.decode_attn that append a row to every layer and attend
  prefill   one prompt on a slot that served another one: Context.reset, compress_prefill, probe, route_budget, commit, then
            `new` generated tokens, Context.fold_tail of them (`fold`), and one attention step
"""
from __future__ import annotations

import numpy as np
import torch

from paper_2607_06519_b200 import binding as B
from paper_2607_06519_b200 import synth

DEVICE = "cuda:0"

# Shape of the repository's workloads (32 query heads on 8 KV heads, head_dim 128); a case overrides what differs.
_BASE = {"path": "decode", "layers": 32, "q_heads": 32, "kv_heads": 8, "head_dim": 128, "dtype": "bf16", "batch": 1, "T": 32768,
         "keep_den": 16, "rule": "entries", "block": 2, "rows": "storage", "probes": 64, "tail": 0, "new": 0, "fold": False,
         "io": "device", "budget": 0.6}


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # one short tensor pair from a caller that owns no context: a handful of launches on little data
        {"name": "unit_509", "path": "unit", "T": 509, "head_dim": 128, "dtype": "bf16", "keep_den": 16},
        # a short conversation that generates, every layer its own small call
        _case("generate_2k", path="generate", T=2047, tail=37, new=4),
        # the repository's headline: one decode step of 32 layers over a 32k context
        _case("decode_32k"),
        # a batch of ragged long sequences that generates (depth cut to 8 layers: every layer's call is the same)
        _case("generate_32k_batch8", path="generate", layers=8, batch=8, tail=64, new=2),
        # the longest context of the repository's workloads (depth cut to 8 layers)
        _case("decode_128k", layers=8, T=131072, keep_den=32),
        # blocks of four layers with probe-scored tokens (the paper's default pairing), driven from host buffers
        _case("decode_32k_block4_tokens_host", rule="tokens", block=4, io="host"),
        # committed rows as 8-bit floats
        _case("decode_32k_e4m3", rows="e4m3"),
        # time to first token of a 32k prompt
        _case("prefill_32k", path="prefill"),
        # the paper's default pairing on a ragged prompt of usual length
        _case("prefill_8k_block4_tokens", path="prefill", T=8191, rule="tokens", block=4, budget=0.4),
        # blocks of four layers with the entry rule
        _case("prefill_12k_block4", path="prefill", T=12289, block=4, budget=0.45),
        # a chat turn: a short prompt, sixteen generated tokens, the periodic refresh, one more step
        _case("turn_1k", path="prefill", T=1024, new=16, fold=True),
        # float32 storage and head_dim 64, as the correctness workload has them, on a longer prompt
        _case("prefill_4k_f32", path="prefill", layers=4, q_heads=4, kv_heads=2, head_dim=64, dtype="f32", T=4099, keep_den=8,
              probes=32, budget=0.65),
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, spread over its logarithm, as likely odd as not."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    path = rng.choice(["unit", "generate", "decode", "decode", "prefill", "prefill"])
    if path == "unit":
        d = rng.choice([64, 128])
        return {"path": "unit", "T": _size(rng, 64, (1 << 20) // d), "head_dim": d, "dtype": rng.choice(["bf16", "f32"]),
                "keep_den": rng.choice([8, 16, 32])}
    c = dict(_BASE, path=path, block=rng.choice([2, 2, 4]), rule=rng.choice(["entries", "entries", "tokens"]),
             keep_den=rng.choice([8, 16, 32]), layers=rng.choice([4, 8, 16, 32]))
    c["kv_heads"] = rng.choice([2, 4, 8])
    c["q_heads"] = c["kv_heads"] * rng.choice([1, 2, 4, 4, 8])
    if rng.random() < 0.2:  # the portable kernels: shorter prompts, fewer layers
        c.update(dtype=rng.choice(["f32", "bf16"]), head_dim=64, layers=rng.choice([4, 8]), kv_heads=2, q_heads=rng.choice([2, 4, 8]),
                 T=_size(rng, 256, 6000), probes=32)
    elif path == "prefill":
        c["T"] = _size(rng, 512, 28000)
        c["probes"] = rng.choice([32, 64, 128])
    else:
        c["T"] = _size(rng, 512, 131072 if c["layers"] <= 8 else 32768)
    if path == "generate":
        # as many sequences as keep tokens x layers x steps in total below the listed batch's
        new = rng.randint(1, 4)
        c["T"] = min(c["T"], 3_000_000 // (c["layers"] * new))
        room = 3_000_000 // (c["T"] * c["layers"] * new)
        c.update(batch=min(room, rng.choice([1, 2, 3, 5, 8])), tail=rng.randint(0, 200), new=new)
    if path == "decode" and c["head_dim"] == 128 and c["q_heads"] <= 4 * c["kv_heads"]:
        c["rows"] = rng.choice(["storage", "storage", "e4m3"])
    if path == "decode":
        c["io"] = rng.choice(["device", "host"])
    if path == "prefill":
        c["budget"] = (0.4 if c["rule"] == "tokens" else 0.45) if c["block"] == 4 else 0.65
        if c["rule"] == "entries" and c["T"] <= 4096 and rng.random() < 0.5:
            c.update(T=(c["T"] + 15) // 16 * 16, new=16, fold=True)
    return c


# ---------------------------------------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    return g


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _lengths(c):
    """Prompt length of every sequence of a batch: the longest first, down to about half of it, odd ones among them."""
    return [max(16, c["T"] - b * c["T"] // (2 * c["batch"]) - b) for b in range(c["batch"])]


def _depth_chain(g, T, heads, d, layers, dtype):
    """The rows [T, heads, d] of `layers` neighbouring layers: synth's recipe (log-normal channel scales, correlated layers,
    a few tokens whose deviation is eight times as large), drawn on the device."""
    rho = 0.7 + 0.25 * torch.rand((), generator=g, device=DEVICE)
    beta = torch.sqrt(1.0 - rho * rho)
    sigma = torch.exp(torch.randn((heads, d), generator=g, device=DEVICE))
    needle = torch.ones((T, heads), device=DEVICE)
    needle.scatter_(0, torch.randint(T, (max(1, T // 512), heads), generator=g, device=DEVICE), 8.0)
    u = torch.randn((T, heads, d), generator=g, device=DEVICE)
    out = [(u * sigma).to(dtype)]
    for _ in range(layers - 1):
        n = torch.randn((T, heads, d), generator=g, device=DEVICE)
        n.mul_(needle.unsqueeze(2)).mul_(beta)
        u = u.mul_(rho).add_(n)
        out.append((u * sigma).to(dtype))
    return out


def _prompt(c, g, T):
    k, v = [], []
    for _ in range(c["layers"] // c["block"]):
        k += _depth_chain(g, T, c["kv_heads"], c["head_dim"], c["block"], _dtype(c))
        v += _depth_chain(g, T, c["kv_heads"], c["head_dim"], c["block"], _dtype(c))
    probe_q = [torch.randn((min(c["probes"], T), c["q_heads"], c["head_dim"]), generator=g, device=DEVICE).to(_dtype(c))
               for _ in range(c["layers"])]
    return k, v, probe_q


def _probe_positions(c, T):
    n = min(c["probes"], T)
    return np.arange(T - n, T, dtype=np.int32)


def _normal(c, g, *shape):
    return torch.randn(shape, generator=g, device=DEVICE).to(_dtype(c))


def _context(c):
    cfg = B.Config(c["layers"], c["q_heads"], c["kv_heads"], c["head_dim"], c["batch"], c["T"], c["tail"] + c["new"] + 1,
                   B.BF16 if c["dtype"] == "bf16" else B.F32, 1, c["keep_den"],
                   B.RESIDUAL_TOKENS if c["rule"] == "tokens" else B.RESIDUAL_ENTRIES, c["block"], c["new"] if c["fold"] else 0,
                   1 if c["rows"] == "e4m3" else 0)
    return B.Context(cfg, device=DEVICE)


def _steps(c, g, n, append):
    """Queries, new rows and output buffers of n attention steps, per layer."""
    L, b = c["layers"], c["batch"]
    s = {"q": _normal(c, g, n, L, b, c["q_heads"], c["head_dim"])}
    s["out"] = torch.empty_like(s["q"])
    if append:
        s["k"] = _normal(c, g, n, L, b, c["kv_heads"], c["head_dim"])
        s["v"] = _normal(c, g, n, L, b, c["kv_heads"], c["head_dim"])
    # one tensor object per layer and step: what a model's layers hand over
    return {name: [list(step.unbind(0)) for step in t.unbind(0)] for name, t in s.items()}, s


def prepare(case, seed):
    c, g = case, _gen(seed)
    if c["path"] == "unit":
        T, d, k = c["T"], c["head_dim"], c["T"] * c["head_dim"] // c["keep_den"]
        x0, x1 = (x[:, 0].contiguous() for x in _depth_chain(g, T, 1, d, 2, _dtype(c)))
        return {"case": c, "x0": x0, "x1": x1, "z0": torch.empty_like(x0), "idx": torch.empty(k, dtype=torch.int32, device=DEVICE),
                "val": torch.empty(k, dtype=_dtype(c), device=DEVICE)}
    ctx = _context(c)
    s = {"case": c, "ctx": ctx}
    if c["path"] == "prefill":
        s["k"], s["v"], s["probe_q"] = _prompt(c, g, c["T"])
        s["pos"] = _probe_positions(c, c["T"])
        exact = 2 * c["layers"] * c["kv_heads"] * c["T"] * c["head_dim"] * (2 if c["dtype"] == "bf16" else 4)
        s["budget"] = int(c["budget"] * exact)
        s["steps"], s["out"] = _steps(c, g, c["new"] + 1, c["new"] > 0)
        return s
    for b, T in enumerate(_lengths(c)):  # committed sequences, routed half shared, a third residual, the rest exact
        k, v, probe_q = _prompt(c, g, T)
        ctx.compress_prefill(b, 0, ctx.n_pairs, T, k, v)
        _, scores = ctx.probe(b, 0, ctx.n_pairs, probe_q, _probe_positions(c, T), 0.0)
        ctx.set_modes(b, synth.quota_modes(scores[..., 0].cpu().numpy()))
        ctx.commit(b)
    if c["path"] == "generate":
        tail, _ = _steps(c, g, 1, False)
        rows = _normal(c, g, 2, c["tail"], c["layers"], c["batch"], c["kv_heads"], c["head_dim"])
        for j in range(c["tail"]):
            for l in range(c["layers"]):
                ctx.decode_attn(l, tail["q"][0][l], rows[0, j, l], rows[1, j, l], out=tail["out"][0][l])
    s["steps"], s["out"] = _steps(c, g, max(1, c["new"]), c["path"] == "generate")
    if c["io"] == "host":
        s["host_q"] = s["out"]["q"][0].cpu().pin_memory()
        s["host_out"] = torch.empty_like(s["host_q"]).pin_memory()
    return s


# ---------------------------------------------------------------------------------------------------------------- a pass
def _attend(ctx, steps, j, append):
    q, out = steps["q"][j], steps["out"][j]
    if append:
        k, v = steps["k"][j], steps["v"][j]
        for l in range(len(q)):
            ctx.decode_attn(l, q[l], k[l], v[l], out=out[l])
    else:
        for l in range(len(q)):
            ctx.decode_attn(l, q[l], out=out[l])


def run(state):
    s, c = state, state["case"]
    if c["path"] == "unit":
        B.compress_unit_noalloc(s["x0"], s["x1"], 1, c["keep_den"], s["z0"], s["idx"], s["val"])
        return s["z0"], s["idx"], s["val"]
    ctx, steps = s["ctx"], s["steps"]
    if c["path"] == "decode":
        if c["io"] == "host":
            return ctx.decode_step_host(s["host_q"], None, None, s["host_out"], B.BF16 if c["dtype"] == "bf16" else B.F32)
        _attend(ctx, steps, 0, False)
        return s["out"]["out"]
    if c["path"] == "generate":
        for b in range(c["batch"]):
            ctx.set_tail_len(b, c["tail"])
        for j in range(c["new"]):
            _attend(ctx, steps, j, True)
        return s["out"]["out"]
    ctx.reset()
    ctx.compress_prefill(0, 0, ctx.n_pairs, c["T"], s["k"], s["v"])
    _, scores = ctx.probe(0, 0, ctx.n_pairs, s["probe_q"], s["pos"], 0.0)
    _, _, modes = ctx.route_budget(0, s["budget"])
    ctx.commit(0)
    for j in range(c["new"]):
        _attend(ctx, steps, j, True)
    if c["fold"]:
        ctx.fold_tail(0, c["new"])
    _attend(ctx, steps, c["new"], False)
    return scores, modes, s["out"]["out"]


# --------------------------------------------------------------------------------------------------- floors and tolerances
def work(case):
    c = case
    if c["path"] == "unit":
        e, n = (2 if c["dtype"] == "bf16" else 4), c["T"] * c["head_dim"]
        return {"bytes": 3 * n * e + n // c["keep_den"] * (4 + e), "flops": 4 * n}
    e = 2 if c["dtype"] == "bf16" else 4
    L, d, H, G = c["layers"], c["head_dim"], c["kv_heads"], c["q_heads"] // c["kv_heads"]
    row_e = 1 if c["rows"] == "e4m3" else e

    def step(T, tail, resid):
        """One attention step of one sequence: dense rows, the residual units' entries (a value and a 16-bit position) or token
        rows, the tail; queries in, outputs out."""
        kept = T * d // c["keep_den"]
        per_head = 2 * T * d * row_e + resid * 2 * kept * (e + 2 if c["rule"] == "entries" else e) + 2 * tail * d * e
        return L * (H * per_head + 2 * c["q_heads"] * d * e), L * 4 * c["q_heads"] * (T + tail) * d

    if c["path"] in ("decode", "generate"):
        total = [0, 0]
        for T in _lengths(c):
            for j in range(max(1, c["new"])):
                by, fl = step(T, c["tail"] + j + 1 if c["path"] == "generate" else 0, 0.35)
                total[0] += by
                total[1] += fl
        return {"bytes": total[0], "flops": total[1]}
    # prefill: every layer's K and V once, the compressed cache once, and the attention steps over it.  The probe's error is a
    # quadratic form of the head_dim x head_dim second moments once there are more probe rows than channels; the token rule's
    # scores need every row.
    n = 2 * L * H * c["T"] * d
    total = [n * e + c["budget"] * n * e, 3 * n]
    units, rows = L // c["block"] * H, c["block"] * G * min(c["probes"], c["T"])
    total[1] += 2 * units * c["T"] * d * (rows if c["rule"] == "tokens" else 2 * min(rows, d * (c["block"] if c["block"] == 4 else 1)))
    for j in range(c["new"] + 1):
        by, fl = step(c["T"], min(j + 1, c["new"]), 0.35)
        total[0] += by
        total[1] += fl
    return {"bytes": total[0], "flops": total[1]}


def tolerance(case):
    if case["path"] == "unit":
        return "exact"  # bit patterns: one addition, one multiplication and one rounding per value, ties to the lowest index
    if case["dtype"] == "f32":
        # against float64 the outputs are off by 1.6e-7 (largest 2.0e-6) and the probe's errors, sums over thousands of keys, by 1e-6
        return {"rel": 4e-6, "max": 1e-5, "differ": 0.0}
    # the rounding of the outputs to bf16: 1.5e-3 (largest 3.8e-3) against float64; before it they are off by 5e-7
    return {"rel": 6e-3, "max": 1.6e-2, "differ": 0.0}
