"""The workloads this framework is timed on: speculative decode rounds, plain decode steps and prompt prefill.

A case is one of
  mode "round"    one speculative round of a serving loop through ``Engine.round_host``: the accept pattern of the round
                  comes from the host (the seeded truncated-geometric pattern, success rate 0.68), k draft steps, one
                  verify pass over k + 1 positions, accept / rollback, and the accept lengths and emitted tokens come
                  back to the host.  k = 0 is plain autoregressive decoding with the full model.
  mode "sampled"  the same round at temperature > 0: the caller refills the uniforms on the device, the library decides
                  the accept lengths itself.
  mode "prefill"  a new request: reset, then ``Engine.prefill`` of the prompts; every prompt's first token is read back.

Models are the shapes of ``hs_inputs.CONFIGS`` with random weights of the documented distributions.  Decode cases hold
random contexts (uniform +-0.5 state, N(0, 1) conv inputs and KV rows, as the tests inject them); a loop that has
generated its share of tokens starts over from its first context, so a state can be run any number of times.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import hs_inputs as hi
from paper_2605_01106_b200 import binding as hs

TEMPERATURE = 0.8
PATTERN = 512                       # rounds of accept pattern kept on the host


# ------------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------------
def _case(mode, model, batch, lo, hi_, k, replay=False, plan="component", name=None):
    """lo, hi: shortest and longest context (decode) or prompt (prefill) of the batch, in tokens."""
    c = {"mode": mode, "model": model, "batch": batch, "lo": lo, "hi": hi_, "k": k, "replay": replay, "plan": plan}
    return dict(c, name=name) if name else c


def listed():
    return [
        # smallest call: the two-layer model, one sequence, a short context - launches and latency only
        _case("round", "cfg1_tiny", 1, 64, 64, 2, name="tiny-b1-k2"),
        # interactive use of the 0.5B-class hybrid: plain decoding, then the same with two drafts per round
        _case("round", "cfg2_0p5b", 1, 512, 512, 0, name="0.5b-b1-plain"),
        _case("round", "cfg2_0p5b", 1, 512, 512, 2, name="0.5b-b1-k2"),
        # a few users with contexts of odd, different lengths, sampled at a temperature
        _case("sampled", "cfg2_0p5b", 3, 177, 901, 4, name="0.5b-b3-k4-sampled"),
        # interactive use of the 3B-class hybrid with long drafts, and a small batch of it with rollback by replay
        _case("round", "cfg3_3b", 1, 2048, 2048, 4, name="3b-b1-k4"),
        _case("round", "cfg3_3b", 8, 1500, 2048, 4, replay=True, name="3b-b8-k4-replay"),
        # the sequential (Gated DeltaNet) hybrid: default draft, and a layer-skipping draft on a small ragged batch
        _case("round", "cfg4_seq", 1, 1024, 1024, 2, name="seq-b1-k2"),
        _case("round", "cfg4_seq", 5, 333, 2111, 4, plan="layerskip33", name="seq-b5-k4-layerskip"),
        # long-context serving at batch 64, the largest state
        _case("round", "cfg5_b64", 64, 4096, 16384, 4, name="0.5b-b64-long-k4"),
        # prompts: one ordinary, one long on the large model, a ragged batch on the sequential hybrid
        _case("prefill", "cfg2_0p5b", 1, 512, 512, 8, name="prefill-0.5b-512"),
        _case("prefill", "cfg3_3b", 1, 2048, 2048, 4, name="prefill-3b-2048"),
        _case("prefill", "cfg4_seq", 4, 150, 1023, 4, name="prefill-seq-ragged4"),
    ]


def _log_int(rng, lo, hi_):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi_)))))


def draw(rng):
    """One more case of the same ranges: every model, batches 1 .. 64 (3B-class: 8), contexts 32 .. 16384 tokens as far
    as the batch-64 workload's cache allows, prompts of up to 2048 tokens, draft lengths 0 .. 8
    (3B-class: 4)."""
    mode = rng.choice(["round"] * 6 + ["sampled"] + ["prefill"] * 3)
    model = rng.choice(["cfg1_tiny", "cfg2_0p5b", "cfg2_0p5b", "cfg3_3b", "cfg4_seq"])
    small = model != "cfg3_3b"
    if mode == "prefill":
        batch = _log_int(rng, 1, 8)
        longest = max(24, min(2048, (4096 if small else 2048) // batch))
        top = _log_int(rng, 24, longest)
        lo = top if batch == 1 else max(8, int(top * rng.uniform(0.2, 0.9)))
        return _case(mode, model, batch, lo, top, rng.choice([4, 8]))
    batch = _log_int(rng, 1, 64 if small else 8)
    k = rng.choice([0, 1, 2, 3, 4, 4, 5, 8] if small else [0, 1, 2, 3, 4, 4])
    if mode == "sampled":
        batch, k = min(batch, 16), max(k, 1)
    longest = min(16384, (600000 if small else 16384) // batch)
    top = _log_int(rng, 32, longest)
    lo = top if batch == 1 else max(16, int(top * rng.uniform(0.25, 1.0)))
    plan = "layerskip33" if mode == "round" and model == "cfg4_seq" and k > 0 and rng.random() < 0.3 else "component"
    return _case(mode, model, batch, lo, top, k, replay=rng.random() < 0.25, plan=plan)


def _lengths(case):
    """Context / prompt lengths of the batch, uniform in [lo, hi]; the last sequence is the longest one."""
    b, lo, top = case["batch"], case["lo"], case["hi"]
    if b == 1 or lo == top:
        return [top] * b
    n = hi.context_lengths(b, lo, top - 1).tolist()               # part of the case: the same for every seed
    n[-1] = top
    return [int(x) for x in n]


# ------------------------------------------------------------------------------------------------
# what a program has in hand before the call
# ------------------------------------------------------------------------------------------------
def _fill(t, kind, g):
    """Seeded random values in a byte tensor, a gigabyte at a time (no temporary of its size)."""
    step = 1 << 30
    for o in range(0, t.numel(), step):
        part = t[o:o + step]
        if kind == "bf16":
            part.view(torch.bfloat16).normal_(generator=g)
        elif kind == "state":
            part.view(torch.float32).uniform_(-0.5, 0.5, generator=g)
        else:
            part.view(torch.float32).normal_(generator=g)


def _random_weights(eng, shape, g):
    """The documented initialisation (hs_inputs.make_weights), drawn on the device."""
    table, _ = hi.blob_layout(shape)
    for (layer, tid), (off, dims, dt) in table.items():
        n = int(np.prod(dims))
        t = eng.t_weights[off:off + n * (2 if dt == "bf16" else 4)].view(torch.bfloat16 if dt == "bf16" else torch.float32)
        if dt == "bf16":
            t.normal_(0.0, 0.02, generator=g)
        elif layer >= 0 and tid == hi.T_A_LOG:
            t.uniform_(0.0, math.log(16.0), generator=g)
        elif layer >= 0 and tid == hi.T_DT_BIAS:
            dt0 = torch.exp(t.uniform_(math.log(1e-3), math.log(1e-1), generator=g))
            t.copy_(dt0 + torch.log(-torch.expm1(-dt0)))
        elif layer >= 0 and tid == hi.T_CONV_W:
            t.uniform_(-0.5, 0.5, generator=g)
        elif layer >= 0 and tid == hi.T_CONV_B:
            t.zero_()
        else:
            t.fill_(1.0)


def _kv_view(eng, shape, cap):
    """The KV cache as bf16 [K | V][attention layer][sequence][kv head][row][head dim]."""
    n_al = sum(shape.layer_type(l) != hi.LAYER_GDN for l in range(shape.L))
    n = 2 * n_al * eng.max_batch * shape.kvh * cap * shape.hd
    return eng.t_kv[:2 * n].view(torch.bfloat16).view(2, n_al, eng.max_batch, shape.kvh, cap, shape.hd)


def _state_view(eng, shape, slots):
    """The recurrent states, float32 [recurrent layer][sequence][slot][elements of one state]."""
    n_rl = sum(shape.layer_type(l) != hi.LAYER_ATT for l in range(shape.L))
    e = shape.H * shape.P * shape.N if shape.arch == hi.ARCH_PARALLEL else shape.gh * shape.gdv * shape.gdk
    n = n_rl * eng.max_batch * slots * e
    return eng.t_snap[:4 * n].view(torch.float32).view(n_rl, eng.max_batch, slots, e)


def _logits_view(eng, shape, row0):
    """Where the library keeps the logits of a pass, as a device tensor [rows][V]: the place in the work buffer that
    holds the values get_logits() just returned (row0).  A program that wants logits on the device reads them there."""
    w = eng.t_work[:eng.sizes.work // 4 * 4].view(torch.float32)
    want = torch.from_numpy(row0).to(w.device)
    for at in (w[:w.numel() - shape.V + 1] == want[0]).nonzero().flatten().tolist():
        if torch.equal(w[at:at + shape.V], want):
            return w[at:]
    raise RuntimeError("the logits of the last pass are not in the work buffer")


def prepare(case, seed):
    shape = hi.CONFIGS[case["model"]]
    prefill = case["mode"] == "prefill"
    batch, k, lens = case["batch"], case["k"], _lengths(case)
    cap = max(lens) + (0 if prefill else shape.gen_tokens) + 2 * (k + 1) + 2
    flags = hs.HS_FLAG_GRAPHS | (hs.HS_FLAG_REPLAY if case["replay"] else 0)
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    eng = hs.Engine(shape, np.zeros(hi.blob_layout(shape)[1], np.uint8), max_batch=batch, max_k=k, kv_capacity=cap, flags=flags)
    _random_weights(eng, shape, g)
    if case["plan"] != "component":
        eng.set_draft_plan(hi.draft_plan(shape, case["plan"]))
    slots = 1 if case["replay"] else k + 1
    st = {"mode": case["mode"], "eng": eng, "k": k, "batch": batch, "lens": lens, "cap": cap, "shape": shape,
          "kv": _kv_view(eng, shape, cap), "states": _state_view(eng, shape, slots)}
    torch.cuda.synchronize()
    # one plain step tells where the logits lie
    for b in range(batch):
        eng.set_context(b, 0, b % shape.V)
    eng.set_batch(batch)
    eng.verify(0)
    st["logits"] = _logits_view(eng, shape, eng.get_logits(1)[0])
    eng.accept_rollback()
    eng.reset()
    if prefill:
        st["prompts"] = [hi.make_prompt(shape.V, n, seed=seed + 1, seq=b) for b, n in enumerate(lens)]
        return st
    with torch.cuda.stream(eng.stream):
        _fill(eng.t_kv[:eng.sizes.kv], "bf16", g)
        _fill(eng.t_snap[:eng.sizes.snap], "state", g)
        _fill(eng.t_conv[:eng.sizes.conv], "conv", g)
    eng.stream.synchronize()
    st["pending"] = [int(hi.make_prompt(shape.V, 1, seed=seed + 1, seq=1000 + b)[0]) for b in range(batch)]
    st["pattern"] = np.stack([hi.forced_accept(k, PATTERN, seq=b, seed=seed + 2) for b in range(batch)], axis=1).astype(np.int32)
    st["round"] = 0
    st["now"] = None                                       # tokens every sequence holds; None: start over
    if case["mode"] == "sampled":
        u = torch.zeros(2 * batch * k + batch, dtype=torch.float32, device=eng.device)
        st["uniforms"], st["gen"] = u, g
        eng.set_sampling(TEMPERATURE, u[:batch * k].view(batch, k), u[batch * k:2 * batch * k].view(batch, k), u[2 * batch * k:])
    torch.cuda.synchronize()
    return st


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def _run_prefill(st):
    eng, k, lens = st["eng"], st["k"], st["lens"]
    eng.reset()
    eng.prefill(st["prompts"])
    first = [eng.get_context(b)[1] for b in range(st["batch"])]       # every prompt's first generated token
    # logits after the longest prompt (the last sequence): last position of the pass over its last k + 1 tokens
    return {"first": first, "logits": st["logits"][(lens[-1] - 1) % (k + 1) * st["shape"].V:][:st["shape"].V],
            "kv": [st["kv"][:, :, b, :, :n] for b, n in enumerate(lens)],
            "states": [st["states"][:, b, (n - 1) % (k + 1)] for b, n in enumerate(lens)]}


def _run_round(st):
    eng, k, batch = st["eng"], st["k"], st["batch"]
    if st["now"] is None or max(st["now"]) + k + 1 > st["cap"]:
        for b in range(batch):                             # every sequence starts over from its first context
            eng.set_context(b, st["lens"][b], st["pending"][b])
        eng.set_batch(batch)
        st["now"] = list(st["lens"])
    if st["mode"] == "sampled":
        with torch.cuda.stream(eng.stream):
            st["uniforms"].uniform_(generator=st["gen"])
        n, emitted = eng.round_host(k)
    else:
        n, emitted = eng.round_host(k, forced_n=st["pattern"][st["round"] % PATTERN])
    st["round"] += 1
    at = st["now"]
    st["now"] = [x + int(m) + 1 for x, m in zip(at, n)]
    # rows appended to the cache: of every sequence in a small batch, of every eighth in a large one
    some = range(0, batch, 1 if batch <= 8 else 8)
    return {"n": n, "emitted": emitted, "logits": st["logits"][:batch * (k + 1) * st["shape"].V],
            "states": st["states"], "kv": [st["kv"][:, :, b, :, at[b]:at[b] + k + 1] for b in some]}


def run(st):
    return _run_prefill(st) if st["mode"] == "prefill" else _run_round(st)


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------
def _layer_weights(s, kind, draft):
    """Matrix elements and float32 parameters of one layer."""
    mlp, attn_rows = 3 * s.ff * s.d, (s.qh + 2 * s.kvh) * s.hd
    if kind == hi.LAYER_PAR:
        rows = 2 * s.d_inner + 2 * s.N + s.H + (0 if draft else attn_rows)
        return rows * s.d + s.d * s.d_inner + (0 if draft else s.d * s.qh * s.hd) + mlp, 2 * s.d + 5 * s.convd + 3 * s.H + s.d_inner
    if kind == hi.LAYER_GDN:
        rows = 2 * s.gh * s.gdk + 2 * s.gh * s.gdv + 2 * s.gh
        return rows * s.d + s.d * s.gh * s.gdv + mlp, 2 * s.d + 5 * s.convd + s.gdv
    return attn_rows * s.d + s.d * s.qh * s.hd + mlp, 2 * s.d


def _pass_work(s, lens, T, draft=False, plan=None, head_rows=None):
    """(bytes, flops) of one pass over T[b] positions behind a context of lens[b] tokens: weights once, states read and
    written once, cache rows read once and the new ones written, embedding rows and logits."""
    by = fl = 0.0
    tokens = sum(T)
    for l in range(s.L):
        kind = s.layer_type(l)
        mode = hi.DRAFT_FULL if not draft else int(plan[l])
        if mode == hi.DRAFT_SKIP or (mode == hi.DRAFT_LINEAR and kind == hi.LAYER_ATT):
            continue
        w, p = _layer_weights(s, kind, draft=mode == hi.DRAFT_LINEAR)
        by += 2 * w + 4 * p
        fl += 2.0 * w * tokens
        if kind != hi.LAYER_ATT:
            e = s.H * s.P * s.N if kind == hi.LAYER_PAR else s.gh * s.gdv * s.gdk
            by += len(lens) * (2 * 4 * e + 2 * 4 * 3 * s.convd)
            fl += (5.0 if kind == hi.LAYER_PAR else 8.0) * e * tokens
        if kind != hi.LAYER_GDN and mode == hi.DRAFT_FULL:
            by += sum(4.0 * s.kvh * s.hd * (n + t) for n, t in zip(lens, T))
            fl += sum(4.0 * s.qh * s.hd * t * (n + (t + 1) / 2) for n, t in zip(lens, T))
    rows = tokens if head_rows is None else head_rows
    by += 2.0 * s.V * s.d + 4 * s.d + tokens * 2 * s.d + rows * 4 * s.V
    fl += 2.0 * s.V * s.d * rows
    return by, fl


def work(case):
    s, lens, k = hi.CONFIGS[case["model"]], _lengths(case), case["k"]
    if case["mode"] == "prefill":
        by, fl = _pass_work(s, [0] * len(lens), lens, head_rows=len(lens))
        return {"bytes": by, "flops": fl}
    plan = hi.draft_plan(s, case["plan"])
    db, df = _pass_work(s, lens, [1] * len(lens), draft=True, plan=plan)
    vb, vf = _pass_work(s, lens, [k + 1] * len(lens))
    return {"bytes": k * db + vb, "flops": k * df + vf}


def tolerance(case):
    """Measured: the same pass with its sums in other orders (projections on the warp-level path, on tcgen05 and without
    tensor cores, every attention form) differs by up to 5.7e-4 in the cache rows - float32 sums that differ in the last
    bits round to the neighbouring bf16 value here and there: 2^-7 of a value - and by up to 9e-5 in logits and states.
    A whole value may differ where two logits tie within that."""
    return {"rel": 2.5e-3, "max": 3.2e-2, "differ": 5e-3}
