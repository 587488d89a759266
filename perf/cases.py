"""What the decode library is timed on: the work a serving program has it do, through its public binding.

Three kinds of pass:
  decode       `steps` decode steps of a batch of sequences whose prompts are in the cache, tokens and
               results in host memory every step, as a generation loop makes them
  first_token  a request's start: its slots reset, its prompts ingested, its first token decoded
  attention    the stand-alone attention kernels on a caller's own cache
Decode steps are forced: every step's input token is given, so that two implementations whose
rounding differs see the same inputs to the end of the pass and not only until the first near-tie.
What a pass returns of its tokens is the logit each one had (two ids in a near-tie have the same).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2603_09215_b200 import binding, synth

ROOM = 16  # passes of a decode case before its sequences start over from their prompts


def _decode(name, shape, batch, len_lo, len_hi, steps, n_text, n_speech, exit_layer, period, random_phase=False,
            sampled=False, conf_start=0):
    return dict(name=name, kind="decode", shape=shape, batch=batch, len_lo=len_lo, len_hi=len_hi, steps=steps,
                n_text=n_text, n_speech=n_speech, exit_layer=exit_layer, period=period, random_phase=random_phase,
                sampled=sampled, conf_start=conf_start)


def listed():
    return [
        # the smallest calls: the four-layer model, one sequence, two cycles of two text and four speech tokens
        _decode("tiny_b1", "tiny", 1, 32, 32, 12, 2, 4, 2, 3),
        # one listener of the 28-layer backbone: an interleave cycle, one text and four speech tokens
        _decode("step_b1", "step", 1, 512, 512, 5, 1, 4, 20, 4),
        # the same backbone decoded as it is used in earnest, by nucleus sampling, after a longer prompt
        _decode("step_b1_sampled", "step", 1, 1337, 1337, 5, 1, 4, 20, 4, sampled=True),
        # the compared method: speech steps leave by the entropy of a late layer's prediction
        _decode("step_b1_conf", "step", 1, 512, 512, 5, 1, 4, 20, 4, conf_start=26),
        # a few listeners at odd lengths and phases: three rows below the exit layer, up to nine above it
        _decode("step_b3", "step", 3, 77, 901, 5, 1, 4, 17, 3, random_phase=True),
        # plain decoding at full depth, what the schedule is compared with
        _decode("step_b12_full", "step", 12, 300, 1500, 5, 1, 4, 20, 1),
        # a loaded server: 64 sequences of ragged length, every one at its own place in its cycle
        _decode("step_b64", "step", 64, 256, 2048, 5, 1, 4, 20, 4, random_phase=True),
        # the 40-layer backbone, sixteen sequences in step: a whole cycle of 13 text and 26 speech tokens
        _decode("glm_b16", "glm", 16, 1024, 1024, 39, 13, 26, 30, 4),
        # long conversations: the cache of 64 sequences of 8192 positions outweighs the model's weights
        _decode("glm_b64_long", "glm", 64, 8192, 8192, 8, 13, 26, 30, 4, random_phase=True),
        # requests that arrive together, prompts of any length, 256 rows a pass
        dict(name="step_prefill_ragged", kind="first_token", shape="step", batch=6, len_lo=100, len_hi=2048, rows=256),
        # one request of the 40-layer backbone with the library's own choice of rows a pass
        dict(name="glm_prefill_b1", kind="first_token", shape="glm", batch=1, len_lo=1024, len_hi=1024, rows=0),
        # attention alone, for a caller with a cache of its own: single rows and refresh blocks, ragged lengths
        dict(name="attention_ragged", kind="attention", q_heads=28, kv_heads=4, head_dim=128, groups=48, grp_rows=4,
             len_lo=200, len_hi=3000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 6 + ["first_token"] * 2 + ["attention"] * 2)
    if kind == "attention":
        kv, g, hd = rng.choice([(4, 7, 128), (2, 16, 128), (2, 2, 64), (8, 4, 128)])
        hi = _log(rng, 64, 6000)
        return dict(kind=kind, q_heads=kv * g, kv_heads=kv, head_dim=hd, groups=_log(rng, 1, 96),
                    grp_rows=rng.choice([1, 1, 2, 3, 4, 8]), len_lo=_log(rng, 16, hi), len_hi=hi)
    shape = rng.choice(["tiny", "step", "step", "glm", "glm"])
    if kind == "first_token":
        hi = _log(rng, 24, 2048)
        return dict(kind=kind, shape=shape, batch=_log(rng, 1, 5), len_lo=_log(rng, 16, hi), len_hi=hi,
                    rows=rng.choice([0, 0, 64, 100, 256]))
    batch = _log(rng, 1, 64)
    hi = _log(rng, 32, min(8192, (131072 if shape == "step" else 524288) // batch))
    layers = synth.SHAPES[shape]["n_layers"]
    n_text, n_speech, steps = {"tiny": (2, 4, 12), "step": (1, 4, 5), "glm": (13, 26, 39 if batch <= 8 else 8)}[shape]
    c = _decode("", shape, batch, _log(rng, 16, hi), hi, steps, n_text, n_speech,
                rng.randint(layers // 2, layers - 1), rng.choice([1, 2, 3, 4, 4, 4, 8]), rng.random() < 0.6)
    c["sampled"] = rng.random() < 0.25
    del c["name"]
    return c


# ------------------------------------------------------------------ what a case says, spelled out
def _lengths(case):
    """Prompt lengths, spread evenly over the case's range and shuffled."""
    n = case.get("batch") or case["groups"]
    lo, hi = case["len_lo"], case["len_hi"]
    out = [lo + (hi - lo) * i // max(1, n - 1) if n > 1 else hi for i in range(n)]
    random.Random(n).shuffle(out)
    return out


def _dims(case):
    L = synth.SHAPES[case["shape"]]["n_layers"]
    d = synth.model_dims(case["shape"], case.get("exit_layer", L * 3 // 4), case.get("period", 4))
    if case.get("conf_start"):
        d.update(conf_modalities=2, conf_start=case["conf_start"], conf_threshold=0.1)
    return d


def _cycle(case):
    """(modalities, counters) of every step of the interleave cycle."""
    n = case["n_text"] + case["n_speech"]
    phi, off = synth.make_phases(case["batch"], case["n_text"], case["n_speech"], case["period"], case["random_phase"])
    out = []
    for g in range(n):
        mc = [synth.interleave(g, case["n_text"], case["n_speech"], int(p), int(o)) for p, o in zip(phi, off)]
        out.append((np.array([m for m, _ in mc], np.uint8), np.array([c for _, c in mc], np.int32)))
    return out


def _max_pending(case):
    return case["n_speech"] + 1 if case["conf_start"] else max(1, case["period"] - 1)


def _heads(case, d):
    L = d["n_layers"]
    return {d["exit_layer"], L} | (set(range(case["conf_start"], L)) if case.get("conf_start") else set())


# ------------------------------------------------------------------ inputs
def _weights(d, heads, gen):
    """Random-init weights of the shape, on the device: N(0, 0.02), gains 1 + N(0, 0.02), bf16."""
    m, F = d["d_model"], d["d_ffn"]
    q, kv, V = d["n_q_heads"] * d["head_dim"], d["n_kv_heads"] * d["head_dim"], d["vocab_text"] + d["vocab_speech"]
    shapes = {"attn_norm": (m,), "wq": (q, m), "wk": (kv, m), "wv": (kv, m), "wo": (m, q), "mlp_norm": (m,),
              "w_gate": (F, m), "w_up": (F, m), "w_down": (m, F), "head_norm": (m,), "head_proj": (V, m)}

    def new(shape, mean):
        return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(mean, 0.02, generator=gen)

    out = {"embed": new((V, m), 0.0)}
    for name in binding.PER_LAYER:
        out[name] = [new(shapes[name], 1.0 if name.endswith("norm") else 0.0)
                     if not name.startswith("head") or layer in heads else None for layer in range(1, d["n_layers"] + 1)]
    return out


def _tokens(d, n, rng):
    return rng.integers(0, d["vocab_text"] + d["vocab_speech"], size=n, dtype=np.int32)


def _prepare_decode(case, gen, rng):
    d, B, steps, lens = _dims(case), case["batch"], case["steps"], _lengths(case)
    w = _weights(d, _heads(case, d), gen)
    ctx = binding.Sparsk(d, w, B, max(lens) + ROOM * steps + 1, _max_pending(case))
    # the prompts' keys and values: N(0, 1), every layer and sequence its own stretch of one pool
    row = d["n_kv_heads"] * d["head_dim"]
    pool = torch.empty((max(lens) + 4096, row), dtype=torch.float16, device="cuda").normal_(generator=gen)
    at = rng.integers(0, 4096, size=(B, d["n_layers"], 2))
    for s, n in enumerate(lens):
        for layer in range(d["n_layers"]):
            a, b = at[s, layer]
            ctx.import_kv(s, layer + 1, 0, pool[a:a + n], pool[b:b + n])
        ctx.set_len(s, n)
    V = d["vocab_text"] + d["vocab_speech"]
    state = dict(case=case, ctx=ctx, lens=lens, used=0, g=0, cycle=_cycle(case), slots=np.arange(B, dtype=np.int32),
                 inputs=_tokens(d, (steps, B), rng), out_tok=np.zeros((steps, B), np.int32),
                 depths=np.zeros((steps, B), np.int32),
                 hidden=torch.zeros((steps, B, d["d_model"]), device="cuda"), logits=torch.zeros((steps, B, V), device="cuda"))
    state["rows"] = [(state["hidden"][i], state["logits"][i]) for i in range(steps)]
    if case["sampled"]:
        state["uniforms"] = list(torch.rand((steps, B), device="cuda", generator=gen).mul_(0.9999))
    return state


def _prepare_first_token(case, gen, rng):
    d, lens = _dims(case), _lengths(case)
    B, V = case["batch"], d["vocab_text"] + d["vocab_speech"]
    ctx = binding.Sparsk(d, _weights(d, _heads(case, d), gen), B, max(lens) + 8, 3, prefill_rows=case["rows"])
    hidden, logits = torch.zeros((B, d["d_model"]), device="cuda"), torch.zeros((B, V), device="cuda")
    ctx.set_debug(hidden, logits)
    prompts = [_tokens(d, n, rng) for n in lens]
    return dict(case=case, ctx=ctx, lens=lens, slots=np.arange(B, dtype=np.int32), prompts=[p[:-1] for p in prompts],
                last=np.array([p[-1] for p in prompts], np.int32), text=np.zeros(B, np.uint8), zero=np.zeros(B, np.int32),
                tok=np.zeros(B, np.int32), depths=np.zeros(B, np.int32), hidden=hidden, logits=logits)


def _attention_rows(case):
    """(slot, first position, rows) of every group: every third one a refresh block."""
    out = []
    for slot, n in enumerate(_lengths(case)):
        rows = min(case["grp_rows"], n) if slot % 3 == 0 else 1
        out.append((slot, n - rows, rows))
    return out


def _prepare_attention(case, gen):
    Hq, Hkv, hd, groups = case["q_heads"], case["kv_heads"], case["head_dim"], _attention_rows(case)
    S, n = case["len_hi"], sum(r for _, _, r in groups)
    q = torch.empty((n, Hq * hd), dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    k, v = (torch.empty((len(groups), Hkv, S, hd), dtype=torch.float16, device="cuda").normal_(generator=gen) for _ in "kv")
    ints = [torch.tensor(x, dtype=torch.int32, device="cuda") for x in (
        [s for s, _, r in groups for _ in range(r)], [p + i for _, p, r in groups for i in range(r)],
        [sum(r for _, _, r in groups[:g]) for g in range(len(groups))], [r for _, _, r in groups])]
    out = torch.zeros_like(q)
    args = binding.attn_args(q, k, v, out, *ints, max(r for _, _, r in groups), S, Hq)
    scratch = torch.empty(binding.attention_scratch_bytes(n, Hq, hd), dtype=torch.uint8, device="cuda")
    return dict(case=case, args=args, scratch=scratch, out=out, keep=(q, k, v, ints))


def prepare(case, seed):
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    if case["kind"] == "attention":
        return _prepare_attention(case, gen)
    rng = np.random.default_rng(seed)
    return (_prepare_decode if case["kind"] == "decode" else _prepare_first_token)(case, gen, rng)


# ------------------------------------------------------------------ one pass
def _chosen(logits, tokens):
    """The logit of every token that was picked."""
    return logits.gather(-1, torch.from_numpy(tokens.astype(np.int64)).cuda()[..., None])[..., 0]


def _run_decode(s):
    case, ctx, steps = s["case"], s["ctx"], s["case"]["steps"]
    if s["used"] == ROOM:  # the cache is full: the sequences start over from their prompts
        for slot, n in enumerate(s["lens"]):
            ctx.set_len(slot, n)
        s["used"] = 0
    for i in range(steps):
        mods, counters = s["cycle"][(s["g"] + i) % len(s["cycle"])]
        ctx.set_debug(*s["rows"][i])
        if case["sampled"]:
            ctx.set_sampling(0.7, 0.9, s["uniforms"][i])
        ctx.decode_step_host(s["slots"], s["inputs"][i], mods, counters, s["out_tok"][i], s["depths"][i])
    s["used"] += 1
    s["g"] += steps
    return dict(hidden=s["hidden"], logits=s["logits"], chosen=_chosen(s["logits"], s["out_tok"]), depths=s["depths"].copy())


def _run_first_token(s):
    ctx = s["ctx"]
    for slot in range(s["case"]["batch"]):
        ctx.reset_slot(slot)
    ctx.prefill(s["slots"], s["prompts"])
    ctx.decode_step_host(s["slots"], s["last"], s["text"], s["zero"], s["tok"], s["depths"])
    # the last layer's cache, which every layer before it has its part in
    L = ctx.dims["n_layers"]
    cache = [ctx.export_kv(slot, L, 0, n) for slot, n in enumerate(s["lens"])]
    return dict(hidden=s["hidden"], logits=s["logits"], chosen=_chosen(s["logits"], s["tok"]), depths=s["depths"].copy(),
                cache=cache)


def run(state):
    kind = state["case"]["kind"]
    if kind == "attention":
        rc = binding.attention(state["args"], state["scratch"])
        if rc != binding.OK:
            raise binding.SparskError(rc, "attention")
        return state["out"]
    return _run_decode(state) if kind == "decode" else _run_first_token(state)


# ------------------------------------------------------------------ what a pass cannot do without
def _layer_params(d):
    qd, kd = d["n_q_heads"] * d["head_dim"], d["n_kv_heads"] * d["head_dim"]
    return 2 * qd * d["d_model"] + 2 * kd * d["d_model"] + 3 * d["d_ffn"] * d["d_model"]


def work(case):
    """Bytes: each active layer's weights once per step (once per request for a prompt), each
    active (sequence, layer)'s cache prefix once, the rows appended, each (head, modality) slice
    used, the embedding rows, the hidden states and logits returned.  Flops: two per weight and
    row, four per query head, position and head dimension."""
    if case["kind"] == "attention":
        groups, row = _attention_rows(case), case["head_dim"] * 2
        kv = sum((p + r) * case["kv_heads"] * row * 2 for _, p, r in groups)
        io = sum(r for _, _, r in groups) * case["q_heads"] * row * 2
        pairs = sum(r * (p + 1) + r * (r - 1) // 2 for _, p, r in groups)
        return {"bytes": kv + io, "flops": pairs * 4 * case["q_heads"] * case["head_dim"]}
    d, lens, B = _dims(case), _lengths(case), case["batch"]
    L, e, m = d["n_layers"], d["exit_layer"], d["d_model"]
    V, params = d["vocab_text"] + d["vocab_speech"], _layer_params(d)
    kvb, att = 2 * d["n_kv_heads"] * d["head_dim"] * 2, 4 * d["n_q_heads"] * d["head_dim"]
    returned = B * (V + m) * 4
    if case["kind"] == "first_token":
        pairs = sum(n * (n + 1) // 2 for n in lens)
        head = d["vocab_text"] * m
        return {"bytes": L * (params * 2 + sum(lens) * kvb) + head * 2 + sum(lens) * m * 2 + returned + 2 * sum(lens) * kvb,
                "flops": L * (sum(lens) * params * 2 + pairs * att) + 2 * B * head}
    bytes_, flops, lens, pend = 0, 0, list(lens), [0] * B
    for i, (mods, counters) in zip(range(case["steps"]), _cycle(case) * (1 + case["steps"] // len(_cycle(case)))):
        depths = [L if m_ == 0 or case["conf_start"] or c % case["period"] == 0 else e for m_, c in zip(mods, counters)]
        bytes_ += params * 2 * max(depths) + B * m * 2 + returned
        heads = {(dep, int(m_)) for dep, m_ in zip(depths, mods)}
        if case["conf_start"] and mods.any():
            heads |= {(layer, 1) for layer in range(case["conf_start"], L)}
        bytes_ += sum((d["vocab_speech"] if m_ else d["vocab_text"]) * m * 2 for _, m_ in heads)
        for b, dep in enumerate(depths):
            rows_up = pend[b] + 1 if dep == L else 0
            bytes_ += (e if dep < L else L) * (lens[b] + 1) * kvb + (e + (L - e) * rows_up) * kvb
            flops += (e + (L - e) * rows_up) * (params * 2 + (lens[b] + 1) * att)
            flops += 2 * m * (d["vocab_speech"] if mods[b] else d["vocab_text"])
            lens[b] += 1
            pend[b] = 0 if dep == L else pend[b] + 1
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    """About four times what other ways through the same arithmetic differ by (the library's other
    kernels, other cuts of the positions, other rows a pass): 3.6e-3 and 2e-2 for the cache of a
    long prompt, 2e-3 and 1.5e-2 for logits.  The stand-alone attention rounds its output to bf16
    (1.7e-3 and 4.7e-3 from 64-bit arithmetic)."""
    return {"rel": 4e-3, "max": 0.02} if case["kind"] == "attention" else {"rel": 1e-2, "max": 0.08}
