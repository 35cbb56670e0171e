"""Cases that stand for the work a user of this library has it do, with what it takes to time
one pass of each and to compare the outputs of two builds.

A decode loop calls the library once per denoising step of a block: the packed attention in
every layer of the model, then the decision and the walk over the draft graph, then the drafting
of the next step's blocks.  ``listed()`` names one case per entry point at sizes of the
configurations of ``workloads.config`` (and one with nothing round about it), ``draw`` spreads
over the ranges around them.  The fields of a case:

  entry    "step"     VerifyStep.run: attention of one layer, decision and walk (device tensors)
           "calls"    the same through the two functions, which allocate what they return
           "model"    the attention of `layers` layers, each into its own output, then decision
                      and walk: a whole forward pass's share of the library
           "host"     VerifyStep.run_host: the step from pinned host buffers, verdict on the host
           "full"     the attention of a full-sequence model, `suffix` trailing masked rows
           "lazy"     decision and walk that evaluate only the nodes the walk reaches
           "sampled"  the decision at temperature > 0
           "lmhead"   the decision fused into the output projection of width `hidden`
           "draft"    the drafts of the next step from the current block's logits
  B N L P  sequences, graph nodes, block length, context keys
  Hq Hkv d query heads, key/value heads, head dimension
  V dtype  vocabulary entries; "bf16" or "f32" for the attention tensors and the logits
  rule S   "threshold" (tau = 0.9) or "tops" with S tokens per step
  depth    levels of the draft graph

Values: q, k, v ~ N(0, 1); logits N(0, 2) clipped at 4 sigma with one planted winner per masked
row, confident (0.92 to 0.999) in the rows a step unmasks and not (0.05 to 0.85) in the others; a
quarter of the true block is decoded already; a child node is its parent's next state with each new
token spoiled with probability 0.2, later siblings unmask other positions.
"""
import math

import numpy as np
import torch

from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads
from paper_2509_18085_b200.step import StepInputs, VerifyStep

_DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}
_TAU = 0.9
_TEMPERATURE = 0.8
_SPOIL = 0.2

# The draft graph of the drafting case: ten formulas over position ranks 0..3 and vocabulary
# ranks 0..2, pruned to three drafts.
_FORMULAS = [[(0, 0)], [(0, 1)], [(1, 0)], [(0, 0), (1, 0)], [(0, 0), (1, 1)], [(0, 1), (1, 0)],
             [(0, 0), (2, 0)], [(0, 0), (1, 0), (2, 0)], [(0, 0), (1, 0), (2, 2)],
             [(0, 0), (1, 0), (2, 0), (3, 0)]]
_CHILDREN = [[3, 4, 6], [5], [3, 5], [7, 8], [], [], [7], [9], [], []]
_BUDGET, _TOP_K = 3, 3


def _from_config(name, entry, index, n_nodes=None, **more):
    c = workloads.config(index, n_nodes)
    case = {"name": name, "entry": entry, "B": c.batch, "N": c.n_nodes, "L": c.block_len, "P": c.prefix_len,
            "Hq": c.n_q_heads, "Hkv": c.n_kv_heads, "d": c.head_dim, "V": c.vocab, "dtype": c.dtype,
            "rule": "tops" if c.rule == workloads.RULE_TOPS else "threshold", "S": c.top_s, "depth": c.depth}
    case.update(more)
    return case


def listed():
    return [
        # the smallest call: one short block, four nodes, fp32; nothing but latency
        _from_config("step tiny f32", "step", 1),
        # a full forward pass at the benchmark's shape: one attention call per layer, one decision
        _from_config("model llada8b", "model", 2, layers=32),
        # one step for a caller whose tensors are in host memory, copies included
        _from_config("host llada8b", "host", 2),
        # grouped-query heads, a longer context, static unmasking
        _from_config("step dream7b-gqa", "step", 3),
        # the largest: four sequences, 4096 context keys, 32 nodes, 4096 logits rows
        _from_config("step long-batched", "step", 4),
        # many drafts of a short block
        _from_config("step short-wide", "step", 5, 64),
        # nothing round: three sequences, 5 x 20 positions, an odd context and vocabulary, d = 64
        {"name": "calls ragged d64", "entry": "calls", "B": 3, "N": 5, "L": 20, "P": 777, "Hq": 24, "Hkv": 8,
         "d": 64, "V": 50257, "dtype": "bf16", "rule": "tops", "S": 2, "depth": 2},
        # a model that caches its prefix only: three trailing masked blocks are queries too
        _from_config("full llada8b", "full", 2, suffix=96),
        # decoding at temperature > 0
        _from_config("sampled llada8b", "sampled", 2),
        # the decision for the accepted path only, on a batch of long graphs
        _from_config("lazy long-batched", "lazy", 4),
        # logits never written: 256 rows against a 126464 x 4096 output embedding
        _from_config("lmhead llada8b", "lmhead", 2, hidden=4096),
        # drafting for the next step
        _from_config("draft llada8b", "draft", 2, 1),
    ]


def _cost(case):
    """Seconds of the case's work at nominal rates, to compare sizes."""
    w = work(case)
    rate = 1.6e15 if case["dtype"] == "bf16" or case["entry"] == "lmhead" else 6e13
    bus = 5e10 if case["entry"] == "host" else 6.5e12
    return w["flops"] / rate + w["bytes"] / bus


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    largest = _cost(_from_config("", "step", 4))
    while True:
        entry = rng.choice(["step"] * 4 + ["calls"] * 3 + ["model"] * 2 + ["host", "full", "full", "lazy", "sampled",
                                                                          "sampled", "lmhead", "draft"])
        Hq, Hkv = rng.choice([(32, 32), (32, 8), (28, 4), (24, 8), (16, 16), (12, 4), (8, 1), (5, 5)])
        dtype = "f32" if rng.random() < 0.15 else "bf16"
        case = {"entry": entry, "B": rng.choice([1, 1, 1, 2, 3, 4]), "N": log_int(2, 64),
                "L": rng.choice([4, 8, 16, 32, 32, rng.randint(5, 64)]), "P": log_int(50, 4096), "Hq": Hq, "Hkv": Hkv,
                "d": rng.choice([128, 128, 64]), "V": log_int(1000, 152064), "dtype": dtype,
                "rule": rng.choice(["threshold", "tops"]), "S": rng.choice([1, 2, 3]), "depth": rng.randint(1, 5)}
        if entry in ("step", "model", "host"):
            case["V"] = max(1000, case["V"] // 8 * 8)  # VerifyStep takes dense rows only
        if entry == "model":
            case["layers"] = rng.randint(8, 32)
        if entry == "full":
            case.update(suffix=log_int(8, 512), d=128, dtype="bf16")
        if entry == "lmhead":
            case.update(hidden=128 * rng.randint(4, 48), dtype="bf16", V=log_int(16000, 152064))
        if entry == "lmhead" and case["B"] * case["N"] * case["L"] > 512:
            continue
        if entry == "draft":
            case["N"] = 1
        logits = case["B"] * case["N"] * case["L"] * case["V"] * (4 if case["dtype"] == "f32" else 2)
        if logits < 1.1e9 and _cost(case) < largest:
            return case


# ---------------------------------------------------------------------------------------------
# Draft graphs
# ---------------------------------------------------------------------------------------------
def _per_step(case):
    return case["S"] if case["rule"] == "tops" else 2


def _levels(case):
    """Level of every node: the drafts fill `depth` levels evenly."""
    n = case["N"] - 1
    depth = max(1, min(case["depth"], n))
    out = [0]
    for i in range(depth):
        out += [i + 1] * (n // depth + (1 if i < n % depth else 0))
    return out[:case["N"]]


def _masked_at(case, level):
    L = case["L"]
    return max(0, L - (L // 4 if L >= 8 else 0) - _per_step(case) * level)


def _masked_rows(case):
    return case["B"] * sum(_masked_at(case, lv) for lv in _levels(case))


def _graphs(case, seed):
    """Block states [B,N,L], planted winners and confidences of the same shape, and parent lists."""
    B, N, L, V = case["B"], case["N"], case["L"], case["V"]
    mask, per = V - 1, _per_step(case)
    levels = _levels(case)
    state = np.full((B, N, L), mask, np.int32)
    tok = np.zeros((B, N, L), np.int32)
    conf = np.zeros((B, N, L))
    lists = []
    for b in range(B):
        rng = np.random.default_rng([seed, b])
        tok[b] = rng.integers(0, V - 1, (N, L))
        conf[b] = rng.uniform(0.05, 0.85, (N, L))
        sure = rng.uniform(0.92, 0.999, (N, L))
        known = rng.permutation(L)[:L - _masked_at(case, 0)]
        state[b, 0, known] = rng.integers(0, V - 1, len(known))
        plan, siblings, before, level = {}, {}, [], [0]
        for n in range(N):
            if n > 0:
                if levels[n] != levels[n - 1]:
                    before, level = level, []
                parent = before[len(level) % len(before)]
                level.append(n)
                k = siblings[parent] = siblings.get(parent, -1) + 1
                order = plan[parent]
                # the parent's own next state first, then sets with one position swapped
                take = list(order[:per])
                if k and len(order) > per:
                    take[(k - 1) % per] = order[per + (k - 1) % (len(order) - per)]
                new = tok[b, parent, take]
                wrong = rng.random(len(take)) < _SPOIL
                state[b, n] = state[b, parent]
                state[b, n, take] = np.where(wrong, (new + 1) % (V - 1), new)
            plan[n] = rng.permutation(np.flatnonzero(state[b, n] == mask))
            conf[b, n, plan[n][:per]] = sure[n, plan[n][:per]]
        lists.append(workloads.structural_parent_lists(state[b], mask))
    cap = (max(1, max(len(i) for _, i in lists)) + 3) // 4 * 4
    off = np.stack([o for o, _ in lists]).astype(np.int32)
    idx = np.zeros((B, cap), np.int32)
    for b, (_, i) in enumerate(lists):
        idx[b, :len(i)] = i
    return state, tok, conf, off, idx


def _logit_of(conf, V):
    """The winner's logit for a confidence, over N(0, 2) noise in the other V - 1 entries."""
    return math.log(V - 1) + 2.0 + torch.log(conf / (1 - conf))


def _logits(case, seed, tok, conf):
    """[B,N,L,V], rows 16-byte aligned: a view of a wider buffer where V is odd."""
    B, N, L, V = case["B"], case["N"], case["L"], case["V"]
    dtype = _DTYPE[case["dtype"]]
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty((B, N, L, (V + 7) // 8 * 8), dtype=dtype, device="cuda")
    for b in range(B):  # by sequence: bounded scratch
        x[b, ..., :V] = (torch.randn((N, L, V), generator=g, device="cuda") * 2).clamp_(-8, 8)
    winner = _logit_of(torch.from_numpy(conf).cuda().clamp_(1e-3, 0.9995), V)
    x.scatter_(3, torch.from_numpy(tok).cuda().long()[..., None], winner.to(dtype)[..., None])
    return x[..., :V]


# ---------------------------------------------------------------------------------------------
# One case: its inputs and a pass
# ---------------------------------------------------------------------------------------------
def _attention_inputs(case, g):
    B, N, L, P, Hq, Hkv, d = (case[k] for k in ("B", "N", "L", "P", "Hq", "Hkv", "d"))
    dtype = _DTYPE[case["dtype"]]

    def r(*shape):
        return torch.randn(shape, generator=g, device="cuda").to(dtype)

    return (r(B, N, L, Hq, d), r(B, P, Hkv, d), r(B, P, Hkv, d), r(B, N, L, Hkv, d), r(B, N, L, Hkv, d))


def _config(case):
    rule = workloads.RULE_TOPS if case["rule"] == "tops" else workloads.RULE_THRESHOLD
    return workloads.Config("case", case["B"], case["N"], case["L"], case["P"], case["Hq"], case["Hkv"], case["d"],
                            case["dtype"], case["V"], rule, top_s=case["S"], threshold=_TAU, depth=case["depth"])


def prepare(case, seed):
    entry = case["entry"]
    s = {"entry": entry, "cfg": _config(case), "seed": seed}
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    if entry == "full":
        B, S, Hq, Hkv, d = case["B"], case["suffix"], case["Hq"], case["Hkv"], case["d"]
        q, kp, vp, kb, vb = _attention_inputs(case, g)
        qs, ks, vs = (torch.randn((B, S, h, d), generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
        s["args"] = (q, qs, kp, vp, ks, vs, kb, vb)
        return s
    state, tok, conf, off, idx = _graphs(case, seed)
    tokens, off, idx = (torch.from_numpy(a).cuda() for a in (state, off, idx))
    if entry == "lmhead":
        H, V = case["hidden"], case["V"]
        w = (torch.randn((V, H), generator=g, device="cuda") * (2.0 / math.sqrt(H))).to(torch.bfloat16)
        h = torch.randn((case["B"], case["N"], case["L"], H), generator=g, device="cuda")
        # the component along the winner's embedding is set to what the confidence asks for
        wt = w[torch.from_numpy(tok).cuda().long()].float()
        along = (_logit_of(torch.from_numpy(conf).cuda(), V).float() - (h * wt).sum(-1)) / (wt * wt).sum(-1)
        s.update(hidden=(h + along[..., None] * wt).to(torch.bfloat16), weight=w, tokens=tokens)
        return s
    logits = _logits(case, seed, tok, conf)
    if entry == "draft":
        s.update(logits=logits[:, 0], tokens=tokens[:, 0].contiguous(), graph=spiffy.draft_graph(_FORMULAS, _CHILDREN))
        return s
    att = _attention_inputs(case, g) if entry in ("step", "calls", "model", "host") else [None] * 5
    x = StepInputs(*att, logits, tokens, off, idx)
    if entry == "host":
        x = StepInputs(*(t.cpu().pin_memory() for t in x.tensors()))
    s["x"] = x
    if entry != "calls":
        # the buffers a decode loop keeps; what a pass leaves untouched reads as zero
        s["step"] = step = VerifyStep(s["cfg"])
        for t in (step.decision.conf, step.decision.top_tok, step.decision.unmask_bits):
            t.zero_()
    if entry == "model":
        s["layers"] = [att] + [_attention_inputs(case, g) for _ in range(case["layers"] - 1)]
        s["outs"] = [torch.empty_like(layer[0]) for layer in s["layers"]]
    return s


def _decision(d):
    return [d.conf, d.top_tok, d.unmask_bits, d.n_unmask, d.dev_status]


def _walk(w):
    return [w.accepted_node, w.n_accepted, w.path, w.next_block, w.dev_status]


def run(s):
    entry, c = s["entry"], s["cfg"]
    if entry == "full":
        return list(spiffy.spiffy_full_sequence_attention(*s["args"]))
    if entry == "lmhead":
        return _decision(spiffy.spiffy_lmhead_decide(s["hidden"], s["weight"], s["tokens"], c.mask_id, c.rule, c.top_s,
                                                     c.threshold))
    if entry == "draft":
        d = spiffy.spiffy_draft_blocks(s["logits"], s["tokens"], c.mask_id, s["graph"], _BUDGET, _TOP_K)
        return [d.tokens, d.kept, d.score, d.parent_off, d.parent_idx, d.dev_status]
    x = s["x"]
    if entry == "calls":
        out = spiffy.spiffy_graph_attention(x.q, x.k_prefix, x.v_prefix, x.k_block, x.v_block)
        d, w = spiffy.spiffy_decide_walk(x.logits, x.block_tokens, x.parent_off, x.parent_idx, c.mask_id, c.rule,
                                         c.top_s, c.threshold)
        return [out] + _decision(d) + _walk(w)
    step = s["step"]
    if entry == "host":
        return list(step.run_host(x))
    if entry == "lazy":
        w = step.decide_accept_lazy(x)
        return _decision(step.decision) + _walk(w)
    if entry == "sampled":
        return _decision(step.decide_sampled(x, _TEMPERATURE, s["seed"]))
    if entry == "model":
        for layer, out in zip(s["layers"], s["outs"]):
            spiffy.spiffy_graph_attention(*layer, out=out, kernel=spiffy.ATTN_AUTO | spiffy.ATTN_EARLY_DEPENDENTS,
                                          dev_status=step.attn_status, workspace=step.attn_ws)
        w = step.decide_accept(x)
        return s["outs"] + _decision(step.decision) + _walk(w)
    w = step.run(x)
    return [step.attn_out, step.attn_status] + _decision(step.decision) + _walk(w)


# ---------------------------------------------------------------------------------------------
# What a pass cannot do without, and how far two correct builds may be apart
# ---------------------------------------------------------------------------------------------
def work(case):
    entry = case["entry"]
    B, N, L, P, Hq, Hkv, d, V = (case[k] for k in ("B", "N", "L", "P", "Hq", "Hkv", "d", "V"))
    e = 4 if case["dtype"] == "f32" else 2
    rows = B * N * L
    if entry == "full":
        S = case["suffix"]
        return {"bytes": e * B * d * (2 * (N * L + S) * Hq + 2 * (P + N * L + S) * Hkv),
                "flops": 4 * B * Hq * d * (N * L * (P + S + L) + S * (P + L + S))}
    if entry == "lmhead":
        H = case["hidden"]
        return {"bytes": 2 * H * (V + rows) + 12 * rows, "flops": 2 * _masked_rows(case) * V * H}
    # nodes outside the accepted path count for nothing in the lazy call: one draft in two or so is accepted
    masked = B * (_masked_at(case, 0) + 0.6 * _masked_at(case, 1)) if entry == "lazy" else _masked_rows(case)
    read = masked * V * e + 12 * rows
    if entry in ("lazy", "sampled", "draft"):
        return {"bytes": read, "flops": 0}
    layers = case.get("layers", 1)
    return {"bytes": read + layers * e * B * d * (2 * N * L * Hq + 2 * (P + N * L) * Hkv),
            "flops": layers * 4 * B * Hq * N * L * (P + L) * d}


def tolerance(case):
    entry = case["entry"]
    if entry == "host":
        return "exact"  # the verdict: tokens, indices and counts
    if entry == "lmhead":
        return {"rel": 1e-4, "max": 1e-2}  # fp32 sums of `hidden` products under an exponential
    if entry == "sampled":
        # a draw within rounding of the edge between two tokens may fall on either side
        return {"rel": 1e-4, "max": 1e-2, "differ": 5e-3}
    if entry in ("lazy", "draft") or case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-3}  # fp32 sums
    return {"rel": 1e-2, "max": 0.1}  # bf16 attention outputs, probabilities rounded to bf16
