"""The work that a user of the draft-then-verify library has it do, as cases that can be timed.

Five families, all through the ``Koala`` class of the package:

  eagle    one whole iteration of an EAGLE-style head: D x (draft, expand), verify, accept
  medusa   one whole iteration of Medusa-style heads on their static tree
  sampled  one iteration of a chain draft with speculative-sampling acceptance (temperature 1)
  decode   plain autoregressive decoding: a one-node tree per sequence, verified and accepted
  prefill  ingestion of a batch of prompts in chunks

on the shapes of ``workloads/configs.py``: the tiny fp32 target and the 7B- and 13B-shaped bf16
targets at full depth.  Weights are random N(0, 0.02); caches, pending hidden states and prompts are
random; accepted lengths are forced from a clipped Poisson(3), because random heads accept nothing.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2408_08146_b200 import Koala
from workloads.configs import EAGLE, FP32, T7_EAGLE, T7_MEDUSA, T13_EAGLE, TINY_EAGLE
from workloads.generate import forced_lengths, medusa_static_tree, torch_dtype, weight_shapes

SHAPES = {"tiny": TINY_EAGLE, "7b": T7_EAGLE, "13b": T13_EAGLE}


def case(family, model, batch=1, context=512, context_min=0, nodes=60, depth=5, topk=10, K=2, chunk=64):
    """context: longest context (prefill: longest prompt); the other sequences go down evenly to context_min."""
    return {"family": family, "model": model, "batch": batch, "context": context,
            "context_min": context_min or context, "nodes": nodes, "depth": depth, "topk": topk, "K": K, "chunk": chunk}


def listed():
    out = []

    def add(name, *a, **kw):
        out.append({"name": name, **case(*a, **kw)})

    # the smallest model: every kernel is a few microseconds, so launches and the host path are the time
    add("tiny_eagle_step", "eagle", "tiny", context=64, nodes=15, depth=4, topk=2)
    # interactive decoding of one sequence with Medusa-style heads (static 64-node tree)
    add("7b_medusa_step", "medusa", "7b", context=512, nodes=64, depth=4)
    # interactive decoding of one sequence with the two-layer EAGLE-style head (dynamic 60-node tree)
    add("7b_eagle_step", "eagle", "7b", context=1024)
    # the same with the largest tree and an odd, long context
    add("7b_eagle_wide_tree_step", "eagle", "7b", context=3989, nodes=128, K=1)
    # temperature-1 decoding: a chain of four drafted tokens, sampled and accepted by probability
    add("7b_sampled_chain_step", "sampled", "7b", context=777, nodes=5, depth=4, topk=1, K=1)
    # one token per forward: the baseline of every speed-up figure, and what a server falls back to
    add("7b_decode", "decode", "7b", context=1024)
    # the same for a ragged batch, on an engine that is otherwise set up for 64-node trees
    add("7b_decode_batch4", "decode", "7b", batch=4, context=1500, context_min=300, nodes=64)
    # a prompt of ordinary length before the first draft
    add("7b_prefill", "prefill", "7b", context=509)
    # a small serving batch, ragged contexts: the configuration of the benchmark
    add("13b_eagle_batch4_step", "eagle", "13b", batch=4, context=2048, context_min=512, nodes=64)
    # the largest iteration: eight sequences of 64 nodes in one verification
    add("7b_medusa_batch8_step", "medusa", "7b", batch=8, context=2048, context_min=700, nodes=64, depth=4)
    # prompts of a serving batch, ragged
    add("13b_prefill_batch4", "prefill", "13b", batch=4, context=1024, context_min=251, nodes=64)
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["eagle", "eagle", "medusa", "sampled", "decode", "prefill"])
    model = rng.choice(["tiny", "7b", "7b", "7b", "13b"])
    batch = rng.choice([1, 1, 1, 2, 3, 4] if model != "7b" else [1, 1, 1, 2, 4, 5, 8])
    if model == "tiny":
        context = _log_int(rng, 20, 400)
    elif family == "prefill":
        context = _log_int(rng, 40, 2048 if batch == 1 else 700)
    else:
        context = _log_int(rng, 128, 4096 if batch <= 2 else 2048)
    context_min = context if batch == 1 else max(16, int(context * rng.uniform(0.25, 1.0)))
    depth = rng.randint(3, 5)
    topk = rng.randint(2, 3) if model == "tiny" else rng.randint(4, 10)
    if family == "sampled":
        depth, topk = rng.randint(2, 5), 1
    K = rng.randint(1, 4) if model == "7b" else rng.randint(1, 2)
    if family == "medusa":
        depth, K = rng.randint(3, 4), rng.randint(1, 2)
    if family == "sampled":
        nodes = depth + 1
    elif family == "decode":
        nodes = rng.choice([1, 32, 60, 64])
    elif family == "prefill":
        nodes = rng.choice([60, 64, 128]) if batch == 1 else 64
    else:
        pool = topk + (depth - 1) * topk * topk if family == "eagle" else topk ** 2
        nodes = min(1 + pool, _log_int(rng, 16, 128) if batch <= 4 else _log_int(rng, 16, 64))
    chunk = min(nodes, rng.choice([32, 48, 64, 128])) if family == "prefill" else 64
    return case(family, model, batch, context, context_min, nodes, depth, topk, K, chunk)


def lengths(c):
    """Context (or prompt) length of every sequence: evenly from the longest down to the shortest."""
    b = c["batch"]
    if b == 1:
        return [c["context"]]
    return [c["context"] - (c["context"] - c["context_min"]) * i // (b - 1) for i in range(b)]


def config(c):
    base = SHAPES[c["model"]]
    common = dict(name="case", B=c["batch"], N=c["nodes"], D=c["depth"], topk=c["topk"], K=c["K"],
                  prompt_len=c["context"], prompt_len_min=0)
    common["S_max"] = (c["context"] + 2 * c["nodes"] + 64 + 127) // 128 * 128
    if c["family"] == "medusa":
        return base.with_(head_kind=T7_MEDUSA.head_kind, n_medusa_heads=c["depth"], **common)
    if c["family"] == "decode" and c["nodes"] == 1:
        common.update(D=1, topk=1, K=0)
    return base.with_(**common)


def _weights(cfg, g):
    """Random weights in the storage dtype; the rows of the LM head differ in length as trained ones do."""
    dt, out = torch_dtype(cfg), {}
    for name, shape in weight_shapes(cfg).items():
        t = torch.empty(shape, dtype=dt, device="cuda")
        out[name] = t.normal_(1.0 if name.endswith("norm") else 0.0, 0.02, generator=g)
    rows = torch.empty(cfg.V, 1, dtype=torch.float32, device="cuda").normal_(0.0, 0.4, generator=g)
    out["lm_head"].mul_(rows.exp().to(dt))
    return out


def prepare(c, seed):
    """The engine with its weights, and what a running program holds between two calls: filled caches, the
    last accepted tokens and their hidden states (prefill: the prompts instead)."""
    cfg = config(c)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rs = np.random.RandomState(int(seed) % (1 << 32))
    tree = medusa_static_tree(cfg.N, cfg.n_medusa_heads, cfg.topk) if c["family"] == "medusa" else None
    eng = Koala(cfg, _weights(cfg, g), static_tree=tree)
    s = SimpleNamespace(case=dict(c), cfg=cfg, eng=eng, buf=eng.buffers())
    lens = lengths(c)
    if c["family"] == "prefill":
        s.prompts = [rs.randint(0, cfg.V, n) for n in lens]
        return s
    for cache in (eng.target_k, eng.target_v, eng.draft_k, eng.draft_v):
        cache.normal_(0.0, 1.0, generator=g)
    # the last iteration accepted a few positions: their hidden states and tokens, and the next root
    pending = [1 + (2 + b) % min(cfg.D + 1, cfg.N) for b in range(cfg.B)]
    i32 = dict(dtype=torch.int32, device="cuda")
    s.start = [(eng.seq_len, torch.tensor(lens, **i32)),
               (s.buf["n_pend"], torch.tensor(pending, **i32)),
               (s.buf["root_tok"], torch.tensor(rs.randint(0, cfg.V, cfg.B), **i32)),
               (s.buf["pend_tok"], torch.tensor(rs.randint(0, cfg.V, (cfg.B, cfg.N)), **i32)),
               (s.buf["pend_hid"], torch.randn(cfg.B, cfg.N, cfg.H, device="cuda", generator=g))]
    if c["family"] == "decode":
        s.parent = torch.full((cfg.B, 1), -1, **i32)
        s.one = torch.ones(cfg.B, **i32)
        s.start = [s.start[0], s.start[2]]     # what a one-token step reads
    elif c["family"] == "sampled":
        s.u = [torch.rand(*shape, device="cuda", generator=g) for shape in ((cfg.B, cfg.D), (cfg.B, cfg.D), (cfg.B,))]
    else:
        s.forced = torch.tensor(forced_lengths(int(seed), cfg.B, hi=cfg.D + 1), **i32)
    return s


def run(s):
    eng, cfg, family = s.eng, s.cfg, s.case["family"]
    if family == "prefill":
        eng.seq_len.zero_()
        eng.prefill(s.prompts, s.case["chunk"])
        n_chunks = -(-max(len(p) for p in s.prompts) // s.case["chunk"])
        last = [len(np.array_split(p, n_chunks)[-1]) for p in s.prompts]      # tokens of the last chunk
        return {"seq_len": eng.seq_len, "root_tok": s.buf["root_tok"], "n_pend": s.buf["n_pend"],
                "pend_hid": [s.buf["pend_hid"][b, :n] for b, n in enumerate(last)],
                "caches": [eng.target_k, eng.target_v, eng.draft_k, eng.draft_v]}
    for now, then in s.start:       # every pass is the same iteration: put back what the last one advanced
        now.copy_(then)
    out = {}
    if family == "decode":
        eng.koala_verify((s.buf["root_tok"].view(cfg.B, 1), s.parent, s.one, 1))
        tokens, length = eng.koala_accept(None)
        # the rows in use: one per sequence
        out["logits"] = s.buf["verify_logits"].view(cfg.B, cfg.N, cfg.V)[:, 0]
        out["hidden"] = s.buf["verify_hid"].view(cfg.B, cfg.N, cfg.H)[:, 0]
    else:
        if family == "sampled":
            eng.koala_set_sampling(s.u[0])
            for p in range(cfg.D):
                eng.koala_draft(p)
                eng.koala_expand_tree(p)
            eng.koala_verify(None)
            tokens, length = eng.koala_accept_sampled(s.u[1], s.u[2])
        else:
            tokens, length = eng.step(s.forced)
        out["logits"], out["hidden"] = s.buf["verify_logits"], s.buf["verify_hid"]
        out["tree_tok"], out["tree_parent"] = s.buf["tree_tok"], s.buf["tree_parent"]
    out.update(tokens=tokens, length=length, seq_len=eng.seq_len,
               caches=[eng.target_k, eng.target_v, eng.draft_k, eng.draft_v])
    return out


def work(c):
    """Every weight matrix once per forward, the caches' context once per forward and layer, logits written once.
    A prompt counts as one forward; draft passes follow one another, so each counts."""
    cfg = config(c)
    e = 4 if cfg.dtype == FP32 else 2
    H, F, V, B = cfg.H, cfg.F, cfg.V, cfg.B
    layer, kv_tok = 4 * H * H + 3 * H * F, 2 * H * e          # weights of a layer; cache bytes of a token and layer
    ctx = lengths(c)
    total = sum(ctx)
    if c["family"] == "prefill":
        # causal attention over the prompt; logits of each sequence's last token; the head's pass over the same tokens
        pairs = sum(n * (n + 1) / 2 for n in ctx)
        layers = cfg.L + cfg.K
        flops = 2.0 * total * (layers * layer + 2 * H * H) + 2.0 * B * H * V + 4.0 * pairs * H * layers
        nbytes = e * (layers * layer + 2 * H * H + H * V + total * H) + total * kv_tok * layers + 4.0 * B * (V + H)
        return {"bytes": nbytes, "flops": flops}
    rows = B * (1 if c["family"] == "decode" else cfg.N)
    per_seq = rows // B
    nbytes = e * (cfg.L * layer + H * V + rows * H) + (total + rows) * kv_tok * cfg.L + 4.0 * rows * (V + H)
    flops = 2.0 * rows * (cfg.L * layer + H * V) + 4.0 * per_seq * total * H * cfg.L
    if c["family"] == "medusa":
        heads = cfg.n_medusa_heads
        nbytes += e * (heads * cfg.K * H * H + H * V) + 4.0 * heads * B * V
        flops += 2.0 * B * heads * (cfg.K * H * H + H * V)
    elif c["family"] in ("eagle", "sampled"):
        for p in range(cfg.D):
            r = B * cfg.topk if p else B * min(cfg.D + 1, cfg.N)
            lm = B * cfg.topk if p else B
            nbytes += e * (cfg.K * layer + 2 * H * H + H * V) + total * kv_tok * cfg.K + 4.0 * lm * V
            flops += 2.0 * r * (cfg.K * layer + 2 * H * H) + 2.0 * lm * H * V + 4.0 * (r // B) * total * H * cfg.K
    return {"bytes": nbytes, "flops": flops}


def tolerance(c):
    if config(c).dtype == FP32:
        return {"rel": 2e-5}
    # bf16 weights and caches; a near-tie among the drafted candidates may order a node differently
    return {"rel": 1e-2, "differ": 0.01}
