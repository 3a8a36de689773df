"""The work that users of this package have it do, as sized cases: one pass is one eviction step of a KV cache.

A step appends the new tokens' K and V rows, attends over the cache, scores every cached token by the output error of
its eviction, selects down to the budget and compacts the cache in place. The caches here are in the steady state a
running system is in: at their budget before the step, so that every step appends ``m`` tokens and evicts as many.

A case's keys:
  batch, q_heads, kv_heads, head_dim, dtype ("bf16" | "f32")
  m         new tokens (= query rows per head) per step: 1 = decode, more = a block of a prompt
  budget    tokens kept per (sequence, KV head)
  ragged    every sequence has a budget of its own, uniform in [3/4 budget, budget]
  base      base score: "last_query" (TOVA), "chunk_sum" (H2O over one block), "accum" (H2O carried across steps),
            "external" (a score of the caller's, such as SnapKV's, handed over at every step)
  method    "caote" | "fast" (FastCAOTE) | "sum_errors" | "post_evict" (the output over the retained tokens is
            returned too) | "greedy" (one token at a time, every eviction changing the scores of the rest)
  compact   "fill" | "stable"
"""
import math

import torch

import paper_2504_14051_b200 as P

RING = 4  # different steps' inputs that a state goes through in turn

# Head counts of the attention layers in use here: grouped-query layers of 7B, 8B, 70B models, ungrouped ones, and one
# with a large group.
HEADS = [(32, 8), (28, 4), (64, 8), (16, 8), (24, 8), (8, 8), (32, 2)]


def _case(name, batch, heads, head_dim, dtype, m, budget, base, ragged=False, method="caote", compact="fill"):
    c = {} if name is None else {"name": name}
    c.update(batch=batch, q_heads=heads[0], kv_heads=heads[1], head_dim=head_dim, dtype=dtype, m=m, budget=budget,
             ragged=ragged, base=base, method=method, compact=compact)
    return c


def listed():
    return [
        # Decode: one new token per sequence.
        # The smallest configuration of the package (fp32, two KV heads, 256 tokens): latency and launches only.
        _case("decode_tiny_f32", 1, (4, 2), 64, "f32", 1, 255, "last_query"),
        # One user's chat on an 8B-class layer with a 2k budget: a few megabytes per step.
        _case("decode_single", 1, (32, 8), 128, "bf16", 1, 2048, "last_query"),
        # A serving batch on a 7B-class layer, ragged budgets up to 8k, accumulated scores.
        _case("decode_batch", 64, (28, 4), 128, "bf16", 1, 8192, "accum", ragged=True),
        # Few sequences with long budgets on a 70B-class layer.
        _case("decode_long", 8, (64, 8), 128, "bf16", 1, 16384, "last_query"),
        # Heads of 64 channels, as small models have them, in a batch of ragged 4k caches.
        _case("decode_d64", 16, (32, 8), 64, "bf16", 1, 4096, "accum", ragged=True),
        # FastCAOTE on a mid-sized batch with an odd budget.
        _case("decode_fast", 24, (28, 4), 128, "bf16", 1, 2999, "accum", ragged=True, method="fast"),
        # Prefill: a block of a prompt goes through a cache that is at its budget.
        # The usual block of 128 tokens at a 4k budget, one layer of one prompt.
        _case("prefill_block", 1, (32, 8), 128, "bf16", 128, 4096, "chunk_sum"),
        # What is left of two prompts after their full blocks.
        _case("prefill_tail", 2, (28, 4), 128, "bf16", 45, 3001, "chunk_sum", ragged=True),
        # Long-context prefill on a 70B-class layer: blocks of 512 at a 16k budget.
        _case("prefill_long", 8, (64, 8), 128, "bf16", 512, 16384, "chunk_sum"),
        # TOVA as the base score of block-wise prefill; the model goes on with the output over the retained tokens.
        _case("prefill_tova", 4, (28, 4), 128, "bf16", 128, 6000, "last_query", method="post_evict"),
        # H2O as the base score, carried from block to block, prompts of different budgets.
        _case("prefill_h2o", 4, (32, 8), 128, "bf16", 128, 8192, "accum", ragged=True),
        # The same base score with greedy eviction of the block's 128 tokens.
        _case("prefill_greedy", 1, (32, 8), 128, "bf16", 128, 4096, "accum", method="greedy"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the ranges of ``listed``: decode and prefill in equal shares, sizes over their logarithm."""
    while True:
        decode = rng.random() < 0.5
        heads = rng.choice(HEADS)
        head_dim = 64 if rng.random() < 0.2 else 128
        dtype = "f32" if rng.random() < 0.1 else "bf16"
        ragged = rng.random() < 0.5
        base = rng.choice(["last_query", "chunk_sum", "accum", "accum", "external"])
        method, compact = "caote", "fill"
        if decode:
            batch, m, budget = _log(rng, 1, 64), 1, _log(rng, 128, 16384)
            method = rng.choice(["caote", "caote", "caote", "fast", "sum_errors", "post_evict"])
            compact = "stable" if rng.random() < 0.1 else "fill"
        else:
            batch, m = _log(rng, 1, 8), rng.choice([128, 128, 512, _log(rng, 2, 512)])
            budget = max(_log(rng, 512, 16384), 2 * m)
            method = rng.choice(["caote", "caote", "caote", "fast", "post_evict", "greedy"])
        if method == "sum_errors" and base not in ("last_query", "chunk_sum"):
            base = "last_query"
        if method == "greedy":
            base, batch, budget, m = "accum", min(batch, 2), min(budget, 8192), min(m, 128)
        if dtype == "f32":
            batch, budget, m = min(batch, 4), min(budget, 2048), min(m, 128)
        c = _case(None, batch, heads, head_dim, dtype, m, budget, base, ragged, method, compact)
        w = work(c)
        if w["bytes"] <= 1.0e9 and w["flops"] <= 2.0e11:
            return c


def _budgets(case, seed):
    b = torch.full((case["batch"],), case["budget"], dtype=torch.int32)
    if case["ragged"]:
        g = torch.Generator().manual_seed(seed)
        b = torch.randint(case["budget"] * 3 // 4, case["budget"] + 1, (case["batch"],), generator=g, dtype=torch.int32)
    return b


def prepare(case, seed):
    """The cache at its budget and the inputs of the next steps.

    Values and keys are normal, with three outlier channels per KV head on the keys and four attention sinks that the
    queries lean towards; H2O sums and external scores are positive with a long tail.
    """
    dev, m, d = "cuda", case["m"], case["head_dim"]
    B, Hq, Hkv = case["batch"], case["q_heads"], case["kv_heads"]
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    cap = (case["budget"] + m + 15) // 16 * 16
    g = torch.Generator(device=dev).manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, generator=g, device=dev)

    mult = torch.ones((Hkv, 1, d), device=dev)
    mult[:, :, torch.randperm(d, generator=g, device=dev)[:3]] = 4.0
    mu = normal(Hkv, 1, d)
    mu = mu / mu.norm(dim=-1, keepdim=True)
    k = normal(B, Hkv, cap, d) * mult
    k[:, :, :4] = 2.0 * math.sqrt(d) * mu
    budgets = _budgets(case, seed).to(dev)
    cache = P.EvictionCache(B, Hq, Hkv, d, cap, m, dtype, budgets, base_mode=case["base"],
                            compact_mode=case["compact"],
                            method="caote" if case["method"] == "greedy" else case["method"])
    heavy = normal(RING, B, Hkv, cap).exp_() if case["base"] in ("accum", "external") else None
    cache.load(k.to(dtype), normal(B, Hkv, cap, d).to(dtype), budgets,
               base=heavy[0] if case["base"] == "accum" else None)
    lean = 2.0 * mu.repeat_interleave(Hq // Hkv, dim=0)
    steps = []
    for i in range(RING):
        steps.append({"q": (normal(B, Hq, m, d) + lean).to(dtype), "k": (normal(B, Hkv, m, d) * mult).to(dtype),
                      "v": normal(B, Hkv, m, d).to(dtype),
                      "h": heavy[i] if case["base"] == "external" else None})
    return {"cache": cache, "steps": steps, "at": 0, "method": case["method"]}


def _bytes_of(t):
    """A cache's rows are moved and never computed: they are handed back as whole numbers, bit for bit."""
    return t.view(torch.int16 if t.dtype == torch.bfloat16 else torch.int32)


def run(state):
    c, s = state["cache"], state["steps"][state["at"] % RING]
    state["at"] += 1
    p, ws = c.params, c.workspace
    if state["method"] == "greedy" or s["h"] is not None:
        # the caller has a part of its own in the step: a scoring of its own, or another selection
        P.caote_append(p, c.K, c.V, c.base, c.pos, c.lens, c.n_seen, s["k"], s["v"], ws)
        if s["h"] is not None:
            c.base.copy_(s["h"])
        if c.method == "fast":
            P.caote_vsum(p, c.V, c.lens, c.vsum)
            P.caote_score_fast(p, s["q"], c.K, c.V, c.lens, c.base, c.vsum, c.o, c.scores, ws)
        else:
            P.caote_score(p, s["q"], c.K, c.V, c.lens, c.base, c.o, c.scores, ws)
        o = c.o
        if state["method"] == "greedy":
            P.caote_select_evict_greedy(p, c.V, c.base, c.lens, c.budget, c.pos, c.evict_idx, None, c.n_evict, ws)
        else:
            P.caote_select_evict(p, c.scores, c.lens, c.budget, c.pos, c.evict_idx, c.n_evict, ws)
        if c.method == "post_evict":
            P.caote_post_evict_output_ws(p, s["q"], c.K, c.V, c.lens, c.evict_idx, c.n_evict, c.o, c.o_post, ws)
            o = c.o_post
        P.caote_compact(p, c.K, c.V, c.base, c.pos, c.lens, c.evict_idx, c.n_evict, c.compact_mode, ws)
    else:
        o = c.step(s["q"], s["k"], s["v"])
    out = {"o": o, "scores": c.scores, "K": _bytes_of(c.K), "V": _bytes_of(c.V), "pos": c.pos, "len": c.lens,
           "n_evict": c.n_evict}
    if c.method == "post_evict":
        out["o_before"] = c.o
    if c.vsum is not None:
        out["vsum"] = c.vsum
    if s["h"] is None and c.params.base_mode == P.binding.BASE_MODES["accum"]:
        out["base"] = c.base
    return out


def work(case):
    """One read of the cache and of the step's inputs, one write of the outputs, of the appended and of the moved rows;
    the two products of attention and the distances (greedy: distances for every pick)."""
    B, Hq, Hkv, d, m = (case[k] for k in ("batch", "q_heads", "kv_heads", "head_dim", "m"))
    e = 2 if case["dtype"] == "bf16" else 4
    n = case["budget"] * (7 / 8 if case["ragged"] else 1.0) + m
    units = B * Hkv
    per_token = 2 * d * e + 4  # K and V rows in, a score out
    if case["base"] in ("accum", "external"):
        per_token += 8 if case["base"] == "accum" else 4
    per_new = 2 * (2 * d * e) + 2 * (2 * d * e)  # appended (read, written), and as many moved by the compaction
    nbytes = units * (n * per_token + m * per_new) + B * Hq * m * d * (e + 4)
    if case["method"] == "post_evict":
        nbytes += B * Hq * m * d * 4
    if case["compact"] == "stable":
        nbytes += units * n * (2 * d * e)  # half of the rows lie behind an evicted token: read and written
    picks = m if case["method"] == "greedy" else 1
    flops = units * (4.0 * (Hq // Hkv) * m * n * d + 3.0 * n * d * picks)
    if case["method"] == "sum_errors":
        flops += units * 3.0 * n * d * (Hq // Hkv - 1)
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    """fp32 sums: about 1e-6 off a computation in 64 bits, whatever the length. bf16 caches: products on the tensor
    cores, whose running sums drift with the length of the chain (o is 5e-6 off at 4 224 tokens and 6.5e-5 at 16 896,
    its largest element 1.9e-4). Whole numbers (positions, lengths, the rows' bits) differ only where two tokens' scores
    tie within that."""
    rel = 1e-5 if case["dtype"] == "f32" else 3e-4 * max(case["budget"] + case["m"], 1700) / 17000
    return {"rel": rel, "max": 4 * rel, "differ": 1e-2}
