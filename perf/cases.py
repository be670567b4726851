"""What is timed of this library: the calls that a serving loop makes for one layer.

Each case is one turn's work on a ragged batch: new tokens go into the paged cache and attend
over it, or one generated token per sequence is appended and attends (decode).  Shapes are those
of this repository's workloads (`efim_synth.workloads`), of its serving replay and of its tests.

Fields of a case
  call        which public calls a pass makes:
              "step"    efim_append_prefill_step, the work list planned inside the call
              "turn"    efim_kv_append, then efim_append_prefill_attn planned inside the call
              "layer"   efim_kv_append, then the planned efim_append_prefill_attn whose lists are
                        in the workspace already: what every layer after a model's first one does
              "decode"  efim_decode_step (append and attention in one call)
              "attend"  efim_kv_append of one token per sequence, then efim_decode_attn
  batch, q_heads, kv_heads, head_dim
  cached_lo, cached_hi   tokens already in the cache, per sequence
  new_lo, new_hi         new tokens per sequence (1 for the decode calls)
  log_lengths            lengths are spread over their logarithm, else uniformly
  half_decode            every second sequence brings a single token (a mixed serving batch)
  interleaved            rotary pairs (2f, 2f+1) instead of (f, f + D/2)
  lse                    the caller asks for the log-sum-exp too
  shape_seed             draws the lengths
"""
import math
import random

import numpy as np
import torch

import paper_2505_21889_b200 as efim

PAGE = 16
ROPE_BASE = 10000.0

# (q heads, kv heads, head_dim): the repository's configurations, and the head_dim 64, small and
# wide-group ones of its tests
HEADS = ((4, 4, 64), (32, 32, 128), (28, 4, 128), (32, 8, 128), (32, 8, 64), (16, 1, 128), (24, 8, 128), (40, 8, 128))
DECODE_CALLS = ("decode", "attend")


def _case(name, call, batch, heads, cached, new=(1, 1), log_lengths=False, half_decode=False, interleaved=False,
          lse=False, shape_seed=0):
    return {"name": name, "call": call, "batch": batch, "q_heads": heads[0], "kv_heads": heads[1],
            "head_dim": heads[2], "cached_lo": cached[0], "cached_hi": cached[1], "new_lo": new[0],
            "new_hi": new[1], "log_lengths": log_lengths, "half_decode": half_decode, "interleaved": interleaved,
            "lse": lse, "shape_seed": shape_seed}


def listed():
    return [
        # One short request on a small layer: nothing but launches and latency.
        _case("turn_one_small", "step", 1, (4, 4, 64), (240, 240), (16, 16)),
        # One user's generated token over a typical infilling prompt: the latency of a decode step.
        _case("decode_one", "decode", 1, (32, 8, 128), (2314, 2314)),
        # Sixteen users, a few typed tokens each over prompts of a few thousand tokens that are cached
        # after the prompt transformation; every batch is new, so it is planned inside the call.
        _case("turn_users", "turn", 16, (32, 8, 128), (1100, 3400), (8, 112), shape_seed=1),
        # The same users when nothing is cached: the whole prompts.
        _case("prompt_users", "turn", 16, (32, 8, 128), (0, 0), (1100, 3500), shape_seed=2),
        # Decode of those users.
        _case("decode_users", "decode", 16, (32, 8, 128), (2000, 2900), shape_seed=3),
        # Equal head counts: 16 infilling requests over 2k to 8k cached tokens, one layer of the turn.
        _case("turn_mha", "layer", 16, (32, 32, 128), (2048, 8192), (32, 256), shape_seed=4),
        # Its decode step.
        _case("decode_mha", "decode", 16, (32, 32, 128), (2080, 8448), shape_seed=4),
        # A mixed serving batch at 7 query heads per kv head: half prefill rows, half single tokens.
        _case("mixed_batch", "layer", 64, (28, 4, 128), (1024, 16384), (1, 512), log_lengths=True, half_decode=True,
              lse=True, shape_seed=5),
        # Decode of such a model: plain decode attention behind the append.
        _case("decode_wide_group", "attend", 64, (28, 4, 128), (1024, 16384), log_lengths=True, lse=True, shape_seed=6),
        # Long prompts, prefix and suffix cached: 128 new tokens over 8,192.
        _case("turn_long", "layer", 8, (32, 8, 128), (8192, 8192), (128, 128)),
        # The same prompts when the suffix has to be recomputed: the largest contraction.
        _case("miss_long", "layer", 8, (32, 8, 128), (5120, 5120), (3200, 3200)),
        # Decode-heavy long-context serving: the largest read.
        _case("decode_long", "decode", 256, (32, 8, 128), (4096, 32768), shape_seed=7),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case of the same ranges, costing at most what the largest listed ones do."""
    while True:
        call = rng.choice(("step", "turn", "layer", "layer", "decode", "decode", "attend"))
        heads = rng.choice(HEADS)
        batch = _log_int(rng, 1, 256)
        cached_hi = _log_int(rng, 64, 32768)
        cached_lo = _log_int(rng, 16, cached_hi)
        log_lengths = rng.random() < 0.5
        new = (1, 1)
        half_decode = False
        if call not in DECODE_CALLS:
            new_hi = _log_int(rng, 1, 4096)
            new = (_log_int(rng, 1, new_hi), new_hi)
            if rng.random() < 0.15:
                cached_lo = cached_hi = 0          # a prompt of which nothing is cached
            half_decode = batch > 1 and rng.random() < 0.25
        c = _case("", call, batch, heads, (cached_lo, cached_hi), new, log_lengths, half_decode, rng.random() < 0.25,
                  rng.random() < 0.5, rng.randrange(1 << 30))
        del c["name"]
        w = work(c)
        # the listed cases end at 2.8 TFLOP and 19 GB; a pass of many tiny tiles takes longer per FLOP
        if w["flops"] <= 1.5e12 and w["bytes"] <= 10e9:
            return c


def _lengths(case):
    """Cached and new tokens of every sequence, from the case alone."""
    rng = random.Random(case["shape_seed"])

    def one(lo, hi):
        return _log_int(rng, lo, hi) if case["log_lengths"] and lo > 0 else rng.randint(lo, hi)
    cached = [one(case["cached_lo"], case["cached_hi"]) for _ in range(case["batch"])]
    new = [one(case["new_lo"], case["new_hi"]) for _ in range(case["batch"])]
    if case["half_decode"]:
        new = [1 if s % 2 else n for s, n in enumerate(new)]
    return np.array(cached, np.int32), np.array(new, np.int32)


def prepare(case, seed):
    """The layer's cache with the earlier turns' keys and values in it, this turn's q/k/v and what a
    serving loop keeps beside them: descriptors, rotary table, workspace, and the plan of a batch whose
    layers share one."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    hq, hkv, d, batch = case["q_heads"], case["kv_heads"], case["head_dim"], case["batch"]
    cached, new = _lengths(case)
    total = cached + new
    need = -(-total // PAGE)
    pages = int(need.sum()) + 16
    s = {"call": case["call"]}

    def normal(*shape):
        return torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
    s["k_pool"], s["v_pool"] = normal(pages, hkv, PAGE, d), normal(pages, hkv, PAGE, d)
    # pages scattered over the pool, as they are after many requests
    order = torch.randperm(pages, generator=gen, device=dev)[: int(need.sum())].to(torch.int32)
    table = torch.full((batch, int(need.max())), -1, dtype=torch.int32, device=dev)
    used = torch.arange(int(need.max()), device=dev)[None, :] < torch.from_numpy(need).to(dev)[:, None]
    table[used] = order
    tokens = int(new.sum())
    s["q"], s["k"], s["v"] = normal(tokens, hq, d), normal(tokens, hkv, d), normal(tokens, hkv, d)
    s["cache"] = efim.Cache(s["k_pool"], s["v_pool"], hq)
    s["batch"] = efim.Batch(cached, new, table)
    s["rope"] = efim.Rope(ROPE_BASE, d, int(total.max()), case["interleaved"])
    s["out"] = torch.empty_like(s["q"])
    s["lse"] = torch.empty((tokens, hq), dtype=torch.float32, device=dev) if case["lse"] else None
    s["status"] = torch.zeros(1, dtype=torch.int32, device=dev)
    if case["call"] in DECODE_CALLS:
        s["ctx"] = torch.from_numpy(total).to(dev)
        s["max_ctx"] = int(total.max())
        need_bytes = efim.efim_decode_workspace_bytes(s["cache"], batch, s["max_ctx"])
    else:
        need_bytes = efim.efim_prefill_workspace_bytes(s["cache"], s["batch"])
    s["workspace"] = torch.empty(max(need_bytes, 256), dtype=torch.uint8, device=dev)
    if case["call"] == "layer":
        # the first layer of the batch leaves the plan's lists in the workspace
        s["plan"] = efim.efim_prefill_plan(s["cache"], s["batch"])
        efim.efim_append_prefill_attn(s["cache"], s["batch"], s["q"], s["out"], s["lse"], 0.0, s["workspace"],
                                      s["status"], plan=s["plan"])
    return s


def run(s):
    """One layer's pass; q is rotated in place where efim_kv_append is called for it, as it is for a
    projection's fresh output."""
    call, cache, batch, rope = s["call"], s["cache"], s["batch"], s["rope"]
    if call == "step":
        efim.efim_append_prefill_step(cache, batch, rope, s["q"], s["k"], s["v"], s["out"], s["lse"], 0.0,
                                      s["workspace"], s["status"])
    elif call == "turn":
        efim.efim_kv_append(cache, batch, rope, s["q"], s["k"], s["v"], s["status"])
        efim.efim_append_prefill_attn(cache, batch, s["q"], s["out"], s["lse"], 0.0, s["workspace"], s["status"])
    elif call == "layer":
        efim.efim_kv_append(cache, batch, rope, s["q"], s["k"], s["v"], s["status"])
        efim.efim_append_prefill_attn(cache, batch, s["q"], s["out"], s["lse"], 0.0, s["workspace"], s["status"],
                                      plan=s["plan"], lists_resident=True)
    elif call == "decode":
        efim.efim_decode_step(cache, batch.desc.batch, s["ctx"], s["max_ctx"], batch.d_block_table, rope, s["q"],
                              s["k"], s["v"], s["out"], s["lse"], 0.0, s["workspace"], s["status"])
    else:
        efim.efim_kv_append(cache, batch, rope, s["q"], s["k"], s["v"], s["status"])
        efim.efim_decode_attn(cache, batch.desc.batch, s["ctx"], s["max_ctx"], batch.d_block_table, s["q"], s["out"],
                              s["lse"], 0.0, s["workspace"], s["status"])
    return {"out": s["out"], "lse": s["lse"], "q": s["q"], "k_pool": s["k_pool"], "v_pool": s["v_pool"],
            "status": s["status"]}


def work(case):
    """Bytes: q, k, v and the cached keys and values read once, the new keys and values, the output, the
    log-sum-exp and, where the append rotates it in place, q written once, a rotary row per new token.
    Operations: two contractions over every (query, visible key) pair."""
    cached, new = (x.astype(np.int64) for x in _lengths(case))
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    tokens = int(new.sum())
    pairs = int((new * cached + new * (new + 1) // 2).sum())
    q_row, kv_row = 2 * hq * d, 2 * 2 * hkv * d
    q_written = 0 if case["call"] in ("step", "decode") else q_row
    n_bytes = tokens * (2 * q_row + q_written + 2 * kv_row + 4 * d + (4 * hq if case["lse"] else 0))
    n_bytes += int(cached.sum()) * kv_row
    return {"bytes": n_bytes, "flops": 4 * d * hq * pairs}


def tolerance(case):
    """About four times the error measured against a recomputation in 64 bits: decode 1.7e-3 (2-norm; the
    rounding of the output to bf16 alone is 1.66e-3) and 4e-3 (largest); append-prefill, whose
    probabilities are bf16 too, 2.4e-3 and 1.2e-2, 3.6e-2 where rows see only a few keys."""
    if case["call"] in DECODE_CALLS:
        return {"rel": 6.5e-3, "max": 1.6e-2}
    return {"rel": 9.5e-3, "max": 0.14 if case["cached_lo"] < 256 else 5e-2}
