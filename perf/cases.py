"""The attention layer as a user of this framework runs it: the measured cases.

A case is one call (or one short sequence of calls) that a program makes per layer, per decode step or per request:

  fused   cascade_attn_sharded on device tensors            prefill of one layer, all shards walked in one call
  rope    cascade_attn_sharded_rope                         the same with unrotated q, k
  nodes   cascade_attn_partials, then cascade_merge         the attention-pass of every node, then the post-pass
  chunk   Plan.advance, then cascade_attn_sharded           one chunk of a chunked prefill over a preallocated cache
  decode  cascade_attn_sharded with one query row           one generated token against a token-sharded cache
  step    cascade_decode_step_rope                          the same with plan advance, cache append and rotary step
  host    cascade_attn_sharded_host                         q, k, v and o in pinned host memory
  prompt  cascade_shard_plan, then cascade_attn_sharded     first layer of a new prompt: its shard map is new too

Output and scratch tensors are allocated once and handed to every call, as a serving program does; "prompt" leaves both to
the library's defaults.
"""
import math

import numpy as np
import torch

from paper_2507_05228_b200 import binding as cb
from paper_2507_05228_b200 import workloads as wl

ROPE_BASE = 500000.0


def _case(name, kind, B, n_q, n_kv, H, Hkv, d, dtype, shards, sharding, **more):
    c = dict(kind=kind, B=B, n_q=n_q, n_kv=n_kv, H=H, Hkv=Hkv, d=d, dtype=dtype, shards=shards, sharding=sharding,
             causal=True, offset=n_kv - n_q, outliers=False, map_per_sequence=False)
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # One encoder layer on a short prompt, two parties, bidirectional: the paper's own latency shape.  Launch bound.
        _case("encoder_128_f32", "fused", 1, 128, 128, 12, 12, 64, "f32", 2, "clusters", causal=False),
        # A batch of full-length encoder sequences through the nodes and the post-pass in fp32.
        _case("encoder_512_b16_f32_nodes", "nodes", 16, 512, 512, 16, 16, 64, "f32", 8, "clusters", causal=False),
        # Heads of 64 columns in bf16, two sequences of an odd length.
        _case("d64_3001_b2_bf16", "fused", 2, 3001, 3001, 16, 4, 64, "bf16", 8, "random"),
        # The prompt of one chat turn: one sequence, 32 query and 8 KV heads, eight random shards.
        _case("prefill_2k", "fused", 1, 2048, 2048, 32, 8, 128, "bf16", 8, "random"),
        # Batched long prompts with the rotary step left to the library; some keys dominate their rows.
        _case("prefill_8k_b4_rope", "rope", 4, 8192, 8192, 32, 8, 128, "bf16", 16, "blocks", outliers=True),
        # The largest: a document of 32768 tokens, 64 query heads, 32 x 32 shards.
        _case("prefill_32k", "fused", 1, 32768, 32768, 64, 8, 128, "bf16", 32, "random"),
        # Nodes and post-pass as separate parties run them, at a length that no tile divides.
        _case("nodes_4099", "nodes", 1, 4099, 4099, 32, 8, 128, "bf16", 16, "clusters"),
        # A request arrives: its shard map is drawn, the plan is built, the first layer runs.
        _case("prompt_1500", "prompt", 1, 1500, 1500, 32, 8, 128, "bf16", 8, "random"),
        # Chunked prefill: 512 new tokens near the end of a cache of 8192.
        _case("chunk_512_of_8k", "chunk", 1, 512, 8192, 32, 8, 128, "bf16", 16, "blocks", offset=6656),
        # A full decode batch over long caches: bound by the reads of the cache.
        _case("decode_16k_b64", "decode", 64, 1, 16384, 32, 8, 128, "bf16", 16, "random"),
        # One user's decode step in the middle of a cache of 4096 rows: latency.
        _case("step_4k_b1", "step", 1, 1, 4096, 32, 8, 128, "bf16", 8, "clusters", offset=2500),
        # The whole call on host buffers: copies in both directions and compute.
        _case("host_2k", "host", 1, 2048, 2048, 32, 8, 128, "bf16", 8, "random"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["fused", "fused", "f32", "d64", "rope", "nodes", "prompt", "chunk", "decode", "step", "host"])
    sharding = rng.choice(["random", "blocks", "clusters"])
    per_seq = rng.random() < 0.25
    if kind == "f32":  # encoder shapes and small causal models in fp32
        n, heads = _log_int(rng, 33, 1024), rng.choice([8, 12, 16])
        return _case(None, rng.choice(["fused", "nodes"]), rng.choice([1, 2, 4, 8]), n, n, heads, heads, 64, "f32",
                     rng.choice([2, 4, 8]), sharding, causal=rng.random() < 0.5, map_per_sequence=per_seq)
    if kind == "d64":
        n, (H, Hkv) = _log_int(rng, 128, 4096), rng.choice([(12, 12), (16, 16), (16, 4), (32, 8)])
        return _case(None, rng.choice(["fused", "nodes"]), 1 if n > 2048 else rng.choice([1, 2]), n, n, H, Hkv, 64, "bf16",
                     rng.choice([2, 4, 8]), sharding, causal=rng.random() < 0.75, map_per_sequence=per_seq)
    H, Hkv = rng.choice([(32, 8), (32, 8), (64, 8), (16, 8), (8, 8)])
    if kind in ("decode", "step"):
        n = _log_int(rng, 512, 16384)
        B = _log_int(rng, 1, max(1, min(64, (64 * 16384) // n)))
        return _case(None, kind, B, 1, n, H, Hkv, 128, "bf16", rng.choice([4, 8, 16]), sharding,
                     offset=rng.randrange(n // 2, n), map_per_sequence=per_seq)
    if kind == "chunk":
        n, rows = _log_int(rng, 1024, 16384), _log_int(rng, 64, 1024)
        return _case(None, kind, rng.choice([1, 2, 4]), rows, n, H, Hkv, 128, "bf16", rng.choice([4, 8, 16]), sharding,
                     offset=rng.randrange(0, n - rows + 1), map_per_sequence=per_seq)
    n = _log_int(rng, 128, {"host": 4096, "nodes": 8192, "prompt": 8192}.get(kind, 24576))
    B = 1 if n > 8192 else rng.choice([1, 2, 4])
    return _case(None, kind, B, n, n, H, Hkv, 128, "bf16", rng.choice([4, 8, 16] if n < 2048 else [8, 16, 32]), sharding,
                 outliers=rng.random() < 0.25, map_per_sequence=per_seq)


def _shard_of(case, n, seed):
    """Token-to-shard map(s) [n] or [B, n]: random equal shards, blocks of 64 dealt in turn, or clusters of 8 tokens."""
    maps = []
    for b in range(case["B"] if case["map_per_sequence"] else 1):
        if case["sharding"] == "random":
            maps.append(wl.shard_map("random", n, case["shards"], np.random.default_rng([seed, b, n])))
        elif case["sharding"] == "blocks":
            maps.append(np.roll(wl.shard_map("block_rr", n, case["shards"], block=64), 64 * b))
        else:
            maps.append(np.roll(cb.cascade_cdelta_shard_map(n, 8, 8 * case["shards"])[0], 8 * b))
    return np.stack(maps) if case["map_per_sequence"] else maps[0]


def prepare(case, seed):
    B, n_q, n_kv, H, Hkv, d = (case[x] for x in ("B", "n_q", "n_kv", "H", "Hkv", "d"))
    kind, dtype = case["kind"], torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    gen = torch.Generator(device="cuda").manual_seed(int(seed))

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).to(dtype)

    q, k, v = normal(B, n_q, H, d), normal(B, n_kv, Hkv, d), normal(B, n_kv, Hkv, d)
    if case["outliers"]:  # one key row in a hundred is eight times as long
        rows = torch.randperm(n_kv, generator=gen, device="cuda")[: max(1, n_kv // 100)]
        k[:, rows] *= 8
    kv_map = _shard_of(case, n_kv, seed)
    if n_q == n_kv:
        q_map, q_shards = kv_map, case["shards"]
    elif n_q == 1:
        q_map, q_shards = np.zeros(kv_map.shape[:-1] + (1,), np.int32), 1
    else:  # a chunk's queries sit in the shards of the tokens they are
        q_map, q_shards = kv_map[..., case["offset"]: case["offset"] + n_q], case["shards"]
    s = dict(case=case, q=q, k=k, v=v, scale=1.0 / math.sqrt(d), q_map=q_map, kv_map=kv_map, q_shards=q_shards)
    if kind == "prompt":
        return s
    plan = s["plan"] = cb.cascade_shard_plan(q_map, kv_map, q_shards, case["shards"], case["offset"], case["causal"])
    call = {"nodes": cb.CALL_PARTIALS, "step": cb.CALL_DECODE_STEP_ROPE, "host": cb.CALL_SHARDED_HOST}.get(kind, cb.CALL_SHARDED)
    code = cb.F32 if case["dtype"] == "f32" else cb.BF16
    s["ws"] = torch.empty(cb.cascade_workspace_bytes(plan, call, code, B, H, Hkv, d), dtype=torch.uint8, device="cuda")
    s["o"] = torch.empty_like(q)
    if kind == "nodes":
        P = case["shards"]
        s["parts"] = (torch.empty((B, P, n_q, H, d), dtype=dtype, device="cuda"),
                      torch.empty((B, P, n_q, H), dtype=torch.float32, device="cuda"),
                      torch.empty((B, P, n_q, H), dtype=torch.float32, device="cuda"))
        s["rows"] = plan.dev_ptr("q_idx")
        s["row_stride"] = n_q if case["map_per_sequence"] else 0
    if kind in ("rope", "step"):
        s["table"] = cb.cascade_rope_table(n_kv, d, ROPE_BASE)
    if kind == "step":
        s["k_new"], s["v_new"] = normal(B, 1, Hkv, d), normal(B, 1, Hkv, d)
    if kind == "host":
        s["q"], s["k"], s["v"] = (t.cpu().pin_memory() for t in (q, k, v))
        s["o"] = torch.empty_like(s["q"]).pin_memory()
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "prompt":
        plan = cb.cascade_shard_plan(s["q_map"], s["kv_map"], s["q_shards"], case["shards"], case["offset"], case["causal"])
        out = cb.cascade_attn_sharded(plan, s["q"], s["k"], s["v"], s["scale"])
        plan.destroy()
        return out
    plan, q, k, v, scale, o, ws = s["plan"], s["q"], s["k"], s["v"], s["scale"], s["o"], s["ws"]
    if kind == "rope":
        return cb.cascade_attn_sharded_rope(plan, q, k, v, scale, s["table"], out=o, want_lse=False, workspace=ws)[0]
    if kind == "nodes":
        parts = cb.cascade_attn_partials(plan, q, k, v, scale, out=s["parts"], workspace=ws)
        merged, _ = cb.cascade_merge(*parts, s["rows"], s["row_stride"], out=o, want_lse=False)
        return parts, merged
    if kind == "step":
        out, _ = cb.cascade_decode_step_rope(plan, q, s["k_new"], s["v_new"], k, v, case["offset"], scale, s["table"], out=o,
                                             want_lse=False, workspace=ws)
        return out, k, v
    if kind == "host":
        cb.cascade_attn_sharded_host(plan, q, k, v, scale, o, ws)
        torch.cuda.current_stream().synchronize()  # the result is read on the host
        return o
    if kind == "chunk":
        plan.advance(case["offset"])
    return cb.cascade_attn_sharded(plan, q, k, v, scale, out=o, want_lse=False, workspace=ws)[0]


def work(case):
    B, n_q, n_kv, H, Hkv, d = (case[x] for x in ("B", "n_q", "n_kv", "H", "Hkv", "d"))
    es = 4 if case["dtype"] == "f32" else 2
    first, last = case["offset"] + 1, min(case["offset"] + n_q, n_kv)  # keys the first and the last query row sees
    if case["causal"]:
        pairs, seen = n_q * (first + last) // 2, last
    else:
        pairs, seen = n_q * n_kv, n_kv
    rows = B * n_q * H
    nbytes = 2 * rows * d * es + 2 * B * seen * Hkv * d * es
    if case["kind"] == "nodes":  # the partials are an output of the nodes and the input of the post-pass
        nbytes += 2 * case["shards"] * rows * (d * es + 8)
    if case["kind"] == "rope":
        nbytes += last * d * 4
    if case["kind"] == "step":
        nbytes += 4 * B * Hkv * d * es
    if case["kind"] == "prompt":
        nbytes += rows * 4 + 8 * n_kv
    return {"bytes": nbytes, "flops": 4 * d * H * B * pairs}


def tolerance(case):
    # fp32 products and sums; bf16 weights and outputs (the row sums stay in fp32)
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}
