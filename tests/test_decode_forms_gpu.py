"""Fused decode where a warp lists its blocks by itself (up to 32 shards, up to ten blocks a warp) and where it requests two blocks
ahead (few KV heads and sequences): edges of both, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2507_05228_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gu():
    import gpu_util
    return gpu_util


@pytest.mark.parametrize("B,n_kv,H,Hkv,P,kv_map,pos", [
    (1, 2049, 64, 8, 8, "random", 2048),      # two blocks ahead, eight heads; one key past a block
    (1, 4097, 32, 8, 32, "contiguous", 4000), # 32 shards, the last ones empty: shard after shard, found by search
    (1, 4097, 32, 8, 33, "contiguous", 4000), # one shard more: the table
    (1, 1281, 8, 8, 5, "random", 1280),       # two blocks ahead, nearly every warp with one block
    (1, 20000, 16, 8, 16, "random", 19000),   # more than ten blocks a warp: two ahead, from the table
    (1, 45000, 16, 8, 5, "random", 44990),    # more than 32 blocks a warp: the list is made a second time
    (3, 3000, 8, 4, 8, "random", 2999),       # 12 KV heads and sequences: their clusters do not all get an SM for each CTA
    (2, 12000, 32, 8, 8, "random", 11999),    # ten CTAs of eight warps a pair, from the table
    (2, 1280, 32, 8, 8, "random", 1279),      # four heads, one block ahead: a block a warp, listed
    (2, 1281, 64, 8, 8, "random", 1280),      # eight heads: a block more, from the table
    (1, 17, 4, 1, 2, "contiguous", 16),       # two blocks, one of them a single key
    (3, 200, 2, 2, 32, "random", 3),          # four keys in all, most shards empty
])
def test_decode_lists_and_widths(gu, B, n_kv, H, Hkv, P, kv_map, pos):
    gu.full_parity(wl.make_workload(f"lists_{B}_{n_kv}_{P}", B, 1, n_kv, H, Hkv, 128, "bf16", "round_robin", kv_map, 1, P, seed=n_kv + P,
                                    q_pos_offset=pos))


@pytest.mark.parametrize("n_kv,H,Hkv,P,pos", [
    (1500, 8, 8, 8, 1400),      # one block a warp, some with two
    (4096, 32, 8, 8, 2500),     # two and three
    (8192, 16, 2, 40, 8000),    # 33 shards and more: the table
    (24000, 16, 8, 16, 23000),  # 18, from the table
])
def test_a_sequence_has_the_same_bits_alone_and_beside_another(gu, n_kv, H, Hkv, P, pos):
    """As many CTAs a sequence in both calls; alone, a warp requests two blocks ahead.  What it adds up, and in which order, stays."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload(f"alone_{n_kv}", 2, 1, n_kv, H, Hkv, 128, "bf16", "round_robin", "random", 1, P, seed=n_kv, q_pos_offset=pos)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    for b in range(2):
        o1, lse1 = cb.cascade_attn_sharded(plan, q[b:b + 1], k[b:b + 1], v[b:b + 1], w.scale)
        assert torch.equal(o1[0], o[b]) and torch.equal(lse1[0], lse[b])
    plan.destroy()


def test_captured_decode_follows_the_plan(gu):
    """Captured where few keys are visible, replayed where many are."""
    from paper_2507_05228_b200 import binding as cb
    B, n_kv, H, Hkv, P = 1, 3000, 32, 8, 8
    w = wl.make_workload("captured_decode", B, n_kv, n_kv, H, Hkv, 128, "bf16", "random", "random", 1, 1, seed=12)
    q, k, v = gu.to_device(w)
    kv_of = np.random.default_rng(1).integers(0, P, n_kv).astype(np.int32)
    plan = cb.cascade_shard_plan(np.zeros(1, np.int32), kv_of, 1, P, 5, True)
    qc = q[:, :1].clone()
    ws = torch.empty(cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.BF16, B, H, Hkv, 128), dtype=torch.uint8, device="cuda")
    o = torch.zeros_like(qc)
    cb.cascade_attn_sharded(plan, qc, k, v, w.scale, out=o, want_lse=False, workspace=ws)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cb.cascade_attn_sharded(plan, qc, k, v, w.scale, out=o, want_lse=False, workspace=ws)
    for pos in (5, 2999, 700):
        qc.copy_(q[:, pos:pos + 1])
        plan.advance(pos)
        graph.replay()
        torch.cuda.synchronize()
        o_ref, _ = oracle.attention_unsharded(w.q[:, pos:pos + 1], w.k, w.v, w.scale, q_pos_offset=pos)
        gu.check_output(o, None, o_ref, None, w.tol, f"replayed at {pos}")
    del graph
    plan.destroy()
