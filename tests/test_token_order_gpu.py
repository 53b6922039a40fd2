"""The fused call on the ALUs takes rows and keys in token order: ragged tiles, prefixes from the plan's own array where the host's
copy of the position may not be used, rows that see nothing."""
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


@pytest.mark.parametrize("n_q,n_kv,H,Hkv,d,B,J,P,dtype,causal,off", [
    (17, 33, 3, 1, 128, 1, 2, 2, "f32", True, 16),     # one row and one key past a tile
    (65, 65, 4, 2, 128, 8, 7, 30, "f32", True, 0),     # shards of two keys
    (100, 300, 6, 2, 64, 1, 3, 5, "f32", True, -30),   # the first rows see nothing
    (90, 200, 2, 2, 128, 40, 3, 4, "f32", False, 0),   # a last tile of 26 rows
    (33, 500, 4, 2, 128, 1, 4, 300, "bf16", True, 467),  # more shards than the tensor cores take
])
def test_fused_alu_call_in_token_order(gu, n_q, n_kv, H, Hkv, d, B, J, P, dtype, causal, off):
    gu.full_parity(wl.make_workload(f"order_{n_q}_{n_kv}", B, n_q, n_kv, H, Hkv, d, dtype, "random", "random", J, P, seed=n_q + P,
                                    causal=causal, q_pos_offset=off, symmetric=False))


@pytest.mark.parametrize("per_map", [False, True])
def test_fused_alu_call_over_resident_rows_and_captured(gu, per_map):
    from paper_2507_05228_b200 import binding as cb
    B, n, n_q, n_kv, H = 2, 300, 40, 120, 2
    rng = np.random.default_rng(per_map)
    w = wl.make_workload("resident_f32", B, n, n, H, H, 128, "f32", "random", "random", 1, 1, seed=8)
    q, k, v = gu.to_device(w)
    maps = B if per_map else 1
    pos = np.sort(np.stack([rng.choice(n, n_kv, replace=False) for _ in range(maps)]), axis=1).astype(np.int32)
    q_of, kv_of = rng.integers(0, 2, (maps, n_q)).astype(np.int32), rng.integers(0, 4, (maps, n_kv)).astype(np.int32)

    def reference(off, rows_of):
        seen = np.stack([rows_of[b % maps][None, :] <= np.arange(off, off + n_q)[:, None] for b in range(B)])
        kk, vv = (np.stack([a[b, rows_of[b % maps]] for b in range(B)]).astype(np.float64) for a in (w.k, w.v))
        s = np.einsum("bqhd,bkhd->bhqk", w.q[:, off:off + n_q].astype(np.float64), kk) * w.scale
        s = np.where(seen[:, None], s, -np.inf)
        e = np.exp(s - s.max(-1, keepdims=True))
        return np.einsum("bhqk,bkhd->bqhd", e / e.sum(-1, keepdims=True), vv)

    plan = cb.cascade_shard_plan_resident(q_of, kv_of, pos, 2, 4, 200)
    sel = [torch.from_numpy(pos[b % maps].astype(np.int64)).cuda() for b in range(B)]
    kr, vr = torch.stack([k[b, sel[b]] for b in range(B)]), torch.stack([v[b, sel[b]] for b in range(B)])
    for b in range(B):
        kr[b, sel[b] > 200 + n_q - 1] = float("nan")
    o, _ = cb.cascade_attn_sharded(plan, q[:, 200:200 + n_q], kr, vr, w.scale)
    gu.check_output(o, None, reference(200, pos), None, w.tol, "resident rows")
    plan.destroy()

    whole = np.tile(np.arange(n_kv, dtype=np.int32), (maps, 1))
    plan = cb.cascade_shard_plan(q_of, kv_of, 2, 4, 10, True)
    qc, o = q[:, 10:10 + n_q].clone(), torch.empty_like(q[:, :n_q])
    graph = torch.cuda.CUDAGraph()
    kc, vc = k[:, :n_kv].clone(), v[:, :n_kv].clone()
    with torch.cuda.graph(graph):
        cb.cascade_attn_sharded(plan, qc, kc, vc, w.scale, out=o, want_lse=False)
    for off in (10, 80, 0):
        qc.copy_(q[:, off:off + n_q])
        plan.advance(off)
        graph.replay()
        torch.cuda.synchronize()
        gu.check_output(o, None, reference(off, whole), None, w.tol, f"replayed at {off}")
    del graph
    plan.destroy()
