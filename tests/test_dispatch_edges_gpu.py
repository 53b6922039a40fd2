"""Sizes at which a kernel or a dispatch rule changes what it does: edges of tiles, remainders, the smallest and the largest
of a range.  Reference and tolerances are those of the parity tests."""
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


@pytest.mark.parametrize("n,H,Hkv,shards,causal", [
    (2, 4, 4, 1, True),        # one tile of one chunk
    (129, 8, 1, 3, True),      # eight stacked heads, a last tile of one row
    (1153, 16, 4, 2, True),    # ten 128-key tiles: every logit buffer and stage is used several times over
    (700, 12, 12, 5, False),   # no stacking, one sub-tile per CTA, bidirectional
    (1500, 6, 2, 40, True),    # three heads per KV head: no stacking although heads are shared; many short shards
])
def test_head_dim_64_on_the_tensor_cores(gu, n, H, Hkv, shards, causal):
    gu.full_parity(wl.make_workload(f"d64_{n}", 2, n, n, H, Hkv, 64, "bf16", "random", "random", shards, shards, seed=n,
                                    causal=causal))


def test_head_dim_64_warps_at_different_speeds(gu):
    """Cold caches and many short shards let the warps of a sub-tile drift a tile apart; every run is the same."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("d64_drift", 2, 1500, 1500, 6, 2, 64, "bf16", "random", "random", 40, 40, seed=1500)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for i in range(20):
        flush.fill_(i)
        o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
        gu.check_output(o, lse, o_ref, lse_ref, w.tol, f"run {i}")
    assert plan.device_status() == 0
    plan.destroy()


def test_head_dim_64_partials_with_cold_caches(gu):
    """Shards of more than one tile, written out while the products of the last two tiles may be under way."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("d64_cold", 1, 300, 700, 4, 4, 64, "bf16", "random", "random", 3, 5, seed=1000, q_pos_offset=400,
                         symmetric=False)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    u, m, e = oracle.attn_pass(w.q, w.k, w.v, w.scale, gu.oracle_plan(w))
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for i in range(20):
        flush.fill_(i)
        parts = cb.cascade_attn_partials(plan, q, k, v, w.scale)
        gu.check_partials(tuple(t.double().cpu().numpy() for t in parts), (u, m, e), w.tol, f"run {i}")
    assert plan.device_status() == 0
    plan.destroy()


def test_head_dim_64_without_a_workspace_takes_the_alu_kernel(gu):
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("d64_nows", 1, 200, 200, 8, 2, 64, "bf16", "random", "random", 3, 3, seed=7)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o = torch.empty_like(q)
    S = cb._strides
    rc = cb.lib().cascade_attn_sharded(plan.handle, cb.BF16, w.B, w.H, w.Hkv, w.d, w.scale, q.data_ptr(), S(q), k.data_ptr(),
                                       S(k), v.data_ptr(), S(v), o.data_ptr(), S(o), None, None, 0,
                                       torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    o_ref, _ = oracle.attention_unsharded(w.q, w.k, w.v, w.scale)
    gu.check_output(o, None, o_ref, None, w.tol, "no workspace")
    plan.destroy()


def test_head_dim_64_with_too_small_a_workspace(gu):
    """Heads of 64 columns never needed scratch memory: what is too small or misaligned for the tensor-core route is left
    alone, and the ALU kernel runs.  The host call's workspace without scratch for its head groups likewise."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("d64_small_ws", 1, 200, 200, 8, 2, 64, "bf16", "random", "random", 3, 3, seed=8)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    u, m, e = oracle.attn_pass(w.q, w.k, w.v, w.scale, gu.oracle_plan(w))
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale)
    need = cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.BF16, 1, 8, 2, 64)
    raw = torch.full((need + 16,), 0x5A, dtype=torch.uint8, device="cuda")
    for ws in (raw[:need - 256], raw[16:], raw[:16]):
        o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale, workspace=ws)
        gu.check_output(o, lse, o_ref, lse_ref, w.tol, "small workspace")
        parts = cb.cascade_attn_partials(plan, q, k, v, w.scale, workspace=ws)
        gu.check_partials(tuple(t.double().cpu().numpy() for t in parts), (u, m, e), w.tol, "small workspace")
    assert (raw == 0x5A).all()
    hq, hk, hv = (t.cpu().pin_memory() for t in (q, k, v))
    ho = torch.empty_like(hq).pin_memory()
    staging = sum((t.numel() * 2 + 255) // 256 * 256 for t in (hq, hk, hv, ho))
    raw = torch.full((staging + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    cb.cascade_attn_sharded_host(plan, hq, hk, hv, w.scale, ho, raw[:staging])
    torch.cuda.synchronize()
    gu.check_output(ho.double().numpy(), None, o_ref, None, w.tol, "host call without scratch")
    assert (raw[staging:] == 0x5A).all()
    with pytest.raises(cb.CascadeError) as ei:
        cb.cascade_attn_sharded_host(plan, hq, hk, hv, w.scale, ho, raw[:staging - 256])
    assert ei.value.status == 4
    plan.destroy()


def test_fp32_host_call_with_any_workspace_that_holds_the_staging(gu):
    """fp32, heads of 64: from the staging alone up to a byte less than all, the head groups take the ALU kernel."""
    from paper_2507_05228_b200 import binding as cb
    B, n, H = 8, 300, 16
    w = wl.make_workload("d64_f32_host_ws", B, n, n, H, H, 64, "f32", "random", "random", 3, 3, seed=10)
    plan = gu.make_plan(w)
    o_ref, _ = oracle.attention_unsharded(w.q, w.k, w.v, w.scale)
    hq, hk, hv = (torch.from_numpy(a).pin_memory() for a in (w.q, w.k, w.v))
    ho = torch.empty_like(hq).pin_memory()
    staging = 4 * ((hq.numel() * 4 + 255) // 256 * 256)
    total = cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED_HOST, cb.F32, B, H, H, 64)
    assert total > staging + 512  # the head groups would use the rest
    raw = torch.full((total + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    for size in (staging, staging + 256, staging + 257, total - 1):
        ho.zero_()
        cb.cascade_attn_sharded_host(plan, hq, hk, hv, w.scale, ho, raw[:size])
        torch.cuda.synchronize()
        gu.check_output(ho.double().numpy(), None, o_ref, None, w.tol, f"host call with {size - staging} bytes of scratch")
        assert (raw[staging:] == 0x5A).all()
    with pytest.raises(cb.CascadeError) as ei:
        cb.cascade_attn_sharded_host(plan, hq, hk, hv, w.scale, ho, raw[:staging - 1])
    assert ei.value.status == 4
    plan.destroy()


@pytest.mark.parametrize("n_q,n_kv,H,Hkv,d,B,shards,dtype,causal", [
    (1, 1, 2, 2, 64, 1, 1, "f32", True),          # one key
    (1, 300, 6, 2, 64, 2, 3, "bf16", True),       # one query row on the ALU route: key groups share the row
    (17, 33, 3, 1, 128, 1, 2, "f32", False),      # one row and one key more than a piece / a tile
    (640, 640, 8, 8, 64, 8, 4, "f32", True),      # on the tensor cores; on the ALUs see the next test
    (512, 512, 4, 4, 128, 12, 4, "f32", False),   # wide form at head_dim 128
    (300, 300, 8, 8, 64, 8, 60, "f32", True),     # the same, with five keys per shard
])
def test_alu_kernel_forms(gu, n_q, n_kv, H, Hkv, d, B, shards, dtype, causal):
    gu.full_parity(wl.make_workload(f"alu_{n_q}_{d}", B, n_q, n_kv, H, Hkv, d, dtype, "random", "random",
                                    1 if n_q == 1 else shards, shards, seed=n_q + d, causal=causal))


@pytest.mark.parametrize("n,H,Hkv,B,J,P,causal", [
    (640, 8, 8, 8, 4, 4, True),     # wide form: 64-row tiles, masked and unmasked 64-key tiles
    (512, 8, 8, 8, 4, 4, False),    # the same without a mask
    (300, 8, 8, 8, 60, 60, True),   # partials a row at a time over five keys per shard; the fused call in the wide form
    (64, 4, 2, 8, 64, 4, True),     # partials of one row per query shard: one row of a tile of 32
])
def test_alu_kernels_without_scratch(gu, n, H, Hkv, B, J, P, causal):
    """fp32, heads of 64: problems that the tensor cores take when a caller brings the scratch, without it."""
    w = wl.make_workload(f"alu_no_ws_{n}", B, n, n, H, Hkv, 64, "f32", "random", "random", J, P, seed=n + 1, causal=causal, symmetric=False)
    gu.full_parity(w, scratch=False)


@pytest.mark.parametrize("n_q,n_kv,P,causal", [(128, 128, 2, True), (129, 200, 2, True), (300, 900, 7, False), (40, 64, 64, True)])
def test_new_plans_have_the_same_arrays_on_the_device(gu, n_q, n_kv, P, causal):
    """vis and pair_class come from the host up to 256 entries and from a kernel above; two plans alive at a time, and a
    third in memory that a destroyed one gave back."""
    from paper_2507_05228_b200 import binding as cb
    rng = np.random.default_rng(n_kv)
    plans = []
    for _ in range(3):
        q_of, kv_of = rng.integers(0, 3, n_q).astype(np.int32), rng.integers(0, P, n_kv).astype(np.int32)
        plan = cb.cascade_shard_plan(q_of, kv_of, 3, P, n_kv - n_q, causal)
        ref = oracle.shard_plan(q_of, kv_of, 3, P, q_pos_offset=n_kv - n_q, causal=causal)
        for f in ("q_off", "q_idx", "q_inv", "kv_off", "kv_idx", "kv_inv", "vis", "pair_class"):
            assert np.array_equal(gu.read_plan_device_array(plan, f)[0], getattr(ref, f)), f
            assert np.array_equal(plan.get(f)[0], getattr(ref, f)), f
        assert plan.device_status() == 0
        plans.append(plan)
        if len(plans) == 2:
            plans.pop(0).destroy()
    for plan in plans:
        plan.destroy()


@pytest.mark.parametrize("n_q,n_kv,H,Hkv,d,B,J,P,dtype,causal", [
    (64, 64, 16, 16, 64, 1, 32, 32, "f32", True),     # partials of two rows and two keys each
    (64, 64, 4, 2, 64, 8, 64, 4, "f32", True),        # one row per query shard: partials on the tensor cores, without scratch see above
    (64, 64, 2, 2, 128, 1, 64, 1, "f32", True),       # fused route, a row at a time
    (333, 333, 8, 8, 64, 1, 32, 12, "f32", False),    # tiles of 10 rows, the last tile of a shard short of keys
    (130, 130, 12, 12, 64, 1, 40, 40, "bf16", True),  # heads of 64 in bf16: partials on the ALUs, the fused call on the tensor cores
    (128, 128, 8, 2, 128, 2, 128, 2, "f32", True),    # head_dim 128
    (1, 1000, 16, 16, 64, 8, 1, 8, "bf16", True),     # one query row
    (300, 300, 4, 2, 128, 1, 290, 280, "bf16", True), # more shards than the tensor cores take, some of them empty
])
def test_row_kernel_forms(gu, n_q, n_kv, H, Hkv, d, B, J, P, dtype, causal):
    """Problems cut so fine that a query row at a time is the faster way for the partials.  (The fused call of most takes tiles of tokens.)"""
    gu.full_parity(wl.make_workload(f"rows_{n_q}_{d}", B, n_q, n_kv, H, Hkv, d, dtype, "random", "random", J, P, seed=n_q + d,
                                    causal=causal, symmetric=False, q_pos_offset=n_kv - n_q))


@pytest.mark.parametrize("n_q,n_kv,same,n_maps", [
    (1, 1, True, 1), (333, 333, True, 2), (333, 333, False, 2), (65536, 65536, True, 1), (1, 65537, False, 1), (65537, 65537, True, 1)])
def test_plan_lists_go_up_narrow_and_once(gu, n_q, n_kv, same, n_maps):
    """Row ids travel as 16 bits up to 65536 rows and as 32 above, and once where both sides have the same lists."""
    from paper_2507_05228_b200 import binding as cb
    rng = np.random.default_rng(n_kv)
    kv_of = rng.integers(0, 4, (n_maps, n_kv)).astype(np.int32)
    q_of = kv_of if same else rng.integers(0, 4, (n_maps, n_q)).astype(np.int32)
    plan = cb.cascade_shard_plan(q_of, kv_of, 4, 4, n_kv - n_q, True)
    for mp in range(n_maps):
        ref = oracle.shard_plan(q_of[mp], kv_of[mp], 4, 4, q_pos_offset=n_kv - n_q, causal=True)
        for f in ("q_off", "q_idx", "q_inv", "kv_off", "kv_idx", "kv_inv", "vis", "pair_class"):
            assert np.array_equal(gu.read_plan_device_array(plan, f)[mp], getattr(ref, f)), f
    plan.destroy()


@pytest.mark.parametrize("B,n_kv,H,Hkv,P,kv_map,pos", [
    (1, 1, 8, 8, 1, "random", 0),            # one key, one block: a single CTA per KV head
    (1, 129, 16, 2, 3, "contiguous", 64),    # two of three shards empty or cut: shard-after-shard order
    (2, 4097, 8, 4, 16, "round_robin", 4096),  # prefixes that differ by one block at most: interleaved order
    (1, 9000, 8, 1, 300, "random", 8999),    # more shards than one table window
    (5, 700, 4, 1, 7, "random", 699),        # fewer than eight (KV head, sequence) pairs: the largest clusters
    (40, 333, 32, 8, 5, "block_rr", 300),    # more pairs than 256: one CTA each
    (20, 2000, 32, 8, 8, "random", 1999),    # more than 128 pairs: clusters of three or more, the last round partly filled
    (45, 1500, 16, 8, 4, "random", 1400),    # clusters of four or five
])
def test_fused_decode_forms(gu, B, n_kv, H, Hkv, P, kv_map, pos):
    gu.full_parity(wl.make_workload(f"dec_{B}_{n_kv}", B, 1, n_kv, H, Hkv, 128, "bf16", "round_robin", kv_map, 1, P,
                                    seed=n_kv, block=16, q_pos_offset=pos))


@pytest.mark.parametrize("B,P,per_seq", [(2, 5, False), (3, 100, True), (2, 300, False)])
def test_decode_step_moves_the_plan_with_few_and_with_many_prefixes(gu, B, P, per_seq):
    """Up to 256 prefixes travel with the launch, more are searched for on the device; either way the plan's arrays end up
    as those of a plan built at that position, the new rows are in the caches, and the output is the oracle's."""
    from oracle import rope
    from paper_2507_05228_b200 import binding as cb
    cap, H, Hkv, d, base = 700, 8, 2, 128, 10000.0
    rng = np.random.default_rng(P)
    maps = rng.integers(0, P, (B, cap)).astype(np.int32) if per_seq else rng.integers(0, P, cap).astype(np.int32)
    q_map = np.zeros((B, 1) if per_seq else (1,), np.int32)
    plan = cb.cascade_shard_plan(q_map, maps, 1, P, 0, True)
    w = wl.make_workload("step", B, cap, cap, H, Hkv, d, "bf16", "random", "random", 1, 1, seed=P)
    q, k, v = gu.to_device(w)
    table = cb.cascade_rope_table(cap, d, base)
    qr = rope.rotary_pos_emb(w.q, np.arange(cap), base, "bf16").astype(np.float32)
    kr = rope.rotary_pos_emb(w.k, np.arange(cap), base, "bf16").astype(np.float32)
    k_cache, v_cache = torch.full_like(k, float("nan")), torch.full_like(v, float("nan"))
    known = torch.from_numpy(wl.bf16_bits(kr).view(np.int16)).cuda().view(torch.bfloat16)
    for pos in (0, 1, 300, 699):
        k_cache[:, :pos], v_cache[:, :pos] = known[:, :pos], v[:, :pos]
        o, lse = cb.cascade_decode_step_rope(plan, q[:, pos:pos + 1], k[:, pos:pos + 1], v[:, pos:pos + 1], k_cache, v_cache,
                                             pos, w.scale, table)
        o_ref, lse_ref = oracle.attention_unsharded(qr[:, pos:pos + 1], kr, w.v, w.scale, causal=True, q_pos_offset=pos)
        gu.check_output(o, lse, o_ref, lse_ref, w.tol, f"step at {pos}")
        got, want = k_cache[:, pos].double().cpu().numpy(), kr[:, pos]
        assert (np.abs(got - want) <= np.maximum(np.abs(want), 2.0 ** -126) * 2.0 ** -7).all()  # one bf16 step
        assert torch.equal(v_cache[:, pos], v[:, pos])
        for b in range(plan.n_maps):
            op = oracle.shard_plan(q_map[b] if per_seq else q_map, maps[b] if per_seq else maps, 1, P, q_pos_offset=pos)
            assert np.array_equal(gu.read_plan_device_array(plan, "vis")[b], op.vis)
            assert np.array_equal(gu.read_plan_device_array(plan, "pair_class")[b], op.pair_class)
            assert np.array_equal(plan.get("vis")[b], op.vis)
    plan.destroy()


@pytest.mark.parametrize("n_maps", [1, 3])
def test_decode_step_of_a_token_in_one_of_several_query_shards(gu, n_maps):
    """The prefixes travel with the launch; the pair classes that the step leaves behind are those of the shard that owns the
    query row, in every map, and a second plan update finds them so."""
    from paper_2507_05228_b200 import binding as cb
    cap, H, Hkv, J, P, B = 300, 8, 2, 6, 5, 3
    rng = np.random.default_rng(n_maps)
    kv_of = rng.integers(0, P, (n_maps, cap)).astype(np.int32)
    q_of = rng.integers(1, J, (n_maps, 1)).astype(np.int32)
    plan = cb.cascade_shard_plan(q_of, kv_of, J, P, 0, True)
    w = wl.make_workload("step_J", B, cap, cap, H, Hkv, 128, "bf16", "random", "random", 1, 1, seed=n_maps)
    q, k, v = gu.to_device(w)
    table = cb.cascade_rope_table(cap, 128, 10000.0)
    for pos in (7, 299):
        cb.cascade_decode_step_rope(plan, q[:, :1], k[:, :1], v[:, :1], k.clone(), v.clone(), pos, w.scale, table)
        for m in range(n_maps):
            ref = oracle.shard_plan(q_of[m], kv_of[m], J, P, q_pos_offset=pos, causal=True)
            for f in ("vis", "pair_class"):
                assert np.array_equal(gu.read_plan_device_array(plan, f)[m], getattr(ref, f)), (f, pos, m)
                assert np.array_equal(plan.get(f)[m], getattr(ref, f)), (f, pos, m)
    plan.destroy()


@pytest.mark.parametrize("n_q,n_kv,H,Hkv,d,B,off,causal", [
    (2, 2, 8, 8, 128, 1, 0, True),           # one tile; the rows see one and two keys
    (65, 1025, 32, 8, 128, 1, 960, True),    # keys shared by clusters of 8; a second query tile of one row, one key past a tile
    (200, 640, 8, 4, 128, 2, 0, True),       # clusters of 8 where the first tiles see fewer than 8 key tiles: idle ranks
    (300, 700, 16, 4, 64, 2, 400, True),     # clusters of 4 at head_dim 64
    (512, 900, 32, 8, 128, 1, 100, True),    # clusters of 2; keys past the last query position are not looked at
    (130, 300, 12, 3, 128, 1, 0, False),     # every key for every row, shared
    (40, 500, 4, 2, 128, 1, -20, True),      # the first rows see nothing
])
def test_fused_route_in_token_order(gu, n_q, n_kv, H, Hkv, d, B, off, causal):
    w = wl.make_workload(f"tok_{n_q}_{n_kv}", B, n_q, n_kv, H, Hkv, d, "bf16", "random", "random", 3, 5, seed=n_q + n_kv,
                         causal=causal, q_pos_offset=off, symmetric=False)
    gu.full_parity(w)


@pytest.mark.parametrize("n,H,Hkv,d", [(1, 8, 8, 64), (15, 8, 1, 128), (17, 8, 1, 128), (129, 4, 4, 128), (257, 6, 3, 64)])
@pytest.mark.parametrize("n_q_extra", [1, 40])
def test_query_boxes_at_the_end_of_the_tensor(gu, n, H, Hkv, d, n_q_extra):
    """The last box of query rows reaches past the tokens of the sequence (here into the next one's, and past the last)."""
    from paper_2507_05228_b200 import binding as cb
    n_q, n_kv = n + n_q_extra, n + 300
    w = wl.make_workload(f"boxes_{n}_{d}", 3, n_q, n_kv, H, Hkv, d, "bf16", "random", "random", 2, 2, seed=n + d,
                         q_pos_offset=n_kv - n_q, causal=True)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, causal=True, q_pos_offset=w.q_pos_offset)
    gu.check_output(o, lse, o_ref, lse_ref, w.tol, w.name)
    assert plan.device_status() == 0
    plan.destroy()


@pytest.mark.parametrize("n_q", [70, 700])
def test_fused_route_with_strides_a_tensor_map_cannot_hold(gu, n_q):
    """K and V of one sequence expanded over the batch (stride 0) go through a copy; the result is the same, bit for bit."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("expanded", 2, n_q, 700, 8, 2, 128, "bf16", "random", "random", 2, 3, seed=n_q, symmetric=False)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    k1, v1 = k[:1].expand(2, -1, -1, -1), v[:1].expand(2, -1, -1, -1)
    o_a, lse_a = cb.cascade_attn_sharded(plan, q, k1, v1, w.scale)
    o_b, lse_b = cb.cascade_attn_sharded(plan, q, k1.contiguous(), v1.contiguous(), w.scale)
    assert torch.equal(o_a, o_b) and torch.equal(lse_a, lse_b)
    table = cb.cascade_rope_table(700, 128, 10000.0)
    o_a, _ = cb.cascade_attn_sharded_rope(plan, q, k1, v1, w.scale, table)
    o_b, _ = cb.cascade_attn_sharded_rope(plan, q, k1.contiguous(), v1.contiguous(), w.scale, table)
    assert torch.equal(o_a, o_b)
    plan.destroy()


@pytest.mark.parametrize("n_q,n_kv,hidden", [
    (300, 300, 200),    # the first tile, and a part of the second
    (64, 1200, 1000),   # keys shared by a cluster: whole parts, and the start of the last one
    (64, 1200, 130),    # only the first part's first tile
])
def test_logits_of_minus_infinity_before_finite_ones(gu, n_q, n_kv, hidden):
    """Keys so long that their logits overflow to -inf have weight 0 (in the fp64 oracle exp(-1e40) is 0 too): the rows that
    see others are the softmax over those, although a first tile leaves them without a finite maximum."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload(f"minus_inf_{hidden}", 1, n_q, n_kv, 8, 2, 128, "bf16", "random", "random", 2, 3, seed=hidden,
                         symmetric=False, q_pos_offset=n_kv - n_q)
    w.q[:] = np.abs(w.q)
    w.k[:, :hidden] = -(2.0 ** 127)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, q_pos_offset=w.q_pos_offset)
    rows = np.arange(n_q) + w.q_pos_offset >= hidden
    gu.check_output(o[:, rows], lse[:, rows], o_ref[:, rows], lse_ref[:, rows], w.tol, "rows with finite logits")
    plan.destroy()


@pytest.mark.parametrize("n_q,n_kv", [(700, 700), (100, 4000)])  # the second shares keys in clusters
def test_row_sums_where_few_keys_dominate(gu, n_q, n_kv):
    """One key in a hundred is eight times as long, so a row's weight sits on a few keys of any tile.  The fused call sums the
    weights in fp32: 2^-22 of each, and logits of up to 40 in fp32, 4e-6 on average with room.  The partials sum the largest
    weight of a tile as its bf16 rounding, which is exact where the key became the reference: on average below a fifth of
    bf16's half step of 2^-9."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("peaked", 1, n_q, n_kv, 8, 2, 128, "bf16", "random", "random", 4, 8, seed=n_q, symmetric=False,
                         q_pos_offset=n_kv - n_q, outlier_frac=0.01)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    _, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    _, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, q_pos_offset=w.q_pos_offset)
    assert np.abs(lse.double().cpu().numpy() - lse_ref).mean() < 4e-6
    _, _, l = cb.cascade_attn_partials(plan, q, k, v, w.scale)
    _, _, e = oracle.attn_pass(w.q, w.k, w.v, w.scale, gu.oracle_plan(w))
    there = e > 0
    assert (np.abs(l.double().cpu().numpy() - e)[there] / e[there]).mean() < 2.0 ** -9 / 5
    plan.destroy()


@pytest.mark.parametrize("n_maps", [1, 2])
def test_fused_route_over_resident_rows(gu, n_maps):
    """Rows with positions of their own: a query sees those at positions up to its own, and what lies behind may be NaN."""
    from paper_2507_05228_b200 import binding as cb
    rng = np.random.default_rng(n_maps)
    n, n_q, n_kv, B = 600, 90, 250, 2
    w = wl.make_workload("resident", B, n, n, 8, 2, 128, "bf16", "random", "random", 2, 2, seed=61)
    q, k, v = gu.to_device(w)
    pos = np.sort(np.stack([rng.choice(n, n_kv, replace=False) for _ in range(n_maps)]), axis=1).astype(np.int32)
    off, q_of, kv_of = 300, rng.integers(0, 2, (n_maps, n_q)).astype(np.int32), rng.integers(0, 4, (n_maps, n_kv)).astype(np.int32)
    plan = cb.cascade_shard_plan_resident(q_of, kv_of, pos, 2, 4, off)
    sel = [torch.from_numpy(pos[b % n_maps].astype(np.int64)).cuda() for b in range(B)]
    kr, vr = torch.stack([k[b, sel[b]] for b in range(B)]), torch.stack([v[b, sel[b]] for b in range(B)])
    qr = q[:, off:off + n_q].contiguous()
    for b in range(B):
        hidden = sel[b] > off + n_q - 1
        kr[b, hidden], vr[b, hidden] = float("nan"), float("nan")
    o, lse = cb.cascade_attn_sharded(plan, qr, kr, vr, w.scale)
    keep = np.full((B, n), -np.inf)
    for b in range(B):
        keep[b, pos[b % n_maps]] = 0.0
    G = 4
    logits = np.einsum("bqhd,bkhd->bhqk", w.q[:, off:off + n_q].astype(np.float64), np.repeat(w.k, G, 2).astype(np.float64)) * w.scale
    causal = np.where(np.arange(n)[None, :] <= np.arange(off, off + n_q)[:, None], 0.0, -np.inf)
    logits = logits + keep[:, None, None, :] + causal[None, None]
    m = logits.max(-1, keepdims=True)
    e = np.exp(logits - m)
    o_ref = np.einsum("bhqk,bkhd->bqhd", e / e.sum(-1, keepdims=True), np.repeat(w.v, G, 2).astype(np.float64))
    lse_ref = (m[..., 0] + np.log(e.sum(-1))).transpose(0, 2, 1)
    gu.check_output(o, lse, o_ref, lse_ref, w.tol, "resident rows, fused")
    plan.destroy()


@pytest.mark.parametrize("d,n_maps,P", [(128, 1, 5), (128, 2, 5), (64, 1, 5), (128, 1, 1)])
def test_captured_call_follows_the_plan(gu, d, n_maps, P):
    """A call captured into a graph is replayed after plan updates outside the graph: it sees what the plan says then, and
    what lies behind the new position may be NaN."""
    from paper_2507_05228_b200 import binding as cb
    n_q, n_kv, B = 64, 600, 2
    w = wl.make_workload("captured", B, n_kv, n_kv, 8, 2, d, "bf16", "random", "random", 1, 1, seed=d + P)
    q, k, v = gu.to_device(w)
    rng = np.random.default_rng(P)
    kv_of = rng.integers(0, P, (n_maps, n_kv)).astype(np.int32)
    q_of = rng.integers(0, 3, (n_maps, n_q)).astype(np.int32)
    plan = cb.cascade_shard_plan(q_of, kv_of, 3, P, 100, True)
    qc, kc, vc = q[:, :n_q].clone(), torch.full_like(k, float("nan")), torch.full_like(v, float("nan"))
    ws = torch.empty(cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.BF16, B, 8, 2, d), dtype=torch.uint8, device="cuda")
    o = torch.zeros_like(qc)
    parts = [t.clone() for t in cb.cascade_attn_partials(plan, qc, k, v, w.scale, workspace=ws)]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        cb.cascade_attn_sharded(plan, qc, kc, vc, w.scale, out=o, want_lse=False, workspace=ws)
        cb.cascade_attn_partials(plan, qc, kc, vc, w.scale, out=parts, workspace=ws)
    for off in (100, 300, 536, 20):
        seen = off + n_q
        qc.copy_(q[:, off:seen])
        kc.fill_(float("nan")), vc.fill_(float("nan"))
        kc[:, :seen], vc[:, :seen] = k[:, :seen], v[:, :seen]
        plan.advance(off)
        graph.replay()
        torch.cuda.synchronize()
        o_ref, lse_ref = oracle.attention_unsharded(w.q[:, off:seen], w.k, w.v, w.scale, q_pos_offset=off)
        gu.check_output(o, None, o_ref, None, w.tol, f"captured at 100, replayed at {off}")
        for b in range(B):
            op = oracle.shard_plan(q_of[b % n_maps], kv_of[b % n_maps], 3, P, q_pos_offset=off, causal=True)
            u, m, e = oracle.attn_pass(w.q[b:b + 1, off:seen], w.k[b:b + 1], w.v[b:b + 1], w.scale, op)
            gu.check_partials(tuple(t[b:b + 1].double().cpu().numpy() for t in parts), (u, m, e), w.tol, f"partials at {off}")
    del graph
    plan.destroy()


@pytest.mark.parametrize("n_q,n_kv", [(300, 300), (64, 1200)])
def test_calls_on_a_plan_whose_status_word_is_set_write_nothing(gu, n_q, n_kv):
    """Once a wait inside the tensor-core kernel has given up, later calls on the plan leave their outputs alone (here the
    word is set from outside; the second size shares keys in clusters).  With the word cleared the plan works again."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("gave_up", 1, n_q, n_kv, 8, 2, 128, "bf16", "random", "random", 2, 3, seed=n_q, symmetric=False,
                         q_pos_offset=n_kv - n_q)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    table = cb.cascade_rope_table(n_kv, 128, 10000.0)
    word = torch.as_tensor(gu._DevicePointer(plan.dev_ptr("q_off") - 256, 1, "<i4"), device="cuda")  # first in the plan's memory
    assert word.item() == 0
    word.fill_(5)
    with pytest.raises(cb.CascadeError) as ei:
        plan.device_status()
    assert ei.value.status == 7
    o = torch.full_like(q, 7.0)
    parts = (torch.full((1, 3, n_q, 8, 128), 7.0, dtype=q.dtype, device="cuda"), torch.full((1, 3, n_q, 8), 7.0, device="cuda"),
             torch.full((1, 3, n_q, 8), 7.0, device="cuda"))
    cb.cascade_attn_sharded(plan, q, k, v, w.scale, out=o)
    cb.cascade_attn_sharded_rope(plan, q, k, v, w.scale, table, out=o)
    cb.cascade_attn_partials(plan, q, k, v, w.scale, out=parts)
    torch.cuda.synchronize()
    assert all((t == 7.0).all() for t in (o, *parts))
    word.fill_(0)
    cb.cascade_attn_sharded(plan, q, k, v, w.scale, out=o)
    o_ref, _ = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, q_pos_offset=w.q_pos_offset)
    gu.check_output(o, None, o_ref, None, w.tol, "after the word was cleared")
    plan.destroy()


@pytest.mark.parametrize("P", [1, 4])
def test_captured_rotary_call(gu, P):
    """Captured, the rotary call copies keys and values in token order; what lies behind the last query may be NaN, and the
    workspace holds the same as after a plain call."""
    from paper_2507_05228_b200 import binding as cb
    n_q, n_kv, off = 64, 400, 200
    w = wl.make_workload("captured_rope", 2, n_q, n_kv, 8, 2, 128, "bf16", "random", "random", 2, P, seed=P, symmetric=False,
                         q_pos_offset=off)
    q, k, v = gu.to_device(w)
    k[:, off + n_q:], v[:, off + n_q:] = float("nan"), float("nan")
    plan = gu.make_plan(w)
    table = cb.cascade_rope_table(n_kv, 128, 10000.0)
    size = cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.BF16, 2, 8, 2, 128)
    ws = [torch.zeros(size, dtype=torch.uint8, device="cuda") for _ in range(2)]
    o = torch.zeros_like(q)
    o_ref, _ = cb.cascade_attn_sharded_rope(plan, q, k, v, w.scale, table, workspace=ws[0])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cb.cascade_attn_sharded_rope(plan, q, k, v, w.scale, table, out=o, want_lse=False, workspace=ws[1])
    for _ in range(2):
        o.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert (o.float() - o_ref.float()).abs().max() <= w.tol and torch.isfinite(o.float()).all()
        assert torch.equal(*ws)
    del graph
    plan.destroy()
