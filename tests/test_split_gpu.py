"""fp32 heads of 64 columns on the tensor cores (operands split into three bf16 parts): edges of its tiles, what it makes of
values out of range, and its error next to that of the ALU kernels.  Two kernels per call tell that the route was taken."""
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


def _fused(cb, plan, q, k, v, scale, workspace=True):
    """The fused call with the workspace it asks for, or without any (then it runs on the ALUs); and how many kernels it ran."""
    o, lse = torch.empty_like(q), torch.empty(q.shape[:3], dtype=torch.float32, device="cuda")
    B, _, H, d = q.shape
    need = cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.F32, B, H, k.shape[2], d)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda") if workspace else None
    S, n0 = cb._strides, cb.lib().cascade_launch_count()
    assert 0 == cb.lib().cascade_attn_sharded(plan.handle, cb.F32, B, H, k.shape[2], d, scale, q.data_ptr(), S(q), k.data_ptr(), S(k),
                                              v.data_ptr(), S(v), o.data_ptr(), S(o), lse.data_ptr(), ws.data_ptr() if workspace else None,
                                              need if workspace else 0, torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return o, lse, cb.lib().cascade_launch_count() - n0


@pytest.mark.parametrize("n_q,n_kv,H,Hkv,J,P,causal,off", [
    (127, 127, 16, 16, 2, 2, False, 0),      # one sub-tile with a row missing
    (129, 193, 16, 16, 3, 1, True, 64),      # a second sub-tile of one row, one key past three tiles
    (257, 257, 16, 16, 4, 4, True, 0),       # a second query tile of one row; the first sub-tile skips tiles of the second
    (300, 300, 16, 4, 5, 3, True, 0),        # four heads a tile
    (40, 640, 16, 2, 1, 2, False, 0),        # eight heads a tile
    (333, 333, 12, 4, 2, 5, True, 0),        # three heads per KV head: no stacking
    (200, 500, 16, 16, 3, 4, True, -60),     # the first rows see nothing
    (300, 300, 16, 16, 60, 2, True, 0),      # rows of many query shards in a tile
])
def test_split_route_at_its_edges(gu, n_q, n_kv, H, Hkv, J, P, causal, off):
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload(f"split_{n_q}_{n_kv}", 8, n_q, n_kv, H, Hkv, 64, "f32", "random", "random", J, P, seed=n_q + P, causal=causal,
                         q_pos_offset=off, symmetric=J == P and n_q == n_kv)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    assert _fused(cb, plan, q, k, v, w.scale)[2] == 2
    plan.destroy()
    gu.full_parity(w)


def test_split_route_where_shards_are_empty(gu):
    """Shards without keys, and shards that a query tile sees nothing of."""
    from paper_2507_05228_b200 import binding as cb
    rng = np.random.default_rng(5)
    n, B, H, P = 400, 8, 16, 6
    w = wl.make_workload("split_empty", B, n, n, H, H, 64, "f32", "random", "random", 2, 2, seed=3)
    w.kv_shard_of = np.where(np.arange(n) < 200, rng.integers(0, 2, n), 4).astype(np.int32)
    w.n_kv_shards = P
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    assert _fused(cb, plan, q, k, v, w.scale)[2] == 2
    plan.destroy()
    gu.full_parity(w)


@pytest.mark.parametrize("n,causal", [(512, False), (1000, True)])
def test_split_route_is_as_exact_as_the_alu_kernels(gu, n, causal):
    """Outputs closer to fp64 than those of the ALU kernels.  The logarithm of the row sum is 6 to 7 in size and rounded to fp32,
    2.1e-8 of it on average, which both carry: 3e-8 in all, with room for the next digit."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload(f"split_err_{n}", 4, n, n, 12, 12, 64, "f32", "random", "random", 4, 4, seed=n, causal=causal)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, causal=causal)
    err = {}
    for ws in (True, False):
        o, lse, n_kernels = _fused(cb, plan, q, k, v, w.scale, ws)
        assert n_kernels == (2 if ws else 1)
        err[ws] = [np.linalg.norm(a.double().cpu().numpy() - r) / np.linalg.norm(r) for a, r in ((o, o_ref), (lse, lse_ref))]
    print(err)
    assert err[True][0] <= err[False][0] and err[True][1] <= 3.2e-8, err
    plan.destroy()


def test_split_route_with_values_out_of_range(gu):
    """Infinite, NaN and very large rows: rows that see none of them are untouched, the others as in fp64 (overflow aside)."""
    from paper_2507_05228_b200 import binding as cb
    B, n, H = 8, 300, 16
    w = wl.make_workload("split_big", B, n, n, H, H, 64, "f32", "random", "random", 3, 3, seed=9)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    q[:, :, 1].abs_()
    k[:, 70, 1] = -(2.0 ** 126)          # logits below every other one: no weight
    k[:, 130, 2, 5] = 2.0 ** 80          # logits of either sign and 2^80
    v[:, 200, 3, 7] = float("inf")
    v[:, 210, 4, 9] = float("nan")
    v[:, 220, 5] = 3.4e38
    q[:, 33, 6, 2] = 2.0 ** 70
    o, lse, n_kernels = _fused(cb, plan, q, k, v, w.scale)
    assert n_kernels == 2 and plan.device_status() == 0
    s = torch.einsum("bqhd,bkhd->bhqk", q.double(), k.double()) * float(np.float32(w.scale))
    s = s.masked_fill(~torch.ones(n, n, dtype=torch.bool, device="cuda").tril(), -torch.inf)
    a = torch.softmax(s, -1)
    o_ref = torch.einsum("bhqk,bkhd->bqhd", a, v.double().nan_to_num(nan=0.0, posinf=0.0))
    assert torch.isinf(o[:, 200:, 3, 7]).all() and torch.isnan(o[:, 210:, 4, 9]).all()
    o[:, 200:, 3, 7] = 0
    o[:, 210:, 4, 9] = 0
    o_ref[:, 200:, 3, 7] = 0
    o_ref[:, 210:, 4, 9] = 0
    assert ((o.double() - o_ref).abs() <= w.tol * o_ref.abs().clamp_min(1.0)).all()
    assert torch.allclose(lse.double(), torch.logsumexp(s, -1).transpose(1, 2), rtol=1e-5, atol=w.tol)
    plan.destroy()


@pytest.mark.parametrize("far", ["key", "value"])
def test_values_out_of_range_touch_their_own_tiles_only(gu, far):
    """Partials of the shards without such a row, and fused rows before the tile that holds it, keep their bits."""
    from paper_2507_05228_b200 import binding as cb
    B, n, H, P = 8, 400, 16, 4
    w = wl.make_workload("split_far", B, n, n, H, H, 64, "f32", "random", "random", 2, P, seed=21, symmetric=False)
    w.kv_shard_of = (np.arange(n) // 8 % P).astype(np.int32)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    ws = torch.empty(cb.cascade_workspace_bytes(plan, cb.CALL_PARTIALS, cb.F32, B, H, H, 64), dtype=torch.uint8, device="cuda")
    n0 = cb.lib().cascade_launch_count()
    clean = [t.clone() for t in cb.cascade_attn_partials(plan, q, k, v, w.scale, workspace=ws)]
    assert cb.lib().cascade_launch_count() - n0 == 2
    o = _fused(cb, plan, q, k, v, w.scale)[0]
    if far == "key":  # in the tile of tokens 192 to 255 both; no other shard has rows in the same block of 64 slots
        k[:, 192, :, 3] = 2.0 ** 70
    else:
        v[:, 200, :, 3] = 2.0 ** 70
    k0 = 0 if far == "key" else 1
    parts = [t.clone() for t in cb.cascade_attn_partials(plan, q, k, v, w.scale, workspace=ws)]
    o_far = _fused(cb, plan, q, k, v, w.scale)[0]
    assert not torch.equal(parts[0][:, k0], clean[0][:, k0])
    for a, b in zip(parts, clean):
        for kk in set(range(P)) - {k0}:
            assert torch.equal(a[:, kk], b[:, kk]), kk
    assert torch.equal(o_far[:, :192], o[:, :192]) and not torch.equal(o_far[:, 192:], o[:, 192:])
    plan.destroy()


@pytest.mark.parametrize("what,size", [("q", -118), ("k", -118), ("v", -118), ("v", -101), ("k", -112), ("one column of v", -120)])
def test_small_values_keep_their_bits(gu, what, size):
    """Below 2^-110 three bf16 parts do not hold an fp32 number.  Rows of queries and keys and columns of values that small go another
    way, in plain fp32.  Bound: a sum of n terms in a chain is off by 2^-24 / sqrt(3) * sqrt(n / 2) of itself in the mean, half an ulp of
    rounding at each of its parts: 1.9e-7 for the 64 products of a tile, 1e-7 for logits near 1 in chains of 16, in the weights and in
    the row sums; 2.4e-7 together, and the worst of 64 columns a tenth more."""
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("split_small", 8, 300, 300, 16, 16, 64, "f32", "random", "random", 3, 3, seed=17)
    q, k, v = gu.to_device(w)
    scale = w.scale
    if what == "one column of v":
        v[..., 5] *= 2.0 ** size
    else:
        {"q": q, "k": k, "v": v}[what].mul_(2.0 ** size)
        if what != "v":
            scale = w.scale * 2.0 ** -size
    s = torch.einsum("bqhd,bkhd->bhqk", q.double(), k.double()) * float(np.float32(scale))
    s = s.masked_fill(~torch.ones(300, 300, dtype=torch.bool, device="cuda").tril(), -torch.inf)
    ref = torch.einsum("bhqk,bkhd->bqhd", torch.softmax(s, -1), v.double())
    plan = gu.make_plan(w)
    err = {}
    for ws in (True, False):
        o, _, n_kernels = _fused(cb, plan, q, k, v, scale, ws)
        assert n_kernels == (2 if ws else 1)
        off = (o.double() - ref).square().sum((0, 1, 2)).sqrt() / ref.square().sum((0, 1, 2)).sqrt()  # of every column
        err[ws] = off.max().item()
    assert err[True] <= 2.7e-7 and err[False] <= 2.7e-7, err
    plan.destroy()


def test_captured_split_calls_follow_the_plan(gu):
    from paper_2507_05228_b200 import binding as cb
    B, n_q, n_kv, H, P = 8, 128, 700, 16, 3
    w = wl.make_workload("split_graph", B, n_kv, n_kv, H, H, 64, "f32", "random", "random", 1, 1, seed=4)
    q, k, v = gu.to_device(w)
    rng = np.random.default_rng(P)
    kv_of, q_of = rng.integers(0, P, n_kv).astype(np.int32), rng.integers(0, 2, n_q).astype(np.int32)
    plan = cb.cascade_shard_plan(q_of, kv_of, 2, P, 100, True)
    qc, kc, vc = q[:, :n_q].clone(), k.clone(), v.clone()
    ws = torch.empty(cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.F32, B, H, H, 64), dtype=torch.uint8, device="cuda")
    o = torch.zeros_like(qc)
    parts = [t.clone() for t in cb.cascade_attn_partials(plan, qc, k, v, w.scale, workspace=ws)]
    n0 = cb.lib().cascade_launch_count()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cb.cascade_attn_sharded(plan, qc, kc, vc, w.scale, out=o, want_lse=False, workspace=ws)
        cb.cascade_attn_partials(plan, qc, kc, vc, w.scale, out=parts, workspace=ws)
    assert cb.lib().cascade_launch_count() - n0 == 4
    for off in (100, 572, 20):
        seen = off + n_q
        qc.copy_(q[:, off:seen])
        kc.fill_(float("nan")), vc.fill_(float("nan"))
        kc[:, :seen], vc[:, :seen] = k[:, :seen], v[:, :seen]
        plan.advance(off)
        graph.replay()
        torch.cuda.synchronize()
        o_ref, _ = oracle.attention_unsharded(w.q[:, off:seen], w.k, w.v, w.scale, q_pos_offset=off)
        gu.check_output(o, None, o_ref, None, w.tol, f"replayed at {off}")
        op = oracle.shard_plan(q_of, kv_of, 2, P, q_pos_offset=off, causal=True)
        u, m, e = oracle.attn_pass(w.q[:, off:seen], w.k, w.v, w.scale, op)
        gu.check_partials(tuple(t.double().cpu().numpy() for t in parts), (u, m, e), w.tol, f"partials at {off}")
    del graph
    plan.destroy()


def test_split_calls_on_a_plan_whose_status_word_is_set_write_nothing(gu):
    from paper_2507_05228_b200 import binding as cb
    w = wl.make_workload("split_gave_up", 8, 300, 300, 16, 16, 64, "f32", "random", "random", 2, 3, seed=2, symmetric=False)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    word = torch.as_tensor(gu._DevicePointer(plan.dev_ptr("q_off") - 256, 1, "<i4"), device="cuda")
    o_ref, _ = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    word.fill_(5)
    o = torch.full_like(q, 7.0)
    parts = cb.cascade_attn_partials(plan, q, k, v, w.scale)
    for t in parts:
        t.fill_(7.0)
    cb.cascade_attn_sharded(plan, q, k, v, w.scale, out=o, want_lse=False)
    cb.cascade_attn_partials(plan, q, k, v, w.scale, out=parts)
    torch.cuda.synchronize()
    assert (o == 7).all() and all((t == 7).all() for t in parts)
    word.fill_(0)
    cb.cascade_attn_sharded(plan, q, k, v, w.scale, out=o, want_lse=False)
    assert torch.equal(o, o_ref) and plan.device_status() == 0
    plan.destroy()


def _partials(cb, plan, q, k, v, scale):
    """The partials with the workspace that they ask for; and how many kernels ran."""
    n0 = cb.lib().cascade_launch_count()
    parts = cb.cascade_attn_partials(plan, q, k, v, scale)
    torch.cuda.synchronize()
    return parts, cb.lib().cascade_launch_count() - n0


@pytest.mark.parametrize("n_kv", [16, 64, 512])
@pytest.mark.parametrize("signs", ["values", "queries and keys", "all"])
def test_split_route_on_values_of_one_sign(gu, n_kv, signs):
    """The tensor core cuts its sums off, which adds up where all products have one sign and one tile holds the keys.  Outputs, maxima
    and sums are closer to fp64 than those of the ALU kernels all the same.  The logarithm of the row sum is 5 to 9 in size and
    rounded to fp32, 2^-24 of it at most; the cut-off logits add as much at most."""
    from paper_2507_05228_b200 import binding as cb
    B, n_q, H, P = 16, 128, 16, 2
    w = wl.make_workload(f"split_sign_{n_kv}", B, n_q, n_kv, H, H, 64, "f32", "random", "random", 2, P, seed=n_kv, causal=False, symmetric=False)
    if signs != "values":
        w.q, w.k = np.abs(w.q), np.abs(w.k)
    if signs != "queries and keys":
        w.v = np.abs(w.v)
    q, k, v = gu.to_device(w)
    plan = gu.make_plan(w)
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale, causal=False)
    refs = (o_ref, lse_ref) + oracle.attn_pass(w.q, w.k, w.v, w.scale, gu.oracle_plan(w))
    err = {}
    for ws in (True, False):
        o, lse, n_kernels = _fused(cb, plan, q, k, v, w.scale, ws)
        assert n_kernels == (2 if ws else 1)
        n0 = cb.lib().cascade_launch_count()
        parts = cb.cascade_attn_partials(plan, q, k, v, w.scale, workspace=None if ws else torch.empty(16, dtype=torch.uint8, device="cuda"))
        torch.cuda.synchronize()
        assert cb.lib().cascade_launch_count() - n0 == (2 if ws else 1)
        err[ws] = [np.linalg.norm(a.double().cpu().numpy() - r) / np.linalg.norm(r) for a, r in zip((o, lse) + tuple(parts), refs)]
    print(err)
    assert all(a <= b for i, (a, b) in enumerate(zip(err[True], err[False])) if i != 1) and err[True][1] <= 2.0 ** -23, err
    plan.destroy()


def test_split_route_with_a_map_per_sequence(gu):
    from paper_2507_05228_b200 import binding as cb
    B, n, H, P = 8, 260, 16, 3
    w = wl.make_workload("split_maps", B, n, n, H, H, 64, "f32", "random", "random", 1, 1, seed=41)
    rng = np.random.default_rng(42)
    q_of, kv_of = rng.integers(0, 2, (B, n)).astype(np.int32), rng.integers(0, P, (B, n)).astype(np.int32)
    q, k, v = gu.to_device(w)
    plan = cb.cascade_shard_plan(q_of, kv_of, 2, P)
    o, lse, n_kernels = _fused(cb, plan, q, k, v, w.scale)
    parts, n_parts = _partials(cb, plan, q, k, v, w.scale)
    assert n_kernels == 2 and n_parts == 2 and plan.device_status() == 0
    o_ref, lse_ref = oracle.attention_unsharded(w.q, w.k, w.v, w.scale)
    gu.check_output(o, lse, o_ref, lse_ref, w.tol, "a map per sequence")
    for b in range(B):
        ref = oracle.attn_pass(w.q[b:b + 1], w.k[b:b + 1], w.v[b:b + 1], w.scale, oracle.shard_plan(q_of[b], kv_of[b], 2, P))
        gu.check_partials(tuple(t[b:b + 1].double().cpu().numpy() for t in parts), ref, w.tol, f"a map per sequence, b={b}")
    plan.destroy()


def test_split_route_over_resident_rows(gu):
    """Rows with positions of their own, a set of them per sequence; those that no query sees hold NaN."""
    from paper_2507_05228_b200 import binding as cb
    B, n, n_q, n_kv, H, off = 8, 600, 130, 300, 16, 300
    rng = np.random.default_rng(43)
    w = wl.make_workload("split_resident", B, n, n, H, H, 64, "f32", "random", "random", 1, 1, seed=44)
    q, k, v = gu.to_device(w)
    pos = np.sort(np.stack([rng.choice(n, n_kv, replace=False) for _ in range(B)]), axis=1).astype(np.int32)
    q_of, kv_of = rng.integers(0, 2, (B, n_q)).astype(np.int32), rng.integers(0, 4, (B, n_kv)).astype(np.int32)
    plan = cb.cascade_shard_plan_resident(q_of, kv_of, pos, 2, 4, off)
    at = torch.from_numpy(pos.astype(np.int64)).cuda()
    kr, vr = (torch.stack([t[b, at[b]] for b in range(B)]) for t in (k, v))
    for b in range(B):
        kr[b, at[b] > off + n_q - 1] = float("nan")
        vr[b, at[b] > off + n_q - 1] = float("nan")
    qr = q[:, off:off + n_q]
    o, lse, n_kernels = _fused(cb, plan, qr, kr, vr, w.scale)
    parts, n_parts = _partials(cb, plan, qr, kr, vr, w.scale)
    assert n_kernels == 2 and n_parts == 2 and plan.device_status() == 0
    seen = at[:, None, :] <= torch.arange(off, off + n_q, device="cuda")[None, :, None]
    s = torch.einsum("bqhd,bkhd->bhqk", qr.double(), kr.double().nan_to_num(0.0)) * float(np.float32(w.scale))
    s = s.masked_fill(~seen[:, None], -torch.inf)
    o_ref = torch.einsum("bhqk,bkhd->bqhd", torch.softmax(s, -1), vr.double().nan_to_num(0.0)).cpu().numpy()
    lse_ref = torch.logsumexp(s, -1).transpose(1, 2).cpu().numpy()
    gu.check_output(o, lse, o_ref, lse_ref, w.tol, "resident rows")
    merged, _ = cb.cascade_merge(*parts, plan.dev_ptr("q_idx"), n_q)
    gu.check_output(merged, None, o_ref, None, w.tol, "resident rows, merged")
    plan.destroy()


@pytest.mark.parametrize("form", ["columns of one tensor", "keys and values of one sequence for all"])
def test_split_route_on_strided_and_expanded_rows(gu, form):
    from paper_2507_05228_b200 import binding as cb
    B, n, H, Hkv = 8, 200, 16, 8
    w = wl.make_workload("split_strides", B, n, n, H, Hkv, 64, "f32", "random", "random", 3, 3, seed=45)
    if form == "columns of one tensor":
        rows = torch.full((B, n, H + 2 * Hkv + 1, 64), float("nan"), device="cuda")
        q, k, v = rows[:, :, :H], rows[:, :, H:H + Hkv], rows[:, :, H + Hkv:H + 2 * Hkv]
        for t, src in zip((q, k, v), gu.to_device(w)):
            t.copy_(src)
    else:
        w.k, w.v = (np.broadcast_to(a[:1], a.shape).copy() for a in (w.k, w.v))
        q, k, v = gu.to_device(w)
        k, v = k[:1].expand(B, -1, -1, -1), v[:1].expand(B, -1, -1, -1)
    plan = gu.make_plan(w)
    need = cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED, cb.F32, B, H, Hkv, 64)
    n0 = cb.lib().cascade_launch_count()
    o, lse = cb.cascade_attn_sharded(plan, q, k, v, w.scale)
    assert need > 0 and cb.lib().cascade_launch_count() - n0 == 2
    parts, n_parts = _partials(cb, plan, q, k, v, w.scale)
    assert n_parts == 2
    gu.check_output(o, lse, *oracle.attention_unsharded(w.q, w.k, w.v, w.scale), w.tol, form)
    gu.check_partials(tuple(t.double().cpu().numpy() for t in parts), oracle.attn_pass(w.q, w.k, w.v, w.scale, gu.oracle_plan(w)), w.tol, form)
    plan.destroy()


def test_split_route_from_host_buffers(gu):
    """The head groups of the host call, two kernels each, against the oracle."""
    from paper_2507_05228_b200 import binding as cb
    B, n, H = 8, 300, 16
    w = wl.make_workload("split_host", B, n, n, H, H, 64, "f32", "random", "random", 3, 3, seed=46)
    plan = gu.make_plan(w)
    hq, hk, hv = (torch.from_numpy(a).pin_memory() for a in (w.q, w.k, w.v))
    ho = torch.empty_like(hq).pin_memory()
    ws = torch.empty(cb.cascade_workspace_bytes(plan, cb.CALL_SHARDED_HOST, cb.F32, B, H, H, 64), dtype=torch.uint8, device="cuda")
    n0 = cb.lib().cascade_launch_count()
    cb.cascade_attn_sharded_host(plan, hq, hk, hv, w.scale, ho, ws)
    torch.cuda.synchronize()
    assert cb.lib().cascade_launch_count() - n0 == 2 * H // 4  # four heads at a time
    gu.check_output(ho.double().numpy(), None, oracle.attention_unsharded(w.q, w.k, w.v, w.scale)[0], None, w.tol, "host buffers")
    plan.destroy()
