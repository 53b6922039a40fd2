// Decode step with a token-sharded KV cache (Appendix F, "Caching"): one new query row per sequence against
// every KV shard.  Each shard is an independent partial (the Attention-Pass algorithm with a single query row) and the K/V rows
// of the cache are read exactly once, so the kernels must be bound by HBM reads of gathered 256-byte rows.
//
// decode_kernel (partials): one CTA = (KV shard, KV head, sequence); decode_fused_kernel: all shards, post-pass included.
// In both, a warp walks blocks of 16 gathered keys with warp-level mma.m16n8k16 products, which keeps the instruction count
// per loaded byte low enough for the memory system to be the limit (plain FMA code was issue-bound at ~60 % of the HBM
// rate).  Keys are the M rows of the logits and head_dim the M rows of the output, so that the G query heads that share the
// KV head ("repeat_kv") are the 8 columns and no row is padding: 16 products and 32 accumulators per block (with the heads as
// M rows it was 32 products, and 8 registers for rows that do not exist).  No staging of K or V is needed because the
// contraction order is free: the k index of an MMA may be any fixed permutation of head_dim / of the keys as long as both
// operands use the same one, so every thread loads 16-byte pieces straight from global memory into fragments
// (x = lane / 4, j = lane % 4):
//   logits  S^T[key, head] : A = K, rows x and x + 8 of the block; B = Q^T; pieces d = 64c + 16j .. + 15 (c < 2)
//   output  O^T[d, head]   : A = V^T, pieces d = 16x .. + 15 of V rows 2j, 2j+1, 2j+8, 2j+9, paired with PRMT;
//                            B = P^T, the bf16 weights of S^T transposed with movmatrix
// so that the loads of a row cover whole 128-byte lines.  (One 32-byte load per piece was 2 to 4 % slower than two of 16
// bytes at every size.)
// 64 registers hold the loads in flight.  Anything else kept through the loop ends up spilled, and a spilled value comes back
// from L2, because the streaming loads evict it from L1: the query fragments therefore live in shared memory.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "cascade_internal.cuh"

namespace cascade {

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 8 x 8 transpose of 16-bit elements across a warp (lane (x, j) holds row x, columns 2j and 2j + 1)
__device__ __forceinline__ uint32_t transpose8(uint32_t v) {
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(v));
  return r;
}

__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 32 bytes, streaming; volatile so that the loads stay where the pipeline below puts them
__device__ __forceinline__ void load32(const __nv_bfloat16* p, uint32_t* r) {
#pragma unroll
  for (int i = 0; i < 8; i += 4)
    asm volatile("ld.global.cs.v4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[i]), "=r"(r[i + 1]), "=r"(r[i + 2]), "=r"(r[i + 3])
                 : "l"(p + 2 * i)
                 : "memory");
}

// Query fragments of a CTA in shared memory: B operand of k-step s, lane (x = head, j) -> its two registers.
struct DecodeQuery {
  uint2 frag[8][32];
};
// Filled by one warp from the thread's pieces qf[8 c + e] = columns 64c + 16j + 2e, + 1 of head x (zero from G on).
__device__ __forceinline__ void publish_query(DecodeQuery& q, const uint32_t (&qf)[16], int lane) {
#pragma unroll
  for (int s = 0; s < 8; ++s) q.frag[s][lane] = make_uint2(qf[2 * s], qf[2 * s + 1]);
}
// The pieces of one head vector.
__device__ __forceinline__ void load_query(const __nv_bfloat16* row, int j, uint32_t (&qf)[16]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(row + 64 * (c >> 1) + 16 * j + 8 * (c & 1)));
    qf[4 * c] = t.x; qf[4 * c + 1] = t.y; qf[4 * c + 2] = t.z; qf[4 * c + 3] = t.w;
  }
}

struct DecodeState {
  float o[8][4];     // o[e][2 r + h]: head 2j + h, column 16x + 2e + r
  float m[2], l[2];  // heads 2j, 2j + 1 (log2 units); l is this thread's share (its key rows x, x + 8)
};
__device__ __forceinline__ void decode_init(DecodeState& st) {
#pragma unroll
  for (int e = 0; e < 8; ++e)
#pragma unroll
    for (int i = 0; i < 4; ++i) st.o[e][i] = 0.f;
  st.m[0] = st.m[1] = -INFINITY;
  st.l[0] = st.l[1] = 0.f;
}

// Walks `count` blocks of 16 keys; block t is the keys kv_idx[at .. at + n - 1] (n >= 1; 16 at most are taken) with
// (at, n) = get(t).
// kAhead: the key rows of block t + kAhead are requested as soon as the logits of block t are formed, its value rows after the
// product of block t, its tokens a block earlier still, all into registers that have just come free: with 1, one memory latency
// per block instead of two and the arithmetic (a block took 3200 cycles one after another).  With 0 nothing is spilled,
// which is the better trade where 16 warps per SM cover the latencies anyway (partials of 64 sequences of 16384 tokens: 630
// us without, 820 with; all shards in one kernel: 711 without, 620 with).  With 2 a warp keeps twice the loads in flight, in
// registers that it has where an SM holds eight warps and no more.  The sums are the same whatever kAhead is.
// gate() is called before the first rows are requested, ready() before the query is used; by a warp without blocks, too.
template <int kAhead, typename Get, typename Gate, typename Ready>
__device__ __forceinline__ void decode_walk(DecodeState& st, const DecodeQuery& q, const PlanDev& pl, const int32_t* kv_idx,
                                            int count, Get get, const __nv_bfloat16* kp, int64_t k_token,
                                            const __nv_bfloat16* vp, int64_t v_token, int lane, float cs, Gate gate, Ready ready) {
  if (count <= 0) {
    gate();
    ready();
    return;
  }
  constexpr int kBuffers = kAhead > 1 ? kAhead : 1;  // of block t: t % kBuffers
  const int x = lane >> 2, j = lane & 3;
  uint32_t ka[kBuffers][16], kb[kBuffers][16], vr[kBuffers][4][8];
  auto token = [&](int2 e) {  // lane l: token of key l (clamped to the last key; masked below)
    return (int)CASCADE_CHECKED((int64_t)__ldg(kv_idx + e.x + min(lane & 15, e.y - 1)), pl.n_kv, pl.status, 106);
  };
  auto load_k = [&](int buf, int tok) {  // rows x and x + 8
    const __nv_bfloat16* r0 = kp + (int64_t)__shfl_sync(0xffffffffu, tok, x) * k_token;
    const __nv_bfloat16* r1 = kp + (int64_t)__shfl_sync(0xffffffffu, tok, x + 8) * k_token;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      load32(r0 + 64 * c, ka[buf] + 8 * c);
      load32(r1 + 64 * c, kb[buf] + 8 * c);
    }
  };
  auto load_v = [&](int buf, int tok) {  // rows 2j, 2j + 1, 2j + 8, 2j + 9
#pragma unroll
    for (int rr = 0; rr < 4; ++rr)
      load32(vp + (int64_t)__shfl_sync(0xffffffffu, tok, 2 * j + (rr & 1) + (rr >> 1) * 8) * v_token, vr[buf][rr]);
  };
  int2 e;
  int tok;
  if constexpr (kAhead > 0) {
    e = get(0);
    tok = token(e);
    const int tok1 = kAhead > 1 && count > 1 ? token(get(1)) : 0;
    gate();
    load_k(0, tok);
    load_v(0, tok);
    if (kAhead > 1 && count > 1) {
      load_k(kBuffers - 1, tok1);
      load_v(kBuffers - 1, tok1);
    }
    if (count > kAhead) tok = token(get(kAhead));
    ready();
  }
  auto block = [&](int t, int buf) {
    if constexpr (kAhead == 0) {
      e = get(t);
      tok = token(e);
      load_k(buf, tok);
      load_v(buf, tok);
    }
    const int n_keys = kAhead > 1 ? get(t).y : e.y;
    const bool more = kAhead > 0 && t + kAhead < count;
    float sc[4] = {0.f, 0.f, 0.f, 0.f};  // (key x, head 2j), (x, 2j + 1), (x + 8, 2j), (x + 8, 2j + 1)
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint2 b = q.frag[i][lane];
      mma_16816(sc, ka[buf][2 * i], kb[buf][2 * i], ka[buf][2 * i + 1], kb[buf][2 * i + 1], b.x, b.y);
    }
    if (more) {
      if (kAhead == 1) e = get(t + 1);
      load_k(buf, tok);
    }
    float alpha[2], p0[2], p1[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float t0 = x < n_keys ? sc[h] * cs : -INFINITY, t1 = x + 8 < n_keys ? sc[2 + h] * cs : -INFINITY;
      float mx = fmaxf(t0, t1);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float m_new = fmaxf(st.m[h], mx);  // finite: key 0 of the block exists
      alpha[h] = ex2f(st.m[h] - m_new);        // ex2(-inf) = 0 on the first block
      p0[h] = ex2f(t0 - m_new);
      p1[h] = ex2f(t1 - m_new);
      st.l[h] = st.l[h] * alpha[h] + (p0[h] + p1[h]);
      st.m[h] = m_new;
    }
    const uint32_t pa = transpose8(pack2_bf16(p0[0], p0[1]));  // -> head x, keys 2j, 2j + 1
    const uint32_t pb = transpose8(pack2_bf16(p1[0], p1[1]));  // -> head x, keys 2j + 8, 2j + 9
    if (__any_sync(0xffffffffu, alpha[0] != 1.f || alpha[1] != 1.f)) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) st.o[i][c] *= alpha[c & 1];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      mma_16816(st.o[i], __byte_perm(vr[buf][0][i], vr[buf][1][i], 0x5410), __byte_perm(vr[buf][0][i], vr[buf][1][i], 0x7632),
                __byte_perm(vr[buf][2][i], vr[buf][3][i], 0x5410), __byte_perm(vr[buf][2][i], vr[buf][3][i], 0x7632), pa, pb);
    if (more) {
      load_v(buf, tok);
      if (t + kAhead + 1 < count) tok = token(get(t + kAhead + 1));
    }
  };
#pragma unroll 1
  for (int t = 0; t < count; t += kBuffers) {
    block(t, 0);
    if constexpr (kBuffers == 2)
      if (t + 1 < count) block(t + 1, 1);
  }
}

// Combines the warps of a CTA (each saw disjoint keys) through shared memory.
template <int G, int NW>
struct DecodeShared {
  float m[NW][G], l[NW][G];
  float o[NW][G][132];
};
template <int G, int NW>
__device__ __forceinline__ void decode_publish(DecodeShared<G, NW>& sh, DecodeState& st, int warp, int lane) {
  const int x = lane >> 2, j = lane & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float l = st.l[h];  // this thread's share of the sum of exponentials -> whole row
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    const int head = 2 * j + h;
    if (head < G) {
      if (x == 0) {
        sh.m[warp][head] = st.m[h];
        sh.l[warp][head] = l;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
        *reinterpret_cast<float2*>(&sh.o[warp][head][16 * x + 2 * e]) = make_float2(st.o[e][h], st.o[e][2 + h]);
    }
  }
}
// Output column `col` of head gg: the maximum n, the weight w and the weighted sum, relative to n.
template <int G, int NW>
__device__ __forceinline__ void decode_combine(const DecodeShared<G, NW>& sh, int gg, int col, float& n, float& w, float& acc) {
  n = -INFINITY;
#pragma unroll
  for (int w2 = 0; w2 < NW; ++w2) n = fmaxf(n, sh.m[w2][gg]);
  const float n_use = n == -INFINITY ? 0.f : n;
  w = 0.f;
  acc = 0.f;
#pragma unroll
  for (int w2 = 0; w2 < NW; ++w2) {
    const float f = ex2f(sh.m[w2][gg] - n_use);  // 0 for a warp that saw no key
    w = fmaf(f, sh.l[w2][gg], w);
    acc = fmaf(f, sh.o[w2][gg][col], acc);
  }
}

// Partials.  Four CTAs per SM at 128 registers per thread (no spills).
template <int G>
__global__ void __launch_bounds__(128, 4) decode_kernel(const __grid_constant__ AttnParams p) {
  constexpr int D = 128;
  constexpr int NW = 4;  // warps per CTA
  __shared__ DecodeShared<G, NW> sh;
  __shared__ DecodeQuery s_q;

  const PlanDev& pl = p.plan;
  const int P = pl.n_kv_shards;
  const int kk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
  const int map = pl.n_maps == 1 ? 0 : b;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x = lane >> 2, j = lane & 3;
  const int32_t* kv_idx = pl.kv_idx + (size_t)map * pl.n_kv + pl.kv_off[(size_t)map * (P + 1) + kk];
  const int n_vis = pl.vis[(size_t)map * pl.n_q * P + kk];  // the single query slot
  const int64_t stat0 = (((int64_t)b * P + kk) * pl.n_q) * p.H + (int64_t)g * G;
  __nv_bfloat16* o_part = static_cast<__nv_bfloat16*>(p.o_part);
  if (n_vis == 0) {  // nothing of this shard is visible: m = -inf, l = 0, u = 0
    for (int gg = 0; gg < G; ++gg) {
      o_part[(stat0 + gg) * D + tid] = __float2bfloat16_rn(0.f);
      if (tid == 0) {
        p.m_part[stat0 + gg] = -INFINITY;
        p.l_part[stat0 + gg] = 0.f;
      }
    }
    return;
  }
  const int tok_q = (int)CASCADE_CHECKED((int64_t)pl.q_idx[(size_t)map * pl.n_q], pl.n_q, pl.status, 107);
  const __nv_bfloat16* kb = static_cast<const __nv_bfloat16*>(p.k) + (int64_t)b * p.ks.batch +
                            (int64_t)g * p.ks.head + 16 * j;
  const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(p.v) + (int64_t)b * p.vs.batch +
                            (int64_t)g * p.vs.head + 16 * x;
  if (warp == 0) {
    uint32_t qf[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) qf[c] = 0u;
    if (x < G)
      load_query(static_cast<const __nv_bfloat16*>(p.q) + (int64_t)b * p.qs.batch + (int64_t)tok_q * p.qs.token +
                     (int64_t)(g * G + x) * p.qs.head, j, qf);
    publish_query(s_q, qf, lane);
  }
  __syncthreads();
  const float cs = p.scale * 1.4426950408889634f;  // logits in log2 units

  DecodeState st;
  decode_init(st);
  decode_walk<0>(st, s_q, pl, kv_idx, (n_vis - warp * 16 + NW * 16 - 1) / (NW * 16),
                     [&](int t) { const int k0 = (t * NW + warp) * 16; return make_int2(k0, n_vis - k0); }, kb, p.ks.token,
                     vb, p.vs.token, lane, cs, []() {}, []() {});
  decode_publish<G, NW>(sh, st, warp, lane);
  __syncthreads();
  // thread = output column
#pragma unroll
  for (int gg = 0; gg < G; ++gg) {
    float n, w, acc;
    decode_combine<G, NW>(sh, gg, tid, n, w, acc);
    o_part[(stat0 + gg) * D + tid] = __float2bfloat16_rn(acc / w);
    if (tid == 0) {
      p.m_part[stat0 + gg] = n * 0.6931471805599453f;  // back to natural-log units
      p.l_part[stat0 + gg] = w;
    }
  }
}

// ---------------------------------------------------------------------------------------------------------------------
// Decode with the post-pass in the same kernel (the fused route): a cluster of CTAs owns one (KV head, sequence), its warps
// share the 16-key blocks of all shards' visible prefixes, and the partial (m, l, o) meet in distributed shared memory, so
// no partial goes to memory and nothing is launched after it.  Bound by HBM reads for large batches and by latency for small
// ones; the number of CTAs per (KV head, sequence) follows from both, see launch_decode_fused.
// With `step` the kernel is the whole decode step of a cache with rotary positions (the tail of the Pre-Pass algorithm,
// then "Caching"): query rows are turned while they are loaded, and the new token's key row is turned and written, with its
// value row, to the caches before anyone reads them.
// Measured (32 query / 8 KV heads): 64 sequences of 16384 tokens in 16 shards 662 us on inputs new to the caches = 6.49 TB/s
// (repeated on the same ones, of which L2 keeps a part, 608; partials and merge as two kernels 825), one sequence 25 us (23
// repeated); the whole step of one sequence at 2500 of 4096 rows 7.6 us (7.1 repeated; with the table behind a barrier and one block
// ahead 10.4 and 9.6).

__device__ __forceinline__ uint32_t rotate_pair2(uint32_t x, uint32_t partner, const float4& cs, float sign) {
  // two neighbouring columns of one half: y = x cos + sign * partner * sin  (sign -1: lower half, +1: upper half)
  const float x0 = __uint_as_float(x << 16), x1 = __uint_as_float(x & 0xffff0000u);
  const float h0 = __uint_as_float(partner << 16), h1 = __uint_as_float(partner & 0xffff0000u);
  return pack2_bf16(x0 * cs.x + sign * (h0 * cs.y), x1 * cs.z + sign * (h1 * cs.w));
}

constexpr int kMaxCluster = 16;
constexpr int kFusedShards = 256;  // KV shards whose table fits in the kernel's shared memory at a time

// kAhead: blocks that a warp requests ahead, see decode_walk; with 2 a CTA has an SM to itself.
template <int G, int kAhead, bool kOneList>
__global__ void __launch_bounds__(256, 3 - kAhead) decode_fused_kernel(const __grid_constant__ AttnParams p,
                                                                      const __grid_constant__ DecodeStep step) {
  constexpr int D = 128, NW = 8;
  __shared__ DecodeShared<G, NW> sh;
  __shared__ DecodeQuery s_q;
  // what the CTAs of the cluster send for this CTA's part of the outputs: [sender][output], and n, w of every head
  __shared__ float s_o[G * D + kMaxCluster], s_n[kMaxCluster][G], s_w[kMaxCluster][G];

  const PlanDev& pl = p.plan;
  const int P = pl.n_kv_shards;
  const int n_cta = gridDim.x, rank = blockIdx.x;  // the cluster spans the x dimension
  const int g = blockIdx.y, b = blockIdx.z;
  const int map = pl.n_maps == 1 ? 0 : b;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int x = lane >> 2, j = lane & 3;
  const int32_t* kv_idx = pl.kv_idx + (size_t)map * pl.n_kv;
  const int32_t* kv_off = pl.kv_off + (size_t)map * (P + 1);
  const int32_t* vis = pl.vis + (size_t)map * P;  // one query row
  grid_go();
  grid_wait();
  const bool vis_given = step.n_vis > 0;          // the prefixes come with the launch (the plan's copy is written below)

  // step: the new token's rows go to the caches first, by warp 0 of the cluster's first CTA (two rotation pairs and four
  // value columns per lane); the cluster barrier below orders them before everyone's reads
  if (step.rope && rank == 0 && warp == 0) {
    const __nv_bfloat16* kn = step.k_new + (int64_t)b * step.kns.batch + (int64_t)g * step.kns.head + 2 * lane;
    const uint32_t lo = *reinterpret_cast<const uint32_t*>(kn), hi = *reinterpret_cast<const uint32_t*>(kn + 64);
    const float4 c2 = __ldg(reinterpret_cast<const float4*>(step.rope + (int64_t)step.position * (D / 2)) + lane);
    const __nv_bfloat16* vn = step.v_new + (int64_t)b * step.vns.batch + (int64_t)g * step.vns.head + 4 * lane;
    const uint2 vx = *reinterpret_cast<const uint2*>(vn);
    __nv_bfloat16* kd = static_cast<__nv_bfloat16*>(const_cast<void*>(p.k)) + (int64_t)b * p.ks.batch +
                        (int64_t)step.position * p.ks.token + (int64_t)g * p.ks.head + 2 * lane;
    *reinterpret_cast<uint32_t*>(kd) = rotate_pair2(lo, hi, c2, -1.f);
    *reinterpret_cast<uint32_t*>(kd + 64) = rotate_pair2(hi, lo, c2, 1.f);
    __nv_bfloat16* vd = static_cast<__nv_bfloat16*>(const_cast<void*>(p.v)) + (int64_t)b * p.vs.batch +
                        (int64_t)step.position * p.vs.token + (int64_t)g * p.vs.head + 4 * lane;
    *reinterpret_cast<uint2*>(vd) = vx;
  }
  // first barrier of the cluster: everyone has started (its shared memory may be written), the new token is in the caches
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");

  // Shards (of a window of kFusedShards) in shared memory: visible keys, first position in kv_idx, 16-key blocks before.
  __shared__ int s_vis[kFusedShards], s_off[kFusedShards], s_before[kFusedShards + 1], s_most;
  auto fill_table = [&](int w0) {
    int most = 0, before = 0;
    const int n_w = min(kFusedShards, P - w0);
    for (int k0 = 0; k0 < n_w; k0 += 32) {
      const int kk = k0 + lane;
      const int v = kk < n_w ? (vis_given ? step.vis[map * P + w0 + kk] : __ldg(vis + w0 + kk)) : 0;
      const int nb = (v + 15) >> 4;
      int incl = nb;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      if (kk < n_w) {
        s_vis[kk] = v;
        s_off[kk] = __ldg(kv_off + w0 + kk);
        s_before[kk] = before + incl - nb;
      }
      before += __shfl_sync(0xffffffffu, incl, 31);
      most = max(most, __reduce_max_sync(0xffffffffu, nb));
    }
    if (lane == 0) {
      s_before[n_w] = before;
      s_most = most;
    }
  };
  if (warp == 0 && !kOneList) fill_table(0);
  if (warp == NW - 1) {
    uint32_t qf[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) qf[c] = 0u;
    if (x < G) {  // (there is one query row, token 0)
      load_query(static_cast<const __nv_bfloat16*>(p.q) + (int64_t)b * p.qs.batch + (int64_t)(g * G + x) * p.qs.head, j, qf);
      if (step.rope) {  // the two pieces hold the two halves of the same pairs
        const float4* cs4 = reinterpret_cast<const float4*>(step.rope + (int64_t)step.position * (D / 2) + 16 * j);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 t = __ldg(cs4 + e);  // pairs 16j + 2e and the next
          const uint32_t lo = qf[e], hi = qf[8 + e];
          qf[e] = rotate_pair2(lo, hi, t, -1.f);
          qf[8 + e] = rotate_pair2(hi, lo, t, 1.f);
        }
      }
    }
    publish_query(s_q, qf, lane);
  }
  const __nv_bfloat16* kb = static_cast<const __nv_bfloat16*>(p.k) + (int64_t)b * p.ks.batch +
                            (int64_t)g * p.ks.head + 16 * j;
  const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(p.v) + (int64_t)b * p.vs.batch +
                            (int64_t)g * p.vs.head + 16 * x;
  const float cs = p.scale * 1.4426950408889634f;  // logits in log2 units
  DecodeState st;
  decode_init(st);

  // Each lane works out one of the warp's next 32 blocks.  kOneList: up to 32 shards, and no warp has more blocks than that; no
  // barrier stands before the requests of the first rows then.  (Table and query behind one barrier, then the list: 3500 cycles
  // before the first request.)
  // Order of the 16-key blocks.  If the visible prefixes are about equally long, block i of every shard comes before block
  // i + 1 of any: shards interleave in the sequence, so the warps of a cluster read one region of the cache together.
  // Otherwise shard after shard, which balances whatever the lengths are.
  __shared__ int2 s_list[NW][32];  // of this warp's next blocks: first position in kv_idx, keys left there
  auto gate = [&]() {  // the caches are complete before their rows are requested
    if (step.rope) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  };
  auto list = [&](int2 e) {  // those of the lanes' blocks that exist; how many
    const uint32_t there = __ballot_sync(0xffffffffu, e.y > 0);
    __syncwarp();
    if (e.y > 0) s_list[warp][__popc(there & ((1u << lane) - 1u))] = e;
    __syncwarp();
    return __popc(there);
  };
  if constexpr (kOneList) {  // lane = shard, then lane = block, in every warp by itself
    const int v = lane < P ? (vis_given ? step.vis[map * P + lane] : __ldg(vis + lane)) : 0;
    const int off = lane < P ? __ldg(kv_off + lane) : 0, nb = (v + 15) >> 4;
    int incl = nb;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), most = __reduce_max_sync(0xffffffffu, nb);
    const bool even = most * P * 4 <= total * 5;
    const int id = rank * NW + warp + lane * n_cta * NW;
    int kk = 0, i;
    if (even) {
      i = id / P;
      kk = id - i * P;
    } else {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {  // the last shard that starts at or before the block
        const int at = __shfl_sync(0xffffffffu, incl - nb, kk + o);
        if (kk + o < P && at <= id) kk += o;
      }
      i = id - __shfl_sync(0xffffffffu, incl - nb, kk);
    }
    const int left = __shfl_sync(0xffffffffu, v, kk) - i * 16, first = __shfl_sync(0xffffffffu, off, kk) + i * 16;
    const int listed = list(make_int2(first, id < (even ? most * P : total) ? left : 0));
    decode_walk<kAhead>(st, s_q, pl, kv_idx, listed, [&](int t) { return s_list[warp][t]; }, kb, p.ks.token, vb, p.vs.token, lane, cs,
                      gate, []() { __syncthreads(); });
  } else {
    gate();
#pragma unroll 1
    for (int w0 = 0; w0 < P; w0 += kFusedShards) {
      if (w0 > 0) {
        __syncthreads();
        if (warp == 0) fill_table(w0);
      }
      __syncthreads();
      const int n_w = min(kFusedShards, P - w0), total = s_before[n_w];
      const bool even = s_most * n_w * 4 <= total * 5;
      const int n_ids = even ? s_most * n_w : total;
#pragma unroll 1
      for (int id0 = rank * NW + warp; id0 < n_ids; id0 += 32 * n_cta * NW) {
        const int id = id0 + lane * n_cta * NW;
        int2 e = make_int2(0, 0);
        if (id < n_ids) {
          int kk, i;
          if (even) {
            kk = id % n_w;
            i = id / n_w;
          } else {
            int lo = 0, hi = n_w - 1;  // the last shard that starts at or before the block: it is not empty
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (s_before[mid] <= id) lo = mid;
              else hi = mid - 1;
            }
            kk = lo;
            i = id - s_before[kk];
          }
          e = make_int2(s_off[kk] + i * 16, s_vis[kk] - i * 16);
        }
        const int listed = list(e);
        decode_walk<kAhead>(st, s_q, pl, kv_idx, listed, [&](int t) { return s_list[warp][t]; }, kb, p.ks.token, vb, p.vs.token, lane, cs,
                          []() {}, []() {});
      }
    }
  }
  decode_publish<G, NW>(sh, st, warp, lane);
  if (!step.rope) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  __syncthreads();
  // The cluster's shares meet: CTA r finishes outputs r * per_cta ... ; every CTA sends it its share of them, and one barrier
  // later everything is in the receiver's own shared memory.
  const int per_cta = (G * D + n_cta - 1) / n_cta;
  auto send = [&](const float* local, int to, float v) {
    uint32_t addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(to));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
  };
  for (int i = tid; i < G * D; i += NW * 32) {
    float n_i, w_i, acc;
    decode_combine<G, NW>(sh, i / D, i % D, n_i, w_i, acc);
    const int to = i / per_cta;
    send(&s_o[rank * per_cta + i - to * per_cta], to, acc);
    if (i % D < n_cta) {  // one thread per (head, receiver)
      send(&s_n[rank][i / D], i % D, n_i);
      send(&s_w[rank][i / D], i % D, w_i);
    }
  }
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  // the plan's own prefixes and pair classes, for later calls on it (the caller's stream orders them after this kernel); of
  // several query shards one owns the only row, and the classes of the others are EMPTY as they were built
  if (vis_given && rank == 0 && g == 0 && (pl.n_maps > 1 || b == 0)) {
    const int J = pl.n_q_shards;
    const int32_t* q_off = pl.q_off + (size_t)map * (J + 1);
    for (int e = tid; e < J * P; e += NW * 32) {
      const int jj = e / P, kk = e - jj * P;
      if (J > 1 && q_off[jj] == q_off[jj + 1]) continue;
      const int v = step.vis[map * P + kk], len = kv_off[kk + 1] - kv_off[kk];
      const_cast<int32_t*>(vis)[kk] = v;
      const_cast<uint8_t*>(pl.pair_class)[((size_t)map * J + jj) * P + kk] =
          v == 0 ? CASCADE_PAIR_EMPTY : (v == len ? CASCADE_PAIR_FULL : CASCADE_PAIR_PARTIAL);
    }
  }
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int mine = min(per_cta, G * D - rank * per_cta);
  for (int o = tid; o < mine; o += NW * 32) {
    const int gg = (rank * per_cta + o) / D, col = (rank * per_cta + o) % D;
    float n_all = -INFINITY;
    for (int r = 0; r < n_cta; ++r) n_all = fmaxf(n_all, s_n[r][gg]);
    const float n_use = n_all == -INFINITY ? 0.f : n_all;
    float w = 0.f, acc = 0.f;
#pragma unroll 4
    for (int r = 0; r < n_cta; ++r) {
      const float f = ex2f(s_n[r][gg] - n_use);
      w = fmaf(f, s_w[r][gg], w);
      acc = fmaf(f, s_o[r * per_cta + o], acc);
    }
    const int h = g * G + gg;
    static_cast<__nv_bfloat16*>(p.o_out)[(int64_t)b * p.os.batch + (int64_t)h * p.os.head + col] =
        __float2bfloat16_rn(w > 0.f ? acc / w : 0.f);
    if (col == 0 && p.lse_out)
      p.lse_out[(int64_t)b * p.H + h] = w > 0.f ? n_use * 0.6931471805599453f + logf(w) : -INFINITY;
  }
}

template <int G, int kAhead>
static cudaError_t launch_fused(const AttnParams& p, const DecodeStep& step, int64_t blocks, int n_cta, cudaStream_t stream) {
  // One list: for as many keys as there are, whatever is visible when the launch runs (every shard may end in a block that is not
  // full, and in the interleaved order the list is a quarter longer).  Up to ten blocks a warp: beyond, the few registers that it
  // costs the walk weigh more (2 sequences of 16384 tokens, 32 / 8 heads, 34.5 us, from the table 32.4).  With four and eight
  // heads and one block ahead they do from the second block on (table -> list, us, 32 / 8 heads: 2 sequences of 1200 keys 9.6 ->
  // 9.2, of 3000 12.5 -> 12.8, of 6500 18.3 -> 19.0; 4 of 700 9.8 -> 9.4, of 1200 11.2 -> 11.7, of 6500 22.7 -> 24.3); with one and
  // two heads the walk from the table spills more (4 sequences of 3000 keys, 16 / 8 heads, 16.3 -> 14.6).
  const int P = p.plan.n_kv_shards;
  const bool one_list = P <= 32 && ((p.plan.n_kv + 15) / 16 + P) * (int64_t)5 / 4 + 1 <= 10 * (int64_t)n_cta * 8 &&
                        (kAhead == 2 || G <= 2 || blocks <= 8 * n_cta);
  auto kernel = one_list ? decode_fused_kernel<G, kAhead, true> : decode_fused_kernel<G, kAhead, false>;
  if (n_cta > 8) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  return launch_dependent(kernel, dim3(n_cta, p.Hkv, p.batch), 256, 0, n_cta, true, stream, p, step);
}

// How many clusters of n_cta CTAs that have an SM each the device holds at a time.
static int clusters_alone(int n_cta) {
  static std::atomic<int16_t> known[64][kMaxCluster + 1];  // number + 1; 0: not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::atomic<int16_t>& entry = known[dev][n_cta];
  if (const int n = entry.load(std::memory_order_relaxed)) return n - 1;
  auto kernel = decode_fused_kernel<8, 2, true>;  // (all forms with two blocks ahead take a whole SM)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_cta);
  cfg.blockDim = dim3(256);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = n_cta;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  cudaError_t e = n_cta > 8 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, kernel, &cfg);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  entry.store((int16_t)(std::min(n, 1000) + 1), std::memory_order_relaxed);
  return n;
}

// f(integral_constant G) for the group sizes the kernels are built for
template <typename F>
static cudaError_t with_group(int G, F f) {
  switch (G) {
    case 1: return f(std::integral_constant<int, 1>());
    case 2: return f(std::integral_constant<int, 2>());
    case 4: return f(std::integral_constant<int, 4>());
    case 8: return f(std::integral_constant<int, 8>());
    default: return cudaErrorInvalidValue;
  }
}

// CTAs per (KV head, sequence) where there are more than 128 pairs: the cluster size of 1 to 6 with the least estimated time.
// 296 CTAs fit at once (two per SM; about 280 in clusters that do not divide a GPC's share).  A round of them takes 8 us and
// what its CTAs take: 2 us per 16-key block of a warp, or what the reads of the round need at 6.8 TB/s, whichever is more; a
// last round with few CTAs is bound by the former.  (One CTA per pair left 24 CTAs to a second round at 320 pairs of 16000
// keys: 568 us, 5 per pair 403; 160 pairs 259 us, 3 per pair 200; 512 pairs 606 us, 2 per pair 638.  At 61 numbers of pairs
// from 144 to 600 and 500 to 16000 keys the choice is within 4 % of the fastest.)
static int cluster_for_many(int64_t pairs, int64_t blocks, int64_t most) {
  int best = 1;
  double least = 0;
  for (int n = 1; n <= std::min<int64_t>(6, most); ++n) {
    const int64_t fit = n <= 2 ? 296 : 280, ctas = pairs * n, rest = ctas % fit;
    const double alone = 2.0 * blocks / (8 * n), reads = fit * (blocks * 16 * 512.0) / n / 6.8e6;  // us
    const double t = (double)(ctas / fit) * (std::max(alone, reads) + 8) +
                     (rest ? std::max(alone, reads * rest / fit) + 8 : 0.0);
    if (n == 1 || t < least) {
      best = n;
      least = t;
    }
  }
  return best;
}

cudaError_t launch_decode_fused(const AttnParams& p, const DecodeStep& step, int64_t n_visible, cudaStream_t stream) {
  // CTAs (of eight warps) per (KV head, sequence): 256 in all, which is what two per SM on most of the chip come to with
  // every warp's loads in flight; more only repeat the set-up (16 sequences of 16384 tokens: 2 per pair 159 us, 4 163 us, 1
  // 165 us).  At most 10 where several pairs want the chip: clusters of 10 fit 11 times with one CTA per SM, clusters of 16
  // only 7 times (one sequence: 10 per pair 20.7 us, 16 22.8 us).  No more than give every warp a block.  More than 128 pairs:
  // see above.  `rule_kv_heads` counts the heads of the whole problem where a call computes a part of them.
  const int64_t pairs = (int64_t)p.rule_kv_heads * p.batch, blocks = std::max<int64_t>(1, (n_visible + 15) / 16);
  const int64_t most = std::min<int64_t>(pairs <= 7 ? kMaxCluster : 10, (blocks + 7) / 8);
  const int n_cta = pairs > 128 ? cluster_for_many(pairs, blocks, most) : (int)std::max<int64_t>(1, std::min(256 / pairs, most));
  // Two blocks ahead where every CTA gets an SM of its own all the same and its warps have a second block: with one, an SM holds
  // half the loads it could (one block ahead -> two, us, on caches new to L2: a step at 2500 rows, 32 / 8 heads, 9.9 -> 7.6; decode on
  // 1400 keys, 8 / 8 heads, 8.2 -> 6.7, on 16384, 32 / 8 heads, 30.7 -> 25.0, on 32768 54 -> 42).  Where the clusters do not all fit
  // that way, a second round costs more: 3 sequences of 8000 keys, 4 KV heads, 21 us, and 28 when CTAs that take a whole SM were
  // launched for them.  Sixteen warps a CTA, with a block ahead each, kept as many loads in flight (16384 keys 22 us, 2500 rows 8.2),
  // but a warp rounds its weights to bf16 against a maximum of its own, so another number of warps changes the result.
  const bool two_ahead = blocks > 8 * n_cta && (int64_t)p.Hkv * p.batch <= clusters_alone(n_cta);
  TimedLaunch timed(stream);
  return with_group(p.G, [&](auto g) {
    return two_ahead ? launch_fused<decltype(g)::value, 2>(p, step, blocks, n_cta, stream)
                     : launch_fused<decltype(g)::value, 1>(p, step, blocks, n_cta, stream);
  });
}

cudaError_t launch_decode(const AttnParams& p, cudaStream_t stream) {
  dim3 grid(p.plan.n_kv_shards, p.Hkv, p.batch);
  TimedLaunch timed(stream);
  const cudaError_t e = with_group(p.G, [&](auto g) {
    decode_kernel<decltype(g)::value><<<grid, 128, 0, stream>>>(p);
    return cudaGetLastError();
  });
  count_launch();
  return e;
}

}  // namespace cascade
