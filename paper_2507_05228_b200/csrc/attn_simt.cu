// Attention-pass on the fp32 ALUs (the Attention-Pass algorithm), used for fp32 inputs and for shapes the tensor-core kernel
// does not take.  Bound by FFMA issue: 4 d FLOP per visible pair and head at 128 FMA lanes per SM.
//
// Both products are register-tiled with packed fma.rn.f32x2.  A warp owns 16 query rows; lane = (row group rg = lane / 8,
// column group cg = lane % 8); a thread owns rows rg + 4 r (r < 4) in both products.
//   q k^T: keys cg + 8 j; the halves of a packed accumulator take the even and the odd terms of the sum over head_dim, so
//          both operands are plain 16-byte pieces of rows (64 keys: 12 loads per 64 packed FMAs).
//   p v:   columns 4 cg + 32 jj .. + 3 as packed pairs; P is written to shared memory twice over, (p, p), so that it needs
//          no duplicating moves (8 loads per 32 packed FMAs).
// Every one of these loads is a single conflict-free wavefront.  K of the next tile is fetched with cp.async while the
// current weights are formed and multiplied with V, and V while the next logits are.
// The key stream is cut into chunks of 16 keys, of one shard (partials) or of the sequence (kTokens, the fused route), so the mask is
// one limit per (row, chunk); tiles that the CTA's first row sees completely skip it.
// Fused, of all shards a query sees a prefix in token order, so rows and keys are taken as they lie: nothing is looked up in the
// plan before they are requested, and a shard of a few keys does not end in a chunk of its own.  (Shard by shard, one sequence of
// 128 tokens had its key rows requested after 7000 of 14000 cycles.)
//
// RW = 4: the four warps own different rows and share the K/V tiles.  RW = 1: all four warps own the same rows and take the
// tiles (32 keys) of the stream in turn; their (m, l, o) are combined at the end.  Small problems and short shards use the
// latter: four times as many CTAs, four times shorter chains, less padding.
// Measured (fp32): 16 sequences of 512 tokens, 16 heads of 64, 8 shards, bidirectional, fused 540 us = 32 TFLOP/s (partials
// and merge 708 us, before 1662 us with one row at a time per warp); one sequence of 128 tokens, 12 heads, 2 shards: 8.4 us
// (in token order; shard by shard 10.5, a row at a time 35).  What bounds it now is shared-memory bandwidth: 448 16-byte loads (4 cycles each) against 2048 packed FMAs
// per warp and 16 x 64 tile.
#include "cascade_internal.cuh"

namespace cascade {

namespace {

__device__ __forceinline__ float4 load4(const __nv_bfloat16* src) {
  const uint2 t = __ldg(reinterpret_cast<const uint2*>(src));
  return make_float4(__uint_as_float(t.x << 16), __uint_as_float(t.x & 0xffff0000u), __uint_as_float(t.y << 16),
                     __uint_as_float(t.y & 0xffff0000u));
}
__device__ __forceinline__ void store4(float* dst, float4 v) { *reinterpret_cast<float4*>(dst) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* dst, float4 v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}
// Four values of a row into shared memory: asynchronously for fp32, converted on the way for bf16; zeros if !there.
__device__ __forceinline__ void stage4(float* dst, const float* src, bool there) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(there ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* src, bool there) {
  *reinterpret_cast<float4*>(dst) = there ? load4(src) : make_float4(0.f, 0.f, 0.f, 0.f);
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ float ex2(float x) {  // 2^x; ex2(-inf) = +0
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ void ffma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float sum2(uint64_t v) {
  float lo, hi;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
  return lo + hi;
}

__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// Shared-memory layout, in floats.
template <int D, int RW>
struct SimtCfg {
  static constexpr int KW = 4 / RW;                       // groups of warps that take tiles in turn
  static constexpr int WR = 16;                           // rows per warp
  static constexpr int R = RW * WR;                       // rows per CTA
  static constexpr int BN = RW == 4 && D == 64 ? 64 : 32; // keys per tile
  static constexpr int NC = BN / 16;                      // chunks per tile
  static constexpr int QP = D + 4, KP = D + 4;            // row pitches
  static constexpr int PP = 2 * 32 + 16;                  // P rows: 32 keys, twice
  static constexpr int kQ = R * QP, kK = BN * KP, kV = BN * D, kP = WR * PP + 4;
  static constexpr int kGroup = kK + kV + RW * kP;        // one group's K, V and P
  static constexpr int kStats = KW > 1 ? KW * WR * 2 : 0;
  static constexpr size_t kBytes = sizeof(float) * (kQ + KW * kGroup + kStats);
  static constexpr int kCtas = RW == 4 ? (D == 64 ? 3 : 2) : (D == 64 ? 2 : 1);
  static_assert(KW == 1 || kK >= WR * D, "a group's output is staged in its K tile");
  static_assert(kCtas * (kBytes + 1024) <= 233472, "CTAs per SM");
};

constexpr int64_t kEnough = 2 * 148;  // CTAs that fill the chip, two per SM

// A tile of the key stream: per chunk of 16 keys its first key in the stream and in the plan's list, and the keys from there on.
template <int NC>
struct SimtTile {
  int t0[NC], n[NC], at[NC];
  bool any, masked;
};

template <typename T, int D, int RW, bool kTokens>
__global__ void __launch_bounds__(128, SimtCfg<D, RW>::kCtas)
attn_simt_kernel(const __grid_constant__ AttnParams p, int parts_per_cta) {
  using C = SimtCfg<D, RW>;
  constexpr int TR = 4, NC = C::NC, BN = C::BN, KJ = BN / 8, DJ = D / 32;
  constexpr int kGroupThreads = RW * 32;
  extern __shared__ __align__(16) float smem_f[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int group = warp / RW, gtid = tid % kGroupThreads;
  const int rg = lane >> 3, cg = lane & 7;
  const int wrow = RW == 4 ? warp * C::WR : 0;  // first row of this warp in the CTA's tile
  float* sQ = smem_f;
  float* sK = smem_f + C::kQ + group * C::kGroup;
  float* sV = sK + C::kK;
  // row rg + 4 r of P starts at (rg + 4 r) PP + 4 (rg / 2): the writes of two row groups and the reads of all four fall
  // into different banks
  float* sP = sV + C::kV + (RW == 4 ? warp * C::kP : 0) + rg * C::PP + 4 * (rg >> 1);

  const PlanDev& pl = p.plan;
  const int P = pl.n_kv_shards;
  const int n_pg = kTokens ? 1 : (P + parts_per_cta - 1) / parts_per_cta;
  const int b = kTokens ? blockIdx.z : blockIdx.z / n_pg;
  const int pg = kTokens ? 0 : blockIdx.z % n_pg;
  const int map = pl.n_maps == 1 ? 0 : b;
  const int h = blockIdx.y;
  const int g = p.G == 1 ? h : h / p.G;
  // the plan's tiles of 64 slots, or of 32 slots in two pieces
  constexpr int kList = RW == 4 ? 1 : 0, kPieces = (32 << kList) / C::R;
  int row0, nrows;  // slots of a query shard, or tokens, the last ones (which see most) first
  if constexpr (kTokens) {
    row0 = (int)(gridDim.x - 1 - blockIdx.x) * C::R;
    nrows = min(C::R, pl.n_q - row0);
  } else {
    const int4 qt = pl.qtiles[kList][(size_t)map * pl.n_qtiles[kList] + blockIdx.x / kPieces];
    row0 = qt.x + (blockIdx.x % kPieces) * C::R;
    nrows = min(C::R, qt.y - (int)(blockIdx.x % kPieces) * C::R);
    if (nrows <= 0) return;
  }
  const int32_t* q_idx = pl.q_idx + (size_t)map * pl.n_q;
  const int32_t* kv_idx = pl.kv_idx + (size_t)map * pl.n_kv;
  const int32_t* kv_off = pl.kv_off + (size_t)map * (P + 1);
  const int32_t* vis = pl.vis + (size_t)map * pl.n_q * P;
  // rows ascend: the first has the shortest prefix of every shard, the last the longest
  const int32_t* vis_first = vis + (size_t)row0 * P;
  const int32_t* vis_last = vis + (size_t)(row0 + nrows - 1) * P;
  auto token_of = [&](int r) {
    if constexpr (kTokens) return (int64_t)(row0 + r);
    else return (int64_t)CASCADE_CHECKED((int64_t)__ldg(q_idx + row0 + r), pl.n_q, pl.status, 104);
  };
  auto seen_by = [&](int r) {  // kTokens: keys of the sequence that the row sees
    if (!pl.causal) return pl.n_kv;
    if (!p.prefix_from_vis) return (int)max((int64_t)0, min((int64_t)pl.n_kv, (int64_t)pl.q_pos_offset + row0 + r + 1));
    const int32_t* of = vis + (size_t)__ldg(pl.q_inv + (size_t)map * pl.n_q + row0 + r) * P;
    int n = 0;
    for (int k = 0; k < P; ++k) n += __ldg(of + k);
    return n;
  };
  const int seen_first = kTokens ? seen_by(0) : 0, seen_last = kTokens ? seen_by(nrows - 1) : 0;
  const T* qb = static_cast<const T*>(p.q) + (int64_t)b * p.qs.batch + (int64_t)h * p.qs.head;
  const T* kb = static_cast<const T*>(p.k) + (int64_t)b * p.ks.batch + (int64_t)g * p.ks.head;
  const T* vb = static_cast<const T*>(p.v) + (int64_t)b * p.vs.batch + (int64_t)g * p.vs.head;

  for (int i = tid; i < C::R * (D / 4); i += 128) {
    const int r = i / (D / 4), c4 = (i % (D / 4)) * 4;
    const int64_t tok = r < nrows ? token_of(r) : (int64_t)0;
    stage4(sQ + r * C::QP + c4, qb + tok * p.qs.token + c4, r < nrows);
  }
  stage_commit();
  auto group_sync = [&]() {
    if constexpr (RW == 4) __syncthreads();
    else __syncwarp();
  };
  // one tile of K or V rows
  constexpr int kPerRow = D / 4, kRowsAtOnce = kGroupThreads / kPerRow;
  const int lr = gtid / kPerRow, lc = (gtid % kPerRow) * 4;
  auto stage_tile = [&](const SimtTile<NC>& t, const T* base, int64_t token_stride, float* dst, int pitch) {
#pragma unroll
    for (int j = 0; j < NC; ++j)
#pragma unroll
      for (int i = 0; i < 16 / kRowsAtOnce; ++i) {
        const int x = i * kRowsAtOnce + lr;
        const bool there = x < t.n[j];
        int64_t tok = 0;
        if constexpr (kTokens) {
          if (there) tok = t.at[j] + x;
        } else if (there) {
          tok = CASCADE_CHECKED((int64_t)__ldg(kv_idx + t.at[j] + x), pl.n_kv, pl.status, 105);
        }
        stage4(dst + (j * 16 + x) * pitch + lc, base + tok * token_stride + lc, there);
      }
    stage_commit();
  };
  const int my_row = wrow + rg;  // this thread's rows: my_row + 4 r
  int seen[kTokens ? TR : 1];
  if constexpr (kTokens) {
#pragma unroll
    for (int r = 0; r < TR; ++r) seen[r] = seen_by(min(my_row + 4 * r, nrows - 1));
  }
  const float cs = p.scale * 1.4426950408889634f;  // raw logits -> log2 units

  float m_run[TR], l_run[TR];  // raw logits; l is this thread's share (its key columns)
  uint64_t acc[TR][2 * DJ];

  const int k_first = kTokens ? 0 : pg * parts_per_cta, k_last = kTokens ? 1 : min(P, (pg + 1) * parts_per_cta);
  for (int part = k_first; part < k_last; ++part) {
#pragma unroll
    for (int r = 0; r < TR; ++r) {
      m_run[r] = -INFINITY;
      l_run[r] = 0.f;
#pragma unroll
      for (int j = 0; j < 2 * DJ; ++j) acc[r][j] = 0;
    }
    // cursor over the chunks of shard `part`, or of the sequence
    int c = group * NC;
    const int need = kTokens ? seen_last : __ldg(vis_last + part);
    const int first = kTokens ? seen_first : __ldg(vis_first + part), at0 = kTokens ? 0 : __ldg(kv_off + part);
    auto next_tile = [&](SimtTile<NC>& t) {
      t.masked = false;
      t.any = c * 16 < need;
#pragma unroll
      for (int j = 0; j < NC; ++j) {
        t.t0[j] = c * 16;
        t.n[j] = need - c * 16;
        t.at[j] = at0 + c * 16;
        t.masked = t.masked || first < c * 16 + 16;
        ++c;
      }
      c += (C::KW - 1) * NC;  // the other groups' tiles
    };
    SimtTile<NC> cur, nxt;
    next_tile(cur);
    group_sync();  // the tiles of the previous part are consumed
    if (cur.any) {
      stage_tile(cur, kb, p.ks.token, sK, C::KP);
      stage_tile(cur, vb, p.vs.token, sV, D);
    }
    // the query rows, staged by all threads, are the oldest group
    if (part == k_first) {
      if (cur.any) stage_wait<2>();
      else stage_wait<0>();
      __syncthreads();
    }
    while (cur.any) {
      stage_wait<1>();  // K is there (V is the later group)
      group_sync();
      // logits: rows my_row + 4 r, keys cg + 8 j
      float s[TR][KJ];
      {
        uint64_t s2[TR][KJ];
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int j = 0; j < KJ; ++j) s2[r][j] = 0;
#pragma unroll 2
        for (int d4 = 0; d4 < D / 4; ++d4) {
          ulonglong2 qf[TR];
#pragma unroll
          for (int r = 0; r < TR; ++r)
            qf[r] = *reinterpret_cast<const ulonglong2*>(sQ + (my_row + 4 * r) * C::QP + d4 * 4);
#pragma unroll
          for (int j = 0; j < KJ; ++j) {
            const ulonglong2 kf = *reinterpret_cast<const ulonglong2*>(sK + (cg + 8 * j) * C::KP + d4 * 4);
#pragma unroll
            for (int r = 0; r < TR; ++r) {
              ffma2(s2[r][j], qf[r].x, kf.x);
              ffma2(s2[r][j], qf[r].y, kf.y);
            }
          }
        }
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int j = 0; j < KJ; ++j) s[r][j] = sum2(s2[r][j]);
      }
      next_tile(nxt);
      group_sync();  // K is consumed
      if (nxt.any) stage_tile(nxt, kb, p.ks.token, sK, C::KP);
      // mask, running maximum, weights
      if (cur.masked) {
#pragma unroll
        for (int r = 0; r < TR; ++r) {
          const int sees = kTokens ? seen[kTokens ? r : 0] : __ldg(vis + (size_t)(row0 + min(my_row + 4 * r, nrows - 1)) * P + part);
#pragma unroll
          for (int j = 0; j < KJ; ++j) {
            const int ch = j >> 1;
            if (cg + 8 * (j & 1) >= sees - cur.t0[ch]) s[r][j] = -INFINITY;
          }
        }
      }
      float alpha[TR];
#pragma unroll
      for (int r = 0; r < TR; ++r) {
        float mx = s[r][0];
#pragma unroll
        for (int j = 1; j < KJ; ++j) mx = fmaxf(mx, s[r][j]);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m_run[r], mx);
        const float m_use = m_new == -INFINITY ? 0.f : m_new;
        alpha[r] = ex2((m_run[r] - m_use) * cs);  // 0 on the first visible tile
        m_run[r] = m_new;
        float ps = 0.f;
#pragma unroll
        for (int j = 0; j < KJ; ++j) {
          s[r][j] = ex2((s[r][j] - m_use) * cs);
          ps += s[r][j];
        }
        l_run[r] = l_run[r] * alpha[r] + ps;
        const uint64_t a2 = pack2(alpha[r], alpha[r]);
#pragma unroll
        for (int j = 0; j < 2 * DJ; ++j) acc[r][j] = fmul2(acc[r][j], a2);
      }
      if (nxt.any) stage_wait<1>();  // V is there (the next K is the later group)
      else stage_wait<0>();
      group_sync();
      // output: rows my_row + 4 r, columns 4 cg + 32 jj, 32 keys at a time
#pragma unroll
      for (int half = 0; half < BN / 32; ++half) {
        __syncwarp();  // the previous weights are consumed
#pragma unroll
        for (int r = 0; r < TR; ++r)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float w = s[r][4 * half + j];
            *reinterpret_cast<float2*>(sP + 4 * r * C::PP + 2 * (cg + 8 * j)) = make_float2(w, w);
          }
        __syncwarp();
        const float* v_half = sV + half * 32 * D + 4 * cg;
#pragma unroll 4
        for (int k2 = 0; k2 < 16; ++k2) {
          ulonglong2 v0[DJ], v1[DJ];
#pragma unroll
          for (int jj = 0; jj < DJ; ++jj) {
            v0[jj] = *reinterpret_cast<const ulonglong2*>(v_half + (2 * k2) * D + 32 * jj);
            v1[jj] = *reinterpret_cast<const ulonglong2*>(v_half + (2 * k2 + 1) * D + 32 * jj);
          }
#pragma unroll
          for (int r = 0; r < TR; ++r) {
            const ulonglong2 pf = *reinterpret_cast<const ulonglong2*>(sP + 4 * r * C::PP + 4 * k2);
#pragma unroll
            for (int jj = 0; jj < DJ; ++jj) {
              ffma2(acc[r][2 * jj], pf.x, v0[jj].x);
              ffma2(acc[r][2 * jj + 1], pf.x, v0[jj].y);
              ffma2(acc[r][2 * jj], pf.y, v1[jj].x);
              ffma2(acc[r][2 * jj + 1], pf.y, v1[jj].y);
            }
          }
        }
      }
      group_sync();  // V is consumed
      if (nxt.any) stage_tile(nxt, vb, p.vs.token, sV, D);
      cur = nxt;
    }

    // ---- write (u, m, l) of the shard or the finished rows
    auto put = [&](int row, int col, float4 o, float m_raw, float l, bool stats) {
      const float inv = l > 0.f ? 1.f / l : 0.f;
      o.x *= inv;
      o.y *= inv;
      o.z *= inv;
      o.w *= inv;
      if constexpr (kTokens) {
        const int64_t tok = row0 + row;
        store4(static_cast<T*>(p.o_out) + (int64_t)b * p.os.batch + tok * p.os.token + (int64_t)h * p.os.head + col,
               o);
        if (stats && p.lse_out)
          p.lse_out[((int64_t)b * pl.n_q + tok) * p.H + h] = l > 0.f ? m_raw * p.scale + logf(l) : -INFINITY;
      } else {
        const int64_t stat = (((int64_t)b * P + part) * pl.n_q + (row0 + row)) * p.H + h;
        store4(static_cast<T*>(p.o_part) + stat * D + col, o);
        if (stats) {
          p.m_part[stat] = l > 0.f ? m_raw * p.scale : -INFINITY;
          p.l_part[stat] = l;
        }
      }
    };
    float* stats = smem_f + C::kQ + C::KW * C::kGroup;  // KW > 1: [group][row][m, l]
    if (C::KW > 1) __syncwarp();                        // the group's K tile is consumed
#pragma unroll
    for (int r = 0; r < TR; ++r) {
      const int row = my_row + 4 * r;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) l_run[r] += __shfl_xor_sync(0xffffffffu, l_run[r], o);
      if (C::KW > 1 && cg == 0) {
        stats[(group * C::WR + row) * 2] = m_run[r];
        stats[(group * C::WR + row) * 2 + 1] = l_run[r];
      }
#pragma unroll
      for (int jj = 0; jj < DJ; ++jj) {
        float4 o;
        unpack2(acc[r][2 * jj], o.x, o.y);
        unpack2(acc[r][2 * jj + 1], o.z, o.w);
        if (C::KW > 1) *reinterpret_cast<float4*>(sK + row * D + 4 * cg + 32 * jj) = o;
        else if (row < nrows) put(row, 4 * cg + 32 * jj, o, m_run[r], l_run[r], cg == 0 && jj == 0);
      }
    }
    if constexpr (C::KW > 1) {
      __syncthreads();
      for (int i = tid; i < nrows * (D / 4); i += 128) {
        const int row = i / (D / 4), col = (i % (D / 4)) * 4;
        float n = -INFINITY;
#pragma unroll
        for (int w = 0; w < C::KW; ++w) n = fmaxf(n, stats[(w * C::WR + row) * 2]);
        const float n_use = n == -INFINITY ? 0.f : n;
        float l = 0.f;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < C::KW; ++w) {
          const float f = ex2((stats[(w * C::WR + row) * 2] - n_use) * cs);
          const float4 t = *reinterpret_cast<const float4*>(smem_f + C::kQ + w * C::kGroup + row * D + col);
          l = fmaf(f, stats[(w * C::WR + row) * 2 + 1], l);
          o.x = fmaf(f, t.x, o.x);
          o.y = fmaf(f, t.y, o.y);
          o.z = fmaf(f, t.z, o.z);
          o.w = fmaf(f, t.w, o.w);
        }
        put(row, col, o, n, l, col == 0);
      }
      __syncthreads();
    }
  }
}

template <typename T, int D, int RW>
cudaError_t launch_rows(const AttnParams& p, int parts_per_cta, cudaStream_t stream) {
  using C = SimtCfg<D, RW>;
  auto kernel = p.fused ? attn_simt_kernel<T, D, RW, true> : attn_simt_kernel<T, D, RW, false>;
  // per function and per device; cheap enough to repeat on every launch
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kBytes);
  if (e != cudaSuccess) return e;
  constexpr int kList = RW == 4 ? 1 : 0, kPieces = (32 << kList) / C::R;
  const int n_pg = p.fused ? 1 : (p.plan.n_kv_shards + parts_per_cta - 1) / parts_per_cta;
  const dim3 grid(p.fused ? (p.plan.n_q + C::R - 1) / C::R : p.plan.n_qtiles[kList] * kPieces, p.H, p.batch * n_pg);
  kernel<<<grid, 128, C::kBytes, stream>>>(p, parts_per_cta);
  count_launch();
  return cudaGetLastError();
}

// Tiles of `height` rows (16 or 64): of tokens (fused), or of the plan's list.
int64_t simt_tiles(const AttnParams& p, int height) {
  return p.fused ? (p.plan.n_q + height - 1) / height : height == 64 ? p.plan.n_qtiles[1] : p.plan.n_qtiles[0];
}

// Whether four row warps share a CTA: when that fills the chip (two CTAs per SM) and does not pad the rows by more than what the
// narrow form's four times larger K/V traffic costs.  It decides how sums are split, so it goes by the heads of the whole
// problem (see AttnParams).
bool use_wide(const AttnParams& p) {
  const int64_t tiles = simt_tiles(p, 64), heads = (int64_t)p.rule_kv_heads * p.G * p.batch;
  const int64_t narrow_rows = (int64_t)p.plan.n_q + (int64_t)(p.fused ? 1 : p.plan.n_q_shards) * 8;  // padded by half a piece a shard
  return tiles * heads * (p.fused ? 1 : p.plan.n_kv_shards) >= kEnough && tiles * 64 * 4 <= narrow_rows * 6;
}

// partials: a CTA walks as many shards of its rows as leaves enough CTAs
int parts_per_cta(const AttnParams& p, int64_t ctas) {
  const int P = p.plan.n_kv_shards;
  return p.fused ? 1 : (int)std::max<int64_t>(1, P / std::min<int64_t>(P, (kEnough + ctas - 1) / ctas));
}
int64_t narrow_pieces(const AttnParams& p) {
  return std::max<int64_t>(1, ((int64_t)p.plan.n_q + (int64_t)p.plan.n_q_shards * 8) / 16);
}

template <typename T, int D>
cudaError_t launch_one(const AttnParams& p, cudaStream_t stream) {
  const int64_t heads = (int64_t)p.H * p.batch;
  if (use_wide(p)) return launch_rows<T, D, 4>(p, parts_per_cta(p, simt_tiles(p, 64) * heads), stream);
  return launch_rows<T, D, 1>(p, parts_per_cta(p, narrow_pieces(p) * heads), stream);
}

}  // namespace

// Estimated time in us, see rows_time.  At head_dim 64 a shard costs an SM 2 us and 6.2 us per 64 keys for 64 rows in the wide
// form, and 2.4 us and 0.45 us (from the fifth on, 0.71) per 32 keys for 16 rows in the narrow one.
double tiles_time(const AttnParams& p) {
  const CutSize c(p);
  const bool d64 = p.d == 64;
  if (use_wide(p)) {
    const double list = simt_tiles(p, 64);
    const double seen = p.fused ? c.seen_at((list + 1) / (2 * list)) : c.seen_by_last(list), chunks = std::ceil(seen * c.n_kv / 16);
    const double cta = d64 ? 2 + 6.2 * (p.fused ? chunks / 4 : c.pieces(seen, 64))
                           : 2 + 5 * (p.fused ? chunks / 2 : c.pieces(seen, 32));
    return list * c.heads * cta * (p.fused ? 1 : c.shards) / kEstimateSms;
  }
  const double pieces = p.fused ? simt_tiles(p, 16) : c.row_tiles(16);
  const double seen = p.fused ? c.seen_at((pieces + 1) / (2 * pieces)) : c.seen_by_last(pieces);
  const double tiles = p.fused ? std::ceil(seen * c.n_kv / 32) : c.pieces(seen, 32);
  const double cta = d64 ? 2.4 + 0.45 * std::min(tiles, 4.0) + 0.71 * std::max(0.0, tiles - 4)
                         : 1 + (p.fused ? 10 : 7.2) * std::max(1.0, tiles / 4);
  const double parts = parts_per_cta(p, std::max<int64_t>(1, (int64_t)(narrow_pieces(p) * c.heads)));
  const double ctas = pieces * c.heads * (p.fused ? 1 : std::ceil(c.shards / parts));
  return cta * parts * std::max(1.0, ctas / kEstimateSms);
}

cudaError_t launch_attn_simt(const AttnParams& p, cascade_dtype_t dtype, cudaStream_t stream) {
  if (0.97 * rows_time(p) < tiles_time(p)) return launch_attn_rows(p, dtype, stream);  // (a tie goes to the simpler kernel)
  if (dtype == CASCADE_BF16) {
    if (p.d == 128) return launch_one<__nv_bfloat16, 128>(p, stream);
    return launch_one<__nv_bfloat16, 64>(p, stream);
  }
  if (p.d == 128) return launch_one<float, 128>(p, stream);
  return launch_one<float, 64>(p, stream);
}

}  // namespace cascade
