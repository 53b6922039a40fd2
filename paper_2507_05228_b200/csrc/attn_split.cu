// fp32 attention-pass on the tensor cores (the Attention-Pass algorithm, and the fused route), head_dim 64.
//
// Every fp32 operand is taken apart into three bf16 numbers, x = x0 + x1 + x2 (each the rounded rest of what came before; 24 bits
// in all, so from 2^-110 on, where the last bit is bf16's smallest number, nothing is left out), and a product x y becomes six bf16 products, those of order up to 2^-16:
//   x0 y2 + x2 y0 + x1 y1 + x0 y1 + x1 y0 + x0 y0;  what is left out (x1 y2, x2 y1, x2 y2) is below 2^-24 |x y|.
// The tensor core cuts its fp32 sums off at every step.  So the small products come first, the large ones of a logit are shared by two
// accumulators (two steps at full size each), and those and the outputs of different key tiles are added up in registers.
// Logits, weights, row sums and outputs stay fp32 as on the ALUs.  Relative error (2-norm, against fp64) at 16 x 512 tokens, 16 heads,
// fused: 1.75e-7, on the ALUs 4.5e-7; m and l of the partials 5.5e-8 and 9.7e-8, on the ALUs 7.7e-8 and 1.65e-7.  With values of one
// sign, where what is cut off adds up, the order is the same (16 to 4000 keys); logits come out 0.7 * 2^-24 small in the mean, so
// where all have one sign the logarithm of the row sum is off by 4.3e-8 of itself, on the ALUs by 3.3e-8.
//
// Work.  A first kernel splits K and V, in shard-major order (kParts) or token order (fused), so that every row is split once.  Then
// a CTA takes two sub-tiles of 128 MMA rows, the Gp heads of one KV head stacked: 2 x 128 / Gp consecutive tokens, whichever query
// shards they are in (their rows of vis say what they see), and walks the keys in tiles of 64: of the KV shards one after another
// (kParts; a tile keeps to its shard, at whose end (u, m, l) is written out) or of the whole sequence.  Consecutive tokens see
// almost the same prefix of a shard, so little is computed in vain under the causal mask.  (Keys and values split by the CTAs
// themselves, by warps of their own or by those of the softmax, were what the products waited for.)
// Warps: 0-7 softmax of sub-tile 0, 8-15 of sub-tile 1 (two threads per MMA row = TMEM lane, each with 32 keys of a tile and 32
// output columns; at the start they split the query rows), 16 issues the products, 17 loads K, 18 V (all parts of a tile in
// one box; it says which sub-tiles see anything of the tile, too, so that the issuing thread has no list to walk).
// TMEM, per sub-tile: logits 3 x 64 columns, to be added up: large products of the first 32 columns of head_dim, of the last 32, and
// small ones.  One instruction multiplies a part of Q with several parts of K, one below the other in shared memory (930 cycles a
// tile where six separate products take 1200, bound by the reads of Q).  The weights, 3 x 32 columns of bf16 pairs, go over the
// logits; output 64.
// Products go out as PV_0(i), QK_0(i+1), PV_1(i), QK_1(i+1): one sub-tile's softmax runs under the other's products, and QK(i+1)
// may overwrite the weights that PV(i) reads, because they execute in this order.  (A warp for either sub-tile: their products
// then alternate one by one, 163 -> 187 us at 16 x 512 tokens, 16 heads, fused.)
// What bounds it: the chain of a sub-tile, weights -> output -> (logits) -> weights, about 5500 cycles a tile, in which the tensor
// cores are busy for 3500; with partials the stores (60 of 234 us at 16 x 512 tokens in 8 shards).
//
// Out of range are values of 2^63 and beyond, infinities and NaN, whose parts could turn a result into NaN that fp32 arithmetic keeps;
// queries and keys all of whose columns are below 2^-100, and columns of values that are in 64 rows, unless they are zero: of those the
// parts lose bits (relative error of the output with all values of size 2^-110 1.2e-7 as ever, 2^-115 1.1e-6, 2^-120 3.5e-5).  Beside a
// larger one, what is lost of a value is below 2^-34 of it.  A tile with such keys or values, and every tile of a CTA with such
// queries, is worked out in plain fp32 by the softmax threads, slowly: fused,
// 16 x 512 tokens, 16 heads, 148 us; with one such key, or value, in every head 1.1 ms, or 1.6; with all of them 7.4, or 12.
#include "tcgen05.cuh"

namespace cascade {
namespace split {

using namespace tc;

constexpr int kThreads = 640, kWarps = kThreads / 32;
constexpr int kM = 128, kN = 64, kD = 64;  // MMA rows, keys per tile, head_dim
constexpr int kMaxShards = 256;
constexpr uint32_t kTmemCols = 512, kSubCols = 256, kOCol = 192;
// 96 registers x 640 threads at launch = 512 x 104 + 128 x 64
constexpr int kRegsSoftmax = 104, kRegsOther = 64;
static_assert(512 * kRegsSoftmax + 128 * kRegsOther <= 96 * kThreads, "setmaxnreg would wait for registers forever");

// shared memory, from a 1024-byte aligned base; operand tiles are [part][row][128 bytes]
constexpr int kQPart = kM * 128, kKvPart = kN * 128;
constexpr int kQTile = 3 * kQPart, kKvTile = 3 * kKvPart;
constexpr int kOffQ = 0, kOffK = kOffQ + 2 * kQTile, kOffV = kOffK + 2 * kKvTile;
constexpr int kOffMax = kOffV + 2 * kKvTile;        // float [2][sub-tile][half][row], maxima of a tile; [..] sums of a shard
constexpr int kOffTab = kOffMax + 3 * 4 * kM * 4;   // int32 [2][2][kMaxShards]: longest and shortest prefix of a sub-tile's rows
constexpr int kOffBar = kOffTab + 4 * kMaxShards * 4;
constexpr int kOffMisc = kOffBar + 32 * 8;          // TMEM address, abort flag, progress words, see WaitCtx
constexpr int kOffFar = kOffMisc + 8 + 4 * kWarps;  // int32: kFarQ, kFarK, kFarV, whether any such row of the CTA is out of range
constexpr int kOffInfo = kOffFar + 4;               // int32 [3]: see tile_info
constexpr int kFarWords = 128;                      // keys, values: a bit for every 64 << far_shift rows, whether one is out of range
constexpr int kOffFarRows = kOffInfo + 12;          // uint32 [2][kFarWords]
constexpr int kSmemBytes = kOffFarRows + 2 * kFarWords * 4 + 1024;
static_assert(kSmemBytes <= 232448, "exceeds the 227 KiB a CTA may use");

// two of each: by sub-tile, or by stage
enum { kFarQ = 1, kFarK = 2, kFarV = 4 };
enum Bar { Q_FULL = 0, S_FULL = 2, P_FULL = 6, O_FULL = 8, K_FULL = 10, K_EMPTY = 12, V_FULL = 14, V_EMPTY = 16, DONE = 18 };

__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// (a, b) -> their three parts, packed
__device__ __forceinline__ void split2(float a, float b, uint32_t& x0, uint32_t& x1, uint32_t& x2) {
  x0 = pack_bf16x2(a, b);
  const float a1 = a - __uint_as_float(x0 << 16), b1 = b - __uint_as_float(x0 & 0xffff0000u);
  x1 = pack_bf16x2(a1, b1);
  x2 = pack_bf16x2(a1 - __uint_as_float(x1 << 16), b1 - __uint_as_float(x1 & 0xffff0000u));
}
// Eight values of a row into the three tiles at `to`; `big` turns NaN if one of them is 2^63 or more, infinite or NaN.
__device__ __forceinline__ void store_split8(uint8_t* to, int64_t part_bytes, const float4& u, const float4& v, uint64_t& big) {
  uint4 x[3];
  split2(u.x, u.y, x[0].x, x[1].x, x[2].x);
  split2(u.z, u.w, x[0].y, x[1].y, x[2].y);
  split2(v.x, v.y, x[0].z, x[1].z, x[2].z);
  split2(v.z, v.w, x[0].w, x[1].w, x[2].w);
#pragma unroll
  for (int i = 0; i < 3; ++i) *reinterpret_cast<uint4*>(to + i * part_bytes) = x[i];
  const uint64_t far = pack2(3.6893488e19f, 3.6893488e19f), zero = pack2(0.f, 0.f);  // 2^65
  big = ffma2(fmul2(pack2(u.x, u.y), far), zero, big);
  big = ffma2(fmul2(pack2(u.z, u.w), far), zero, big);
  big = ffma2(fmul2(pack2(v.x, v.y), far), zero, big);
  big = ffma2(fmul2(pack2(v.z, v.w), far), zero, big);
}
__device__ __forceinline__ bool is_big(uint64_t big) {
  float a, b;
  unpack2(big, a, b);
  return !(a + b == 0.f);
}

// bits i of `some` and `most`: whether x[i] is not zero, and whether it is 2^-100 or more
__device__ __forceinline__ void note_size(const float4& u, const float4& v, uint32_t& some, uint32_t& most) {
  const float x[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    some |= x[i] != 0.f ? 1u << i : 0u;
    most |= fabsf(x[i]) >= 7.888609e-31f ? 1u << i : 0u;
  }
}
// Whether the row of eight threads that this thread is in has no such value of 2^-100 or more, and is not zero.  By whole warps.
__device__ __forceinline__ bool is_small_row(uint32_t some, uint32_t most, int lane) {
  const uint32_t any = __ballot_sync(0xffffffffu, some != 0), big = __ballot_sync(0xffffffffu, most != 0), row = 0xffu << (lane & 24);
  return (any & row) != 0 && (big & row) == 0;
}

__device__ __forceinline__ void zero8(float* to) {
  if ((reinterpret_cast<uint64_t>(to) & 31) == 0) {
    asm volatile("st.global.v8.f32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"l"(to), "f"(0.f) : "memory");
  } else {
    *reinterpret_cast<float4*>(to) = make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(to + 4) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}
__device__ __forceinline__ void tma_box4(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tmem_st1(uint32_t addr, uint32_t v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(addr), "r"(v) : "memory");
}

// Splits K and V, 64 rows of a head a block: a thread has 8 columns of two key rows and two value rows.  Positions that no query
// sees are zeros, see gather.cu.  Bound by HBM: 4 bytes an element read, 6 written.
__global__ void __launch_bounds__(256) split_kv_kernel(const __grid_constant__ AttnParams p, uint8_t* k_out, uint8_t* v_out,
                                                       uint8_t* k_far, uint8_t* v_far, bool token_order) {
  grid_wait();
  grid_go();
  const PlanDev& pl = p.plan;
  const int g = blockIdx.y, b = blockIdx.z, P = pl.n_kv_shards;
  const int map = pl.n_maps == 1 ? 0 : b;
  const int c8 = threadIdx.x & 7, r0 = blockIdx.x * 64 + (threadIdx.x >> 3);
  const float* kb = static_cast<const float*>(p.k) + (int64_t)b * p.ks.batch + (int64_t)g * p.ks.head + c8 * 8;
  const float* vb = static_cast<const float*>(p.v) + (int64_t)b * p.vs.batch + (int64_t)g * p.vs.head + c8 * 8;
  const int32_t* last_vis =  // of the last query row: the longest prefixes
      pl.vis + ((size_t)map * pl.n_q + CASCADE_CHECKED((int64_t)__ldg(pl.q_inv + (size_t)map * pl.n_q + pl.n_q - 1), pl.n_q, pl.status, 112)) * P;
  float4 x[2][4];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int r = r0 + 32 * j;
#pragma unroll
    for (int e = 0; e < 4; ++e) x[j][e] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r >= pl.n_kv) continue;
    const int other = __ldg((token_order ? pl.kv_inv : pl.kv_idx) + (size_t)map * pl.n_kv + r);
    const int slot = (int)CASCADE_CHECKED((int64_t)(token_order ? other : r), pl.n_kv, pl.status, 113);
    const int64_t tok = CASCADE_CHECKED((int64_t)(token_order ? r : other), pl.n_kv, pl.status, 114);
    const int kk = (int)CASCADE_CHECKED((int64_t)__ldg(pl.kv_slot_shard + (size_t)map * pl.n_kv + slot), P, pl.status, 115);
    if (slot - __ldg(pl.kv_off + (size_t)map * (P + 1) + kk) >= __ldg(last_vis + kk)) continue;
    x[j][0] = __ldcs(reinterpret_cast<const float4*>(kb + tok * p.ks.token));
    x[j][1] = __ldcs(reinterpret_cast<const float4*>(kb + tok * p.ks.token) + 1);
    x[j][2] = __ldcs(reinterpret_cast<const float4*>(vb + tok * p.vs.token));
    x[j][3] = __ldcs(reinterpret_cast<const float4*>(vb + tok * p.vs.token) + 1);
  }
  const int64_t mat = (int64_t)b * p.Hkv + g, part_bytes = (int64_t)p.batch * p.Hkv * pl.n_kv * 128;
  uint64_t far[2] = {pack2(0.f, 0.f), pack2(0.f, 0.f)};
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool small_k = false;
  uint32_t some_v = 0, most_v = 0;  // a bit for each column of this thread
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int r = r0 + 32 * j;
    uint32_t some = 0, most = 0;
    note_size(x[j][0], x[j][1], some, most);
    note_size(x[j][2], x[j][3], some_v, most_v);
    small_k |= is_small_row(some, most, lane);
    if (r >= pl.n_kv) continue;
    const int64_t at = (mat * pl.n_kv + r) * 128 + c8 * 16;
    store_split8(k_out + at, part_bytes, x[j][0], x[j][1], far[0]);
    store_split8(v_out + at, part_bytes, x[j][2], x[j][3], far[1]);
  }
  __shared__ uint32_t s_size[8][4];  // of the warp's rows: columns 0 to 31 and 32 to 63 that are not zero, and that reach 2^-100
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const uint32_t bits = __reduce_or_sync(0xffffffffu, (c8 >> 2) == (w & 1) ? (w < 2 ? some_v : most_v) << 8 * (c8 & 3) : 0u);
    if (lane == 0) s_size[warp][w] = bits;
  }
  const int any_k = __syncthreads_or(is_big(far[0]) || small_k);
  uint32_t size[4] = {0, 0, 0, 0};
  if (warp == 0)
    for (int w = 0; w < 8; ++w)
      for (int i = 0; i < 4; ++i) size[i] |= s_size[w][i];
  const int any_v = __syncthreads_or(is_big(far[1]) || (size[0] & ~size[2]) || (size[1] & ~size[3]));
  if (threadIdx.x == 0) {
    k_far[mat * gridDim.x + blockIdx.x] = any_k != 0;
    v_far[mat * gridDim.x + blockIdx.x] = any_v != 0;
  }
}

// The split keys and values, [3 parts][batch * KV heads][n_kv rows][64] bf16: a box is 64 rows of all parts.  far: for every 64
// rows of a head whether one of them is out of range.
struct SplitArgs {
  CUtensorMap k, v;
  const uint8_t *k_far, *v_far;
};

// The tiles of a CTA: up to 64 keys of one KV shard (kParts), or of the sequence.
struct TileSeq {
  const volatile int32_t* need;
  int n_parts, k, t0, n;
  __device__ __forceinline__ TileSeq(const volatile int32_t* longest, int parts) : need(longest), n_parts(parts), k(0), t0(-kN) {}
  __device__ __forceinline__ bool next() {
    t0 += kN;
    while (k < n_parts && t0 >= need[k]) {
      ++k;
      t0 = 0;
    }
    if (k >= n_parts) return false;
    n = min(kN, need[k] - t0);
    return true;
  }
};

template <bool kParts>
__global__ void __launch_bounds__(kThreads, 1) attn_split_kernel(const __grid_constant__ AttnParams p, int lg, int tile_major,
                                                                 const __grid_constant__ SplitArgs sp) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  auto bar = [&](int i) { return smem_base + (uint32_t)(kOffBar + 8 * i); };
  auto longest = [&](int s) { return reinterpret_cast<volatile int32_t*>(smem + kOffTab) + s * kMaxShards; };
  auto shortest = [&](int s) { return longest(2 + s); };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  const PlanDev& pl = p.plan;
  const int P = pl.n_kv_shards, n_parts = kParts ? P : 1;
  const int Gp = 1 << lg, R = kM >> lg, n_hg = p.H >> lg, n_qt = (pl.n_q + 2 * R - 1) / (2 * R);
  int tile, hg, b;  // with few CTAs per SM the longest first, otherwise one head's after another, see attn_tc.cu
  if (tile_major) {
    const int per_tile = n_hg * p.batch, rem = blockIdx.x % per_tile;
    tile = blockIdx.x / per_tile;
    hg = rem % n_hg;
    b = rem / n_hg;
  } else {
    tile = blockIdx.x % n_qt;
    hg = (blockIdx.x / n_qt) % n_hg;
    b = blockIdx.x / n_qt / n_hg;
  }
  const int map = pl.n_maps == 1 ? 0 : b, h0 = hg * Gp, g = h0 / p.G;
  const int tok0 = (n_qt - 1 - tile) * 2 * R, n_sub = pl.n_q - tok0 > R ? 2 : 1;
  auto n_tok = [&](int s) { return min(R, pl.n_q - tok0 - s * R); };
  const int32_t* q_inv = pl.q_inv + (size_t)map * pl.n_q;
  const int32_t* kv_idx = pl.kv_idx + (size_t)map * pl.n_kv;
  const int32_t* kv_off = pl.kv_off + (size_t)map * (P + 1);
  const int32_t* vis = pl.vis + (size_t)map * pl.n_q * P;
  auto vis_row = [&](int token) {
    return vis + (size_t)CASCADE_CHECKED((int64_t)__ldg(q_inv + token), pl.n_q, pl.status, 110) * P;
  };
  grid_go();
  const float* qb = static_cast<const float*>(p.q) + (int64_t)b * p.qs.batch + (int64_t)tok0 * p.qs.token + (int64_t)h0 * p.qs.head;
  // MMA row r of sub-tile s = (token r / Gp, head r % Gp); rows past the end repeat the last token, their results are discarded
  auto q_row = [&](int s, int r) {
    return qb + (int64_t)(s * R + min(r >> lg, n_tok(s) - 1)) * p.qs.token + (int64_t)(r & (Gp - 1)) * p.qs.head;
  };
  // The query rows are on their way during the set-up; eight threads a row, 32 rows at a time.
  float4 qu[4], qv[4];
  if (warp < 8 * n_sub) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4* src = reinterpret_cast<const float4*>(q_row(warp >> 3, ((tid & 255) >> 3) + 32 * j)) + 2 * (tid & 7);
      qu[j] = __ldg(src);
      qv[j] = __ldg(src + 1);
    }
  }

  int* const any_far = reinterpret_cast<int*>(smem + kOffFar);
  auto far_kinds = [&]() { return *const_cast<volatile int*>(any_far); };
  auto far_rows = [&](int is_v) { return reinterpret_cast<volatile uint32_t*>(smem + kOffFarRows) + is_v * kFarWords; };
  const int blocks = (pl.n_kv + 63) / 64, far_shift = max(0, 32 - __clz((blocks - 1) / (32 * kFarWords)));
  // [0], [1]: tile of either stage: keys, + 256 if sub-tile 0 sees any of them (sub-tile 1 sees all that there are); [2]: tiles
  volatile int* const tile_info = reinterpret_cast<volatile int*>(smem + kOffInfo);
  WaitCtx<false, kWarps> wc;
  wc.misc = smem_base + (uint32_t)kOffMisc;
  wc.status = pl.status;
  if (warp == 16) {
    if (lane == 0) {
      mbar_init(bar(DONE), 1);
      for (int i = 0; i < 2; ++i) {
        mbar_init(bar(Q_FULL + i), 2 * kM);
        mbar_init(bar(K_FULL + i), 2);  // the bytes, and the flags
        mbar_init(bar(K_EMPTY + i), 1);
        mbar_init(bar(V_FULL + i), 2);
        mbar_init(bar(V_EMPTY + i), 1);
        mbar_init(bar(S_FULL + i), 1);
        mbar_init(bar(P_FULL + i), 2 * kM);
        mbar_init(bar(O_FULL + i), 1);
      }
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      // once a wait has given up, later calls on the plan write nothing: the abort flag is raised from the start
      int32_t gave_up;
      asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(gave_up) : "l"(pl.status) : "memory");
      wc.store(1, gave_up != 0);
      for (int w = 0; w < kWarps; ++w) wc.store(2 + w, 0);
      *any_far = 0;
    }
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_base + (uint32_t)kOffMisc),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (warp < 4) {  // prefixes of a sub-tile's last token (longest) and of its first (shortest)
    const int s = warp & 1;
    if (s < n_sub) {
      const int32_t* row = vis_row(tok0 + s * R + (warp < 2 ? n_tok(s) - 1 : 0));
      volatile int32_t* tab = warp < 2 ? longest(s) : shortest(s);
      int sum = 0, tiles = 0;
      for (int k = lane; k < P; k += 32) {
        const int n = __ldg(row + k);
        if (kParts) tab[k] = n;
        sum += n;
        tiles += (n + kN - 1) / kN;
      }
      sum = __reduce_add_sync(0xffffffffu, sum);
      tiles = kParts ? __reduce_add_sync(0xffffffffu, tiles) : (sum + kN - 1) / kN;
      if (!kParts && lane == 0) tab[0] = sum;
      if (warp == n_sub - 1 && lane == 0) tile_info[2] = tiles;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  auto note = [&](int v) {
    if (lane == 0) wc.note(warp, v);
  };
  auto landed = [&](uint32_t full, uint32_t parity) {  // what is under way, whatever the abort flag says
    for (int i = 0; i < 1 << 14 && !mbar_try_wait(full, parity); ++i) {
    }
  };
  // K/V row of key x of tile (k, t0)
  auto kv_row = [&](int k, int t0, int x) {
    if constexpr (!kParts) return (int64_t)(t0 + x);
    else return (int64_t)CASCADE_CHECKED((int64_t)__ldg(kv_idx + __ldg(kv_off + k) + t0 + x), pl.n_kv, pl.status, 111);
  };
  const float* kb = static_cast<const float*>(p.k) + (int64_t)b * p.ks.batch + (int64_t)g * p.ks.head;
  const float* vb = static_cast<const float*>(p.v) + (int64_t)b * p.vs.batch + (int64_t)g * p.vs.head;

  if (warp < 16) {
    // ------------------------------------------------------------------ query rows, softmax, output
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    const int s = warp >> 3, half = (warp >> 2) & 1, m = tid & 127;  // sub-tile, keys and columns 32 * half .., MMA row
    if (s < n_sub) {
      uint64_t big = pack2(0.f, 0.f);
      bool small = false;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int r = ((tid & 255) >> 3) + 32 * j;
        uint32_t some = 0, most = 0;
        note_size(qu[j], qv[j], some, most);
        small |= is_small_row(some, most, lane);
        store_split8(smem + kOffQ + s * kQTile + r * 128 + (((tid & 7) ^ (r & 7)) << 4), kQPart, qu[j], qv[j], big);
      }
      if (is_big(big) || small) atomicOr(any_far, kFarQ);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> tensor-core reads
      mbar_arrive(bar(Q_FULL + s));

      const bool row_ok = (m >> lg) < n_tok(s);
      const int token = tok0 + s * R + min(m >> lg, n_tok(s) - 1), head = h0 + (m & (Gp - 1));
      const int32_t* my_vis = vis_row(token);
      const int64_t slot = (my_vis - vis) / P;
      int seen_all = 0;  // keys of the sequence that this row sees
      if constexpr (!kParts)
#pragma unroll 8
        for (int k = 0; k < P; ++k) seen_all += __ldg(my_vis + k);
      const uint32_t s_addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)s * kSubCols, o_addr = s_addr + kOCol;
      const float cs = p.scale * 1.4426950408889634f;  // raw logits -> log2 units
      const uint64_t cs2 = pack2(cs, cs);
      constexpr int kCols = 32;  // keys of a tile and output columns of this thread
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
      float m_run = -INFINITY;           // raw logits; of the shard whose tiles are under way
      uint64_t l_run[2] = {0ull, 0ull};  // this thread's keys, in four sums, whose roundings average out
      auto both = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + s) : "memory"); };  // the threads of the sub-tile
      volatile float* const max_mine = reinterpret_cast<volatile float*>(smem + kOffMax) + (2 * s + half) * kM + m;
      const int to_other = half ? -kM : kM;

      // The thread's columns of its row, 32 bytes at a time (whole 64-byte pieces of rows through shared memory were slower).
      auto store_row = [&](const float* x, float inv, float* dst) {
        if (!dst) return;
        if ((reinterpret_cast<uint64_t>(dst) & 31) == 0) {
#pragma unroll
          for (int j = 0; j < kCols; j += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + j), "f"(x[j] * inv), "f"(x[j + 1] * inv),
                         "f"(x[j + 2] * inv), "f"(x[j + 3] * inv), "f"(x[j + 4] * inv), "f"(x[j + 5] * inv), "f"(x[j + 6] * inv),
                         "f"(x[j + 7] * inv)
                         : "memory");
        } else {
#pragma unroll
          for (int j = 0; j < kCols; j += 4)
            *reinterpret_cast<float4*>(dst + j) = make_float4(x[j] * inv, x[j + 1] * inv, x[j + 2] * inv, x[j + 3] * inv);
        }
      };
      auto out_row = [&](int k) -> float* {  // of shard k (kParts), or the finished row
        if (!row_ok || wc.load(1)) return nullptr;
        if constexpr (kParts)
          return static_cast<float*>(p.o_part) + ((((int64_t)b * P + k) * pl.n_q + slot) * p.H + head) * kD + kCols * half;
        else
          return static_cast<float*>(p.o_out) + (int64_t)b * p.os.batch + (int64_t)token * p.os.token + (int64_t)head * p.os.head +
                 kCols * half;
      };
      auto put_stats = [&](int k, float m_raw, float l) {
        if (!row_ok || half || wc.load(1)) return;
        if constexpr (kParts) {
          const int64_t at = (((int64_t)b * P + k) * pl.n_q + slot) * p.H + head;
          p.m_part[at] = l > 0.f ? m_raw * p.scale : -INFINITY;
          p.l_part[at] = l;
        } else if (p.lse_out) {
          p.lse_out[((int64_t)b * pl.n_q + token) * p.H + head] = l > 0.f ? m_raw * p.scale + logf(l) : -INFINITY;
        }
      };
      auto seen_of = [&](int k, int t0, int n) { return min(n, (kParts ? __ldg(my_vis + k) : seen_all) - t0); };
      // whether a key (is_v: value) row that the products of tile (k, t0) read is out of range
      auto far_tile = [&](int is_v, int k, int t0, int n) {
        const int row = (kParts ? __ldg(kv_off + k) : 0) + t0, last = min(row + (n + 15) / 16 * 16, pl.n_kv) - 1;
        const int b0 = row / 64 >> far_shift, b1 = last / 64 >> far_shift;
        return (((far_rows(is_v)[b0 / 32] >> (b0 & 31)) | (far_rows(is_v)[b1 / 32] >> (b1 & 31))) & 1u) != 0;
      };
      auto slow_dot = [&](int k, int t0, int x) {  // the logit of key x of tile (k, t0) in plain fp32
        const float4 *q4 = reinterpret_cast<const float4*>(q_row(s, m)), *k4 = reinterpret_cast<const float4*>(kb + kv_row(k, t0, x) * p.ks.token);
        float4 dot = make_float4(0.f, 0.f, 0.f, 0.f);  // in four sums, whose roundings average out
#pragma unroll 1
        for (int c = 0; c < kD / 4; ++c) {
          const float4 a = __ldg(q4 + c), d = __ldg(k4 + c);
          dot = make_float4(fmaf(a.x, d.x, dot.x), fmaf(a.y, d.y, dot.y), fmaf(a.z, d.z, dot.z), fmaf(a.w, d.w, dot.w));
        }
        return (dot.x + dot.y) + (dot.z + dot.w);
      };
      // The output of tile (k, t0): added to what the shard's earlier tiles gave, scaled by alpha, and written if it is the shard's last.
      auto fold = [&](int k, int t0, int n, int i, float alpha) {
        wait_bar(wc, bar(O_FULL + s), (uint32_t)(i & 1), 3, i);
        tc_fence_after();
        const bool opens = t0 == 0, closes = t0 + kN >= longest(s)[k];
        uint32_t o[kCols];
        auto products = [&]() {
          CASCADE_TMEM_LD32(o_addr + (uint32_t)(kCols * half), o, 0);
          tmem_wait_ld();
        };
        if (kParts) products();  // (in front 228.4 -> 221.2 us at 16 x 512 tokens, 8 shards; fused 147.7, in front 151.2)
        if (__any_sync(0xffffffffu, (far_kinds() & kFarV) && far_tile(1, k, t0, n))) {
          const int seen = seen_of(k, t0, n);
          const float m_use = m_run == -INFINITY ? 0.f : m_run;
#pragma unroll
          for (int c = 0; c < kCols; ++c) o[c] = 0u;
#pragma unroll 1
          for (int x = 0; x < seen; ++x) {  // (the weights themselves are gone by now)
            const float w = ex2((slow_dot(k, t0, x) - m_use) * cs);
            const float4* v4 = reinterpret_cast<const float4*>(vb + kv_row(k, t0, x) * p.vs.token + kCols * half);
#pragma unroll
            for (int c = 0; c < kCols; c += 4) {
              const float4 v = __ldg(v4 + c / 4);
              o[c] = __float_as_uint(fmaf(w, v.x, __uint_as_float(o[c])));
              o[c + 1] = __float_as_uint(fmaf(w, v.y, __uint_as_float(o[c + 1])));
              o[c + 2] = __float_as_uint(fmaf(w, v.z, __uint_as_float(o[c + 2])));
              o[c + 3] = __float_as_uint(fmaf(w, v.w, __uint_as_float(o[c + 3])));
            }
          }
          __syncwarp();
        } else if (!kParts) {
          products();
        }
#pragma unroll
        for (int j = 0; j < kCols; ++j) acc[j] = opens ? __uint_as_float(o[j]) : fmaf(acc[j], alpha, __uint_as_float(o[j]));
        if (closes) {
          float lo, hi;
          unpack2(fadd2(l_run[0], l_run[1]), lo, hi);
          max_mine[8 * kM] = lo + hi;
          both();
          const float l = lo + hi + max_mine[8 * kM + to_other];
          put_stats(k, m_run, l);
          store_row(acc, l > 0.f ? 1.f / l : 0.f, out_row(k));
        }
      };

      float alpha = 0.f;
      int i = 0, prev_k = 0, prev_t0 = 0, prev_n = 0;  // tiles of this sub-tile so far, and the latest of them
      TileSeq seq(longest(s), n_parts);
      while (seq.next()) {
        if (i > 0) fold(prev_k, prev_t0, prev_n, i - 1, alpha);
        const int n = seq.n;
        const int seen = seen_of(seq.k, seq.t0, n);  // (ahead of the wait, which hides the load)
        wait_bar(wc, bar(S_FULL + s), (uint32_t)(i & 1), 1, i);
        tc_fence_after();
        const int far = far_kinds();
        if (__any_sync(0xffffffffu, (far & (kFarQ | kFarK)) && ((far & kFarQ) || far_tile(0, seq.k, seq.t0, n)))) {
#pragma unroll 1
          for (int x = kCols * half; x < min(n, kCols * half + kCols); ++x) {
            const float dot = slow_dot(seq.k, seq.t0, x);
            __syncwarp();
            tmem_st1(s_addr + (uint32_t)x, __float_as_uint(dot));
            tmem_st1(s_addr + 64 + (uint32_t)x, 0u);
            tmem_st1(s_addr + 128 + (uint32_t)x, 0u);
          }
          tmem_wait_st();
        }
        uint32_t sr[kCols];
        {
          uint32_t s1[kCols], s2[kCols];  // (what the tile does not have is masked)
          CASCADE_TMEM_LD32(s_addr + (uint32_t)(128 + kCols * half), s2, 0);
          CASCADE_TMEM_LD32(s_addr + (uint32_t)(64 + kCols * half), s1, 0);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < kCols; ++j) s1[j] = __float_as_uint(__uint_as_float(s1[j]) + __uint_as_float(s2[j]));
          CASCADE_TMEM_LD32(s_addr + (uint32_t)(kCols * half), sr, 0);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < kCols; ++j) sr[j] = __float_as_uint(__uint_as_float(sr[j]) + __uint_as_float(s1[j]));
        }
        tc_fence_before();  // the weights go over the logits when both halves have theirs: after the barrier below
        if (n < kN || seq.t0 + kN > shortest(s)[seq.k]) {  // warp-uniform
          const int lc = seen - kCols * half;
          const uint32_t mk = lc >= 32 ? 0xffffffffu : (lc <= 0 ? 0u : ((1u << lc) - 1u));
#pragma unroll
          for (int j = 0; j < kCols; ++j)
            if (!((mk >> j) & 1u)) sr[j] = 0xff800000u;  // -inf
        }
        if (seq.t0 == 0) {
          m_run = -INFINITY;
          l_run[0] = l_run[1] = 0ull;
        }
        float mx[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          mx[c] = __uint_as_float(sr[16 * c]);
#pragma unroll
          for (int j = 1; j < 15; j += 2) mx[c] = fmax3(mx[c], __uint_as_float(sr[16 * c + j]), __uint_as_float(sr[16 * c + j + 1]));
          mx[c] = fmaxf(mx[c], __uint_as_float(sr[16 * c + 15]));
        }
        mx[0] = fmaxf(mx[0], mx[1]);
        max_mine[4 * kM * (i & 1)] = mx[0];
        both();
        tc_fence_after();
        const float m_new = fmaxf(m_run, fmaxf(mx[0], max_mine[4 * kM * (i & 1) + to_other]));
        const float m_use = m_new == -INFINITY ? 0.f : m_new;
        alpha = ex2((m_run - m_use) * cs);  // 0 on the first visible tile
        m_run = m_new;
        const uint64_t neg = pack2(-m_use, -m_use);
        uint64_t sum[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) sum[c] = pack2(0.f, 0.f);
        uint32_t w0[16], w1[16], w2[16];
#pragma unroll
        for (int j = 0; j < kCols; j += 2) {
          float x0, x1;
          unpack2(fmul2(fadd2(pack2(__uint_as_float(sr[j]), __uint_as_float(sr[j + 1])), neg), cs2), x0, x1);
          x0 = ex2(x0);
          x1 = ex2(x1);
          sum[(j >> 1) & 3] = fadd2(sum[(j >> 1) & 3], pack2(x0, x1));
          split2(x0, x1, w0[j >> 1], w1[j >> 1], w2[j >> 1]);
        }
        CASCADE_TMEM_ST16(s_addr + (uint32_t)(16 * half), w0);
        CASCADE_TMEM_ST16(s_addr + (uint32_t)(32 + 16 * half), w1);
        CASCADE_TMEM_ST16(s_addr + (uint32_t)(64 + 16 * half), w2);
        const uint64_t alpha2 = pack2(alpha, alpha);
        l_run[0] = ffma2(l_run[0], alpha2, fadd2(sum[0], sum[1]));
        l_run[1] = ffma2(l_run[1], alpha2, fadd2(sum[2], sum[3]));
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar(P_FULL + s));
        prev_k = seq.k;
        prev_t0 = seq.t0;
        prev_n = n;
        ++i;
      }
      if (i > 0) fold(prev_k, prev_t0, prev_n, i - 1, alpha);
      // what no row of the sub-tile sees anything of was never walked (32 bytes a store, as store_row: 4 x 1000 causal tokens in 16
      // shards of blocks of 64, 12 heads, 169 -> 127 us)
#pragma unroll 1
      for (int k = 0; k < n_parts; ++k) {
        if (longest(s)[k] > 0) continue;
        put_stats(k, -INFINITY, 0.f);
        float* dst = out_row(k);
        if (!dst) continue;
#pragma unroll 1
        for (int c = 0; c < kCols; c += 8) zero8(dst + c);
      }
      tc_fence_before();
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == 16) {
      // ---------------------------------------------------------------- products, all from one thread
      const int n_tiles = tile_info[2];
      if (elect_one() && n_tiles > 0) {
        constexpr uint32_t hi = desc_hi(1024), idesc_pv = make_idesc(kM, kD, 0, 1), next_stage = kKvTile >> 4;
        const uint32_t q_lo = desc_lo(smem_base + kOffQ, 16), k_lo = desc_lo(smem_base + kOffK, 16);
        const uint32_t v_lo = desc_lo(smem_base + kOffV, kKvPart);
        auto issue_qk = [&](int s, int i) {
          const uint32_t a = q_lo + (uint32_t)(s * (kQTile >> 4)), b = k_lo + (uint32_t)(i & 1) * next_stage, d = tmem + (uint32_t)s * kSubCols;
          // part qp of Q with parts kp .. kp + n - 1 of K, 16 columns of head_dim from 16 ks on, to columns 64 to ..
          auto mul = [&](int qp, int kp, int n, int ks, int to, bool add) {
            mma_ss(d + (uint32_t)(to * kN), a + (uint32_t)((qp * kQPart + ks * 32) >> 4), b + (uint32_t)((kp * kKvPart + ks * 32) >> 4), hi,
                   make_idesc(kM, n * kN, 0, 0), add);
          };
#pragma unroll
          for (int x = 0; x < 3; ++x)
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) mul(x, 0, 3 - x, ks, x, x + ks > 0);
#pragma unroll
          for (int ks = 2; ks < 4; ++ks) {
            mul(0, 2, 1, ks, 2, true);
            mul(1, 0, 1, ks, 2, true);
            mul(1, 1, 1, ks, 2, true);
            mul(2, 0, 1, ks, 2, true);
          }
#pragma unroll
          for (int ks = 2; ks < 4; ++ks) mul(0, 0, 2, ks, 1, true);
          mma_commit(bar(S_FULL + s));
        };
        auto issue_pv = [&](int s, int i, int n) {
          // parts of the weights and the values, smallest products first
          constexpr int kA[6] = {0, 2, 1, 0, 1, 0}, kB[6] = {2, 0, 1, 1, 0, 0};
          const uint32_t b = v_lo + (uint32_t)(i & 1) * next_stage, d = tmem + (uint32_t)s * kSubCols;
#pragma unroll
          for (int x = 0; x < 6; ++x)
#pragma unroll
            for (int ks = 0; ks < kN / 16; ++ks)
              if (16 * ks < n)
                mma_ts(d + kOCol, d + (uint32_t)(32 * kA[x] + 8 * ks), b + (uint32_t)((kB[x] * kKvPart + ks * 2048) >> 4), hi, idesc_pv,
                       x + ks > 0);
          mma_commit(bar(O_FULL + s));
        };
        uint32_t done0 = 0;  // tiles of sub-tile 0 that are finished (the other one sees them all)
        // When a wait has given up, no stage is given back that may not be full (the loader would have a second load counted on its
        // barrier while the first is under way), and the loop ends.
        bool fed = wait_bar(wc, bar(K_FULL), 0u, 7);
        int info = tile_info[0];
        wait_bar(wc, bar(Q_FULL), 0u, 6);
        if (n_sub == 2) wait_bar(wc, bar(Q_FULL + 1), 0u, 6);
        tc_fence_after();
        if (info & 256) issue_qk(0, 0);
        if (n_sub == 2) issue_qk(1, 0);
        if (fed) mma_commit(bar(K_EMPTY));
        for (int i = 0; i < n_tiles && fed && !wc.load(1); ++i) {
          const bool more = i + 1 < n_tiles;
          int next = 0;
          fed = wait_bar(wc, bar(V_FULL + (i & 1)), (uint32_t)((i >> 1) & 1), 4, i);
          if (info & 256) {
            wait_bar(wc, bar(P_FULL), done0 & 1, 5, i);
            tc_fence_after();
            issue_pv(0, i, info & 255);
            ++done0;
          }
          if (n_sub == 1 && fed) mma_commit(bar(V_EMPTY + (i & 1)));
          if (more) {
            fed = wait_bar(wc, bar(K_FULL + ((i + 1) & 1)), (uint32_t)(((i + 1) >> 1) & 1), 7, i) && fed;
            next = tile_info[(i + 1) & 1];
            if (next & 256) issue_qk(0, i + 1);
            if (n_sub == 1 && fed) mma_commit(bar(K_EMPTY + ((i + 1) & 1)));
          }
          if (n_sub == 2) {
            wait_bar(wc, bar(P_FULL + 1), (uint32_t)(i & 1), 5, i);
            tc_fence_after();
            issue_pv(1, i, info & 255);
            if (fed) mma_commit(bar(V_EMPTY + (i & 1)));
            if (more) {
              issue_qk(1, i + 1);
              if (fed) mma_commit(bar(K_EMPTY + ((i + 1) & 1)));
            }
          }
          info = next;
        }
        mma_commit(bar(DONE));
        landed(bar(DONE), 0u);
      }
      __syncwarp();
    } else if (warp < 19) {
      // ---------------------------------------------------------------- loads of the split rows
      const bool is_v = warp == 18, leader = elect_one();
      const int full = is_v ? V_FULL : K_FULL, empty = is_v ? V_EMPTY : K_EMPTY;
      const uint32_t to = smem_base + (uint32_t)(is_v ? kOffV : kOffK);
      grid_wait();  // the copies are written by the grid in front
      // The rows out of range, for the softmax threads: all of them before the first tile, so that which tiles are worked out in plain
      // fp32 depends on the rows alone and not on how far ahead this warp is.
      auto note_far = [&]() {
        volatile uint32_t* bits = far_rows(is_v);
        for (int w = lane; w < kFarWords; w += 32) bits[w] = 0u;
        __syncwarp();
        const volatile uint8_t* flags = (is_v ? sp.v_far : sp.k_far) + ((int64_t)b * p.Hkv + g) * blocks;
#pragma unroll 4
        for (int x = lane; x < blocks; x += 32)
          if (flags[x]) {
            atomicOr(const_cast<uint32_t*>(bits) + (x >> far_shift) / 32, 1u << ((x >> far_shift) & 31));
            atomicOr(any_far, is_v ? kFarV : kFarK);
          }
        __syncwarp();
      };
      TileSeq seq(longest(n_sub - 1), n_parts);  // the later sub-tile sees all that the earlier one does
      int i = 0;
      for (; seq.next(); ++i) {
        note(8 * i + 1);
        if (i >= 2 && !wait_bar(wc, bar(empty + (i & 1)), (uint32_t)(((i >> 1) & 1) ^ 1), 9 + is_v, i)) break;
        if (leader) {
          if (!is_v) tile_info[i & 1] = seq.n + (seq.t0 < longest(0)[seq.k] ? 256 : 0);
          mbar_expect_tx(bar(full + (i & 1)), kKvTile);
          const int row = (kParts ? __ldg(kv_off + seq.k) : 0) + seq.t0;  // first row of the tile in the split copies
          tma_box4(to + (uint32_t)((i & 1) * kKvTile), is_v ? &sp.v : &sp.k, 0, row, b * p.Hkv + g, 0, bar(full + (i & 1)));
        }
        if (i == 0) note_far();  // (while the box is on its way)
        if (leader) mbar_arrive(bar(full + (i & 1)));
        __syncwarp();
      }
      if (wc.load(1))
        for (int j = max(0, i - 2); j < i; ++j) landed(bar(full + (j & 1)), (uint32_t)((j >> 1) & 1));
    }
  }
  grid_wait();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace split

namespace {
int split_stacked_log2(int G) {  // heads per tile, as in attn_tc.cu
  int lg = 0;
  while (lg < 3 && G % (2 << lg) == 0) ++lg;
  return lg;
}

// [3 parts][batch * KV heads][rows][64] bf16; box = 64 rows of all parts
bool encode_split(CUtensorMap* map, void* base, int64_t rows, int64_t mats) {
  const cuuint64_t dims[4] = {64, (cuuint64_t)rows, (cuuint64_t)mats, 3};
  const cuuint64_t strides[3] = {128, (cuuint64_t)rows * 128, (cuuint64_t)(rows * mats) * 128};
  const cuuint32_t box[4] = {64, 64, 1, 3}, estr[4] = {1, 1, 1, 1};
  EncodeTiledFn fn = encode_tiled_fn();
  return fn && fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

// Estimated time in us, see rows_time: the copies, and CTAs one per SM.  A CTA takes 5 us, 2.1 or 2.6 us a tile with one or two
// sub-tiles (2.2 or 3.2 with every SM busy), and more for every shard that it writes out.  At 300 random sizes (2 to 1500 tokens, 2 to
// 128 (head, sequence) pairs, 1 to 32 shards, both routes) within -3 and +27 % of what was measured in eight of ten.
double split_time(const AttnParams& p) {
  const CutSize c(p);
  const int lg = split_stacked_log2(p.G);
  const double pairs = std::ceil(c.n_q / (256 >> lg)), ctas = pairs * c.heads / (1 << lg);
  const bool two = p.plan.n_q > (128 >> lg);
  const double parts = p.fused ? 0 : c.shards;
  auto tiles = [&](double seen) { return p.fused ? std::ceil(seen * c.n_kv / 64) : c.shards * c.pieces(seen, 64); };
  const double copy = 3 + c.heads / p.G * c.n_kv * 64 * 20 / 5.5e6;
  const double alone = 5 + (two ? 2.6 : 2.1) * tiles(c.seen_at(1.0)) + (two ? 1.3 : 0.7) * parts;
  const double cta = 5 + (two ? 3.2 : 2.2) * tiles(c.seen_at((pairs + 1) / (2 * pairs))) + (two ? 2.4 : 1.2) * parts;
  return copy + std::max(alone, std::ceil(ctas / kEstimateSms) * cta);
}

// Workspace: the split copies of K and of V, each rounded up to 256 bytes, then their flags.
size_t split_ws_bytes(const PlanDev& d, int batch, int Hkv) {
  const size_t mats = (size_t)batch * Hkv, copy = (3 * mats * d.n_kv * 128 + 255) / 256 * 256;
  return 2 * copy + (2 * mats * ((d.n_kv + 63) / 64) + 255) / 256 * 256;
}

cudaError_t launch_attn_split(const AttnParams& p, void* workspace, cudaStream_t stream) {
  const int64_t mats = (int64_t)p.batch * p.Hkv, copy = (3 * mats * p.plan.n_kv * 128 + 255) / 256 * 256;
  const int blocks = (p.plan.n_kv + 63) / 64;
  uint8_t* k = static_cast<uint8_t*>(workspace);
  uint8_t* v = k + copy;
  uint8_t* k_far = v + copy;
  uint8_t* v_far = k_far + mats * blocks;
  split::SplitArgs sp = {};
  sp.k_far = k_far;
  sp.v_far = v_far;
  if (!encode_split(&sp.k, k, p.plan.n_kv, mats) || !encode_split(&sp.v, v, p.plan.n_kv, mats)) {
    set_error("fp32 attention on the tensor cores: could not build the TMA descriptors of the split keys and values");
    return cudaErrorInvalidValue;
  }
  cudaError_t e = launch_dependent(split::split_kv_kernel, dim3(blocks, p.Hkv, p.batch), 256, 0, 1, true, stream, p, k, v, k_far, v_far,
                                   p.fused != 0);
  if (e != cudaSuccess) return e;
  auto kernel = p.fused ? split::attn_split_kernel<false> : split::attn_split_kernel<true>;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, split::kSmemBytes);
  if (e != cudaSuccess) return e;
  const int lg = split_stacked_log2(p.G), R = split::kM >> lg;
  const int64_t ctas = (int64_t)((p.plan.n_q + 2 * R - 1) / (2 * R)) * (p.H >> lg) * p.batch;
  if (ctas >= (int64_t)1 << 31) return cudaErrorInvalidConfiguration;
  TimedLaunch timed(stream);
  return launch_dependent(kernel, dim3((unsigned)ctas), split::kThreads, split::kSmemBytes, 1, true, stream, p, lg,
                          (int)(ctas <= 8 * 148), sp);
}

}  // namespace cascade
