// Attention-pass on the 5th-generation tensor cores (tcgen05 + TMEM) for bf16, head_dim 128 and 64.
//
// Work decomposition.  The M dimension of one MMA tile (128 rows) is filled with (query row, head) pairs: the
// Gp query heads that read the same KV head ("repeat_kv", the Attention-Pass algorithm) are stacked next to each other,
// so a tile covers only 128 / Gp consecutive query rows.  One CTA owns two such sub-tiles (the next 128 / Gp rows, same
// heads), which share every K/V tile.
//
// Fused route (not kWalk).  The Post-Pass algorithm makes of the partials of all KV shards exactly the softmax over all keys,
// and of those a query sees a prefix in token order.  So the CTA takes 256 / Gp consecutive tokens and walks the keys in
// token order, 128 at a time, straight from the caller's K and V; the carry n, w, o of the Post-Pass algorithm is the running
// max / sum / output of the streaming softmax, and one output row is written at the end.  Only the last tile or two need the
// causal mask.  Where there are few query tiles, a cluster of 2, 4 or 8 CTAs shares the keys of one and adds up through
// distributed shared memory.
// Measured, 32 query / 8 KV heads: 2048 tokens, 8 random shards 41.9 us; 512 queries against 7168 cached tokens 69 us; 32768
// tokens, 64 / 8 heads, 32 random shards 15.6 ms; 2 x 3001 tokens, 16 / 4 heads of 64 columns 76 us.  (This order of work alone,
// against shard by shard from gathered copies with query tiles inside one shard: 67 -> 47 us, 127 -> 80 us, 16.7 -> 16.0 ms and
// 124 -> 85 us; the rest is what stands beside the code below.)
//
// Partials (kWalk, the Attention-Pass algorithm for every pair of the query tile).  The rows are consecutive slots of one
// query shard and the KV shards are walked one after another: each shard's visible prefix (as seen by the CTA's last row,
// which has the longest one) is cut into chunks of 32 keys, and up to four chunks form one MMA tile.  A tile never mixes two
// shards: at every shard boundary that shard's (u, m, l) is written out and the statistics and the accumulator start over.
// (A CTA per (query tile, KV shard) pair would pay the CTA set-up once per pair.)
//
// Warp roles (12 warps):
//   0-3   softmax of sub-tile 0, 4-7 softmax of sub-tile 1: thread = MMA row = TMEM lane.  Reads the logits S with
//         tcgen05.ld, applies the mask (the row sees a prefix of the keys), writes the weights P as bf16 back into the TMEM
//         columns of S, keeps the running max / sum while the products run, rescales the output accumulator in TMEM in
//         the rare case that a weight is far above the reference maximum, and runs the epilogue: the scaled output
//         row goes through shared memory (the Q / K tiles are free by then), from where the warp stores whole rows.
//         kWalk writes rows out at every shard boundary, see store_rows.
//   8     MMA issuer: S_s = Q_s K^T (operands in shared memory) and O_s += P_s V (P from TMEM), issued as
//         PV_0(i), QK_0(i+1), PV_1(i), QK_1(i+1) so that the tensor pipe works on one sub-tile while the other is in
//         its softmax.  QK_s(i+1) overwrites the columns PV_s(i) reads P from; MMAs execute in issue order, which
//         makes that safe without a barrier.  The whole warp runs the loop and one elected lane issues, so that
//         descriptors and addresses stay warp-uniform.
//   9-10  loaders: TMA box loads, completion counted in bytes on an mbarrier, data written in the 128-byte-swizzled
//         layout the MMA descriptors expect.  Warp 9 streams the K tiles and warp 10 the V tiles: 128 rows at a time from
//         the caller's tensors, or with kWalk 32 at a time from the shard-major copies that the gather pass (gather.cu)
//         wrote, where the visible prefix of a shard is a contiguous run of rows.  An index-mapped gather straight from
//         the caller's tensors was far too slow for the K/V stream (measured: one 512-byte TMA row gather per ~36
//         cycles per SM; 16-byte cp.async: one 512-byte request per ~90 cycles per warp).  The two query
//         sub-tiles come once per CTA, as boxes requested during the set-up; where their tokens are not consecutive (kWalk),
//         where they are turned on the way (rotary step), or where their strides do not fit a tensor map, the softmax threads
//         gather them themselves (plain 16-byte loads).
//   11    works out the CTA's keys (kWalk: the table of the shards it sees anything of) and looks at the status word, then idles; it also keeps the
//         register-reallocation groups of four warps whole.
// The grid is launched as a programmatic dependent (partials: only after a gather).  After a gather everything up to the
// loaders' first TMA load may run while the copies are still being written; otherwise the set-up of the block scheduler
// and of the parameters overlaps the tail of whatever kernel comes before.
// Every mbarrier wait is bounded: on expiry the CTA raises a flag, records a code in the plan's status word
// and drains without waiting again.
#include <float.h>

#include <algorithm>

#include "tcgen05.cuh"

namespace cascade {
namespace tc {

constexpr int kThreads = 384;
constexpr int kM = 128;                  // MMA rows per sub-tile
constexpr int kNMax = 128;               // keys per KV tile (upper bound)
constexpr int kHalfBytes = kM * 128;     // one 64-column half of a 128-row tile: 128 rows of 128 bytes
constexpr uint32_t kTmemCols = 512;
// How far a row may rise above its reference maximum before it is rescaled: by its logits (log2 units), or, where the maximum of
// a tile comes after its weights (kLateMax), by the sum of the tile's weights.  (bf16 and fp32 keep their relative precision at
// any scale; the sums of 2^20 tiles and the products with values below 2^40 stay in range.)  With weights of 8 bits and the
// maximum at hand the bound is low: a row that a new key dominates is rescaled, so that the key's weight is 1 and exact.
constexpr float kRescaleBf16 = 8.f, kRescaleTwoParts = 60.f;
constexpr float kRescaleSum = 1.1529215e18f;  // 2^60
// setmaxnreg only redistributes the registers the CTA was launched with (168 per thread x 384 threads = 64512), and
// all four warps of an allocation group execute the same instruction: 8 warps x 32 x 216 + 4 warps x 32 x 72 = 64512.
// An increase that asks for more than the launch grant never returns.
constexpr int kRegsSoftmax = 216;
constexpr int kRegsOther = 72;
static_assert(8 * 32 * kRegsSoftmax + 4 * 32 * kRegsOther <= 168 * kThreads, "setmaxnreg would wait for registers forever");
constexpr int kChunk = 32;                // keys per chunk of the KV stream
constexpr int kChunkBytes = kChunk * 128; // one 64-column half of a chunk in a tile
constexpr int kMaxShards = 256;           // KV shards per CTA whose bookkeeping fits in shared memory
constexpr int kMaxStages = 4;

// What depends on the head_dim D.
//   D = 128: TMEM = S0 | S1 | O0 | O1, 128 columns each; the probabilities P_s overwrite the start of S_s, so the next
//            logits of a sub-tile wait for the product that reads its P.
//   D = 64:  TMEM = three logit buffers of 128 columns | O0 | O1 of 64.  The sub-tiles take turns on the three buffers
//            (sub-tile s, tile i: buffer (2 i + s) mod 3), so the next logits of a sub-tile are computed while it is still
//            in the softmax of the current tile.  P is kept to twice the precision there: a bf16 part and the bf16
//            rest, which together fill the 128 columns of the buffer they overwrite.
// kBoxes (partials, see launch_attn_tc_partials) has a staging area of its own for finished rows, which at D = 128 takes the place
// of the second K and V stages.
template <int D, bool kBoxes>
struct Cfg {
  static constexpr int kHalves = D / 64;
  static constexpr int kTileBytes = kHalves * kHalfBytes;  // [halves][128 rows][128 bytes]
  static constexpr int kKStages = D == 64 ? 4 : (kBoxes ? 1 : 2);  // (D = 128: a third stage bought nothing)
  static constexpr int kVStages = D == 64 ? 3 : (kBoxes ? 1 : 2);
  static constexpr bool kRing = D == 64;                   // three logit buffers, P in two parts
  static constexpr uint32_t kOCol = kRing ? 384u : 256u;   // first accumulator column
  // Output rows.  The last ones of a CTA are staged where Q and K were, padded by 16 bytes; with kBoxes all of them in an area
  // of their own, per warp [halves][32 rows][128 bytes], swizzled like the operand tiles.
  static constexpr int kStageWarpBytes = kHalves * 32 * 128, kRowBytes = D * 2, kStageRowBytes = kRowBytes + 16;
  static constexpr int kStageBytes = kBoxes ? 8 * kStageWarpBytes : 2 * kM * kStageRowBytes;
  // shared memory map (offsets from a 1024-byte aligned base)
  static constexpr int kOffQ = 0;
  static constexpr int kOffK = kOffQ + 2 * kTileBytes;
  static constexpr int kOffV = kOffK + kKStages * kTileBytes;
  static constexpr int kOffStage = kBoxes ? kOffV + kVStages * kTileBytes : kOffQ;
  static constexpr int kOffBar = kOffV + kVStages * kTileBytes + (kBoxes ? kStageBytes : 0);
  static_assert(kBoxes || kStageBytes <= kOffV, "the output staging area must fit in the Q and K tiles");
  static constexpr int kNumBars = 32;
  static constexpr int kOffMisc = kOffBar + kNumBars * 8;   // tmem slot, abort flag, 12 progress words
  static constexpr int kOffShard = kOffMisc + 64;           // int32 [5][kMaxShards], see ShardTab
  static constexpr int kSmemBytes = kOffShard + 5 * kMaxShards * 4 + 1024;  // + alignment slack
  static_assert(kSmemBytes <= 232448, "exceeds the 227 KiB a CTA may use");
};

enum Bar {
  Q_FULL = 0,                       // [2]
  K_FULL = 2,                       // [kKStages]
  K_EMPTY = K_FULL + kMaxStages,    // [kKStages]
  V_FULL = K_EMPTY + kMaxStages,    // [kVStages]
  V_EMPTY = V_FULL + kMaxStages,    // [kVStages]
  S_FULL = V_EMPTY + kMaxStages,    // [2]; kRing: [2][2], see s_full
  P_FULL = S_FULL + 4,              // [2]; kRing: [2][2], see p_full
  O_FULL = P_FULL + 4,              // [2] the last product of a sub-tile is in
  CHECKED = O_FULL + 2,             // [1] the plan's status word has been looked at
  O_RDY = CHECKED + 1               // [2]  kWalk: the accumulator of a sub-tile holds a finished shard;
                                    //      kRing: the product of a sub-tile's latest tile is in its accumulator
};
constexpr int kBars = O_RDY + 2;
static_assert(kBars <= Cfg<128, false>::kNumBars && kBars <= 32, "barrier table too small");

// TMA box loads, 64 elements wide: rows land as 128 bytes each.  32 rows of the 3-D tensor [matrix z][row y][column x]
// (shard-major copies), or 128 rows of the 4-D tensor [sequence w][head z][row y][column x].
__device__ __forceinline__ void tma_tile4(uint32_t dst, const CUtensorMap* map, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_tile3(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_store4(const CUtensorMap* map, int x, int y, int z, int w, uint32_t src) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4}], [%5];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z), "r"(w), "r"(src)
               : "memory");
}
// All threads of the cluster (each warp where it stands in its role).
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// 16 bytes into the shared memory of CTA `to` of the cluster, at the address `local` has in this one
__device__ __forceinline__ void st_cluster(uint32_t local, int to, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  uint32_t addr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(local), "r"(to));
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}


// Bookkeeping of the shards of which the CTA sees anything ("active" shards, in walk order), in shared memory.
struct ShardTab {
  int32_t need[kMaxShards];    // visible prefix of the CTA's last row = keys of the shard that are walked
  int32_t first[2][kMaxShards];  // visible prefix of the first row of sub-tile 0 / 1: chunks below it need no mask
  int32_t slot0[kMaxShards];   // position of the shard's first key in the shard-major K/V copies
  int32_t kk[kMaxShards];      // shard id
};
// Cursor over the chunk stream: chunk c of active shard j.
struct ChunkCursor {
  int j, c, nc;  // nc = chunks of shard j
  __device__ __forceinline__ void start(const ShardTab* t, int n_act) {
    j = 0;
    c = 0;
    nc = n_act > 0 ? (t->need[0] + kChunk - 1) / kChunk : 0;
  }
  // moves to the next chunk; returns true if that entered a new shard
  __device__ __forceinline__ bool advance(const ShardTab* t, int n_act) {
    if (++c < nc) return false;
    ++j;
    c = 0;
    nc = j < n_act ? (t->need[j] + kChunk - 1) / kChunk : 0;
    return true;
  }
};

// Chunk count and shard-start flag of consecutive tiles, for the roles that do not walk the chunks themselves.
template <bool kWalk>
struct TileSeq {
  const ShardTab* t;
  int n_act, n_keys, i, j, c, nc;
  __device__ __forceinline__ TileSeq(const ShardTab* tab, int n_active, int keys)
      : t(tab), n_act(n_active), n_keys(keys), i(0), j(0), c(0) {
    nc = (kWalk && n_act > 0) ? (t->need[0] + kChunk - 1) / kChunk : 0;
  }
  // the next tile: its chunks; first = it opens a shard (kWalk) or the whole stream
  __device__ __forceinline__ int next(bool& first) {
    if constexpr (!kWalk) {
      first = i == 0;
      const int n = min(4, (n_keys - 4 * kChunk * i + kChunk - 1) / kChunk);
      ++i;
      return n;
    } else {
      first = c == 0;
      const int n = min(4, nc - c);
      c += n;
      if (c >= nc) {
        ++j;
        c = 0;
        nc = j < n_act ? (t->need[j] + kChunk - 1) / kChunk : 0;
      }
      return n;
    }
  }
};

struct TmaArgs {
  // kWalk: the shard-major copies as [batch * kv_heads][n_kv][head_dim];
  // otherwise K and V rows in token order as [batch][kv_heads][rows that are seen][head_dim]
  CUtensorMap k, v;
  // kWalk: where finished rows go, o_part as [batch * KV shards][n_q slots][heads][head_dim]; a box is the rows of one warp:
  // 32 / Gp slots x Gp heads
  CUtensorMap o;
  int o_valid;  // 0: the threads store their rows themselves
  // Fused route without a rotary step: the query rows as [batch][tokens][heads][head_dim]; a box is one sub-tile, 128 / Gp
  // tokens x Gp heads, 64 columns
  int q_valid;  // 0: the threads load them
  CUtensorMap q;
};

// kRope: the query rows are turned by the rotary embedding of their positions while they are staged (the key rows
// were turned by the gather pass), the Pre-Pass algorithm.
// kWalk: the partials of EVERY KV shard for one query tile in one CTA (the attention-pass of the nodes AttnNode_{j,1..beta}
// one after another): the shards are walked as in the fused mode, but a tile never mixes two shards, and at a shard
// boundary the softmax threads write that shard's (u, m, l) out and start over.  The query tile, the TMEM allocation,
// the barriers and the K/V pipelines are set up once per query tile instead of once per (query tile, KV shard).
template <int D, bool kRope, bool kWalk, bool kBoxes>
__global__ void __launch_bounds__(kThreads, 1) attn_tc_kernel(const __grid_constant__ AttnParams p, int lg,
                                                              int tile_major, int lg_split, int early, int after_gather,
                                                              const __grid_constant__ TmaArgs tma) {
  using C = Cfg<D, kBoxes>;
  constexpr int kD = D, kTileBytes = C::kTileBytes, kKStages = C::kKStages, kVStages = C::kVStages;
  constexpr int kOffQ = C::kOffQ, kOffK = C::kOffK, kOffV = C::kOffV, kOffMisc = C::kOffMisc;
  constexpr bool kRing = C::kRing;
  static_assert(!kRope || D == 128, "the rotary step is fused for head_dim 128 only");
  constexpr bool kLateMax = !kWalk && !kRing;  // see below
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t bar0 = smem_base + C::kOffBar;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  // Logits of sub-tile s, tile i.  With kRing they may be two tiles ahead of a softmax thread, which a phase parity cannot
  // tell from "not there yet": even and odd tiles have a barrier each (tile i + 2 is issued after the thread's P(i)).
  auto s_full = [&](int s, int i) { return bar(S_FULL + (kRing ? 2 * (i & 1) : 0) + s); };
  // Weights of sub-tile s, tile i.  With kRing a warp can be done with tile i + 1 before another has arrived for tile i, and
  // on one barrier its arrival would complete the other's phase; it cannot get to tile i + 2 (PV(i) waits for everyone).
  auto p_full = [&](int s, int i) { return bar(P_FULL + (kRing ? 2 * (i & 1) : 0) + s); };
  auto s_parity = [&](int i) { return (uint32_t)((kRing ? i >> 1 : i) & 1); };
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  ShardTab* tab = reinterpret_cast<ShardTab*>(smem + C::kOffShard);
  volatile int* stream_info = reinterpret_cast<volatile int*>(smem + kOffMisc + 56);  // [0] active shards, [1] chunks

  // lg = log2(Gp): Gp heads stacked per tile, R = 128 / Gp slots per sub-tile, 2 R slots per CTA
  const int Gp = 1 << lg, R = kM >> lg;
  const PlanDev& pl = p.plan;
  const int P = pl.n_kv_shards;
  // Block index -> (query tile, sequence, head group).  The tiles are listed by decreasing work.  With few CTAs per SM the
  // query tile is the slowest index, so that the heaviest CTAs of all heads and sequences start first and the light ones
  // fill the tail.  For a large problem the head group is slowest instead: the CTAs running at any time then read the
  // K/V of few KV heads, which keeps that stream in L2.  (The grid has an axis for each, and what is a power of two is
  // shifted: the divisions of a flat index took 900 of the 5300 cycles before a CTA's first logits.)
  const int split = 1 << lg_split;
  const int ts = 3 - lg;  // kWalk: tile list of 2 R = 256 >> lg slots
  const int n_qt = kWalk ? pl.n_qtiles[ts] : (pl.n_q + 2 * R - 1) >> (8 - lg);
  int tile_idx, hg, b, part_of_keys = 0;  // part_of_keys: rank in the cluster that shares a query tile's keys
  if (tile_major) {
    hg = (int)blockIdx.x >> lg_split;
    part_of_keys = (int)blockIdx.x & (split - 1);
    b = blockIdx.y;
    tile_idx = blockIdx.z;
  } else {
    tile_idx = blockIdx.x;
    hg = blockIdx.y;
    b = blockIdx.z;
  }
  // A gather right before this grid runs after all that came before it, and writes only what the loaders read: they wait
  // for it.
  grid_go();
  if (!after_gather) grid_wait();
  const int map = pl.n_maps == 1 ? 0 : b;
  const int h0 = hg * Gp;  // first of the Gp stacked heads
  const int per_kv = p.G >> lg;  // head groups per KV head
  const int g = per_kv == 1 ? hg : hg / per_kv;
  int row0, nrows;         // kWalk: slots of the shard-major order; otherwise tokens
  if constexpr (kWalk) {
    const int4 qt = pl.qtiles[ts][(size_t)map * pl.n_qtiles[ts] + tile_idx];
    row0 = qt.x;
    nrows = qt.y;
    if (nrows == 0) {  // padding entry (uniform for the CTA)
      grid_wait();
      return;
    }
  } else {
    row0 = (n_qt - 1 - tile_idx) * 2 * R;
    nrows = min(2 * R, pl.n_q - row0);
  }
  const int n_sub = nrows > R ? 2 : 1;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int32_t* q_idx = pl.q_idx + (size_t)map * pl.n_q;
  const int32_t* kv_off = pl.kv_off + (size_t)map * (P + 1);
  const int32_t* vis = pl.vis + (size_t)map * pl.n_q * P;
  // Token of a row, and (not kWalk) how many K/V rows it sees: a prefix of the tensors, because the mask is causal in
  // positions and the rows ascend in position.
  auto token_of = [&](int row) {
    return kWalk ? (int)CASCADE_CHECKED((int64_t)__ldg(q_idx + row), pl.n_q, pl.status, 108) : row;
  };
  auto seen_by = [&](int token) {
    if (!pl.causal) return pl.n_kv;
    if (!p.prefix_from_vis) return (int)max((int64_t)0, min((int64_t)pl.n_kv, (int64_t)pl.q_pos_offset + token + 1));
    const int32_t* v = vis + (size_t)__ldg(pl.q_inv + (size_t)map * pl.n_q + token) * P;  // rows at positions of their own
    int n = 0;
    for (int kk = 0; kk < P; ++kk) n += __ldg(v + kk);
    return n;
  };
  // Query sub-tiles (row r = slot r / Gp, head r % Gp): the 128 softmax threads of a sub-tile gather it from the
  // caller's tensor, 16 bytes per thread and row, half a warp per 256-byte row.  The loads are issued here, before the
  // set-up below, and land in shared memory (128-byte-swizzled [2][128][128 B] layout) after it.  Rows past the end
  // of the sub-tile repeat its last row (their results are discarded).
  constexpr int kRowChunks = kD / 8;            // 16-byte pieces of a row
  constexpr int kRowsPerPass = 128 / kRowChunks;  // rows the 128 threads of a sub-tile load at a time
  uint4 qv[kRowChunks];
  const int q_chunk = tid & (kRowChunks - 1);
  const int q_row = (tid & 127) / kRowChunks;
  const float4* rope_row[kRope ? 8 : 1];  // this thread's slice of the table row of each of its query rows
  float4 cs[kRope ? 4 : 1][4];            // (cos, sin) of four rows: 8 pairs each
  const bool q_boxes = !kWalk && !kRope && tma.q_valid;
  if (!q_boxes && warp < 8 && (warp >> 2) < n_sub) {
    const int s = warp >> 2;
    const int sub_row0 = row0 + s * R;
    const int sub_nrows = min(R, nrows - s * R);
    if constexpr (kRope) {
      // Rotary staging: a thread holds both halves of 8 rotation pairs of a row (columns 8 c .. and 64 + 8 c ..),
      // 8 threads per row, 8 rows per thread, and the (cos, sin) of the first four of its rows; the table rows of the
      // other four are fetched while those are turned.
      const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(p.q) + (int64_t)b * p.qs.batch + (tid & 7) * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int r = (tid >> 3 & 15) + 16 * j;
        const int tok = token_of(sub_row0 + min(r >> lg, sub_nrows - 1));
        const __nv_bfloat16* row = qb + (int64_t)tok * p.qs.token + (int64_t)(h0 + (r & (Gp - 1))) * p.qs.head;
        qv[2 * j] = __ldg(reinterpret_cast<const uint4*>(row));
        qv[2 * j + 1] = __ldg(reinterpret_cast<const uint4*>(row + 64));
        // (a row before position 0 sees nothing, so its angle is of no account; the table starts at 0)
        rope_row[j] = reinterpret_cast<const float4*>(p.rope + (int64_t)max(0, pl.q_pos_offset + tok) * 64 + (tid & 7) * 8);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) cs[j][e] = __ldg(rope_row[j] + e);
    } else {
      const __nv_bfloat16* qb = static_cast<const __nv_bfloat16*>(p.q) + (int64_t)b * p.qs.batch + q_chunk * 8;
#pragma unroll
      for (int j = 0; j < kRowChunks; ++j) {
        const int r = q_row + kRowsPerPass * j;
        const int tok = token_of(sub_row0 + min(r >> lg, sub_nrows - 1));
        qv[j] = __ldg(reinterpret_cast<const uint4*>(qb + (int64_t)tok * p.qs.token +
                                                     (int64_t)(h0 + (r & (Gp - 1))) * p.qs.head));
      }
    }
  }
  int32_t gave_up = 0;  // warp 11: whether a wait of an earlier call on this plan gave up; used after the set-up
  if (warp == 11) {     // the warp without a role of its own
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(gave_up) : "l"(pl.status) : "memory");
    if constexpr (kWalk) {
      // Compact the shards of which the CTA's last row (longest prefix; rows ascend) sees something, with what the
      // roles need per shard, and count the tiles of the stream.
      const int32_t* need_of = vis + (size_t)(row0 + nrows - 1) * P;
      const int32_t* first0 = vis + (size_t)row0 * P;
      const int32_t* first1 = vis + (size_t)(row0 + (n_sub - 1) * R) * P;
      int n_act = 0, n_tiles = 0;
      for (int base = 0; base < P; base += 32) {
        const int kk = base + lane;
        const int nd = kk < P ? __ldg(need_of + kk) : 0;
        const uint32_t act = __ballot_sync(0xffffffffu, nd > 0);
        if (nd > 0) {
          const int pos = n_act + __popc(act & ((1u << lane) - 1u));
          tab->need[pos] = nd;
          tab->first[0][pos] = __ldg(first0 + kk);
          tab->first[1][pos] = __ldg(first1 + kk);
          tab->slot0[pos] = __ldg(kv_off + kk);
          tab->kk[pos] = kk;
        }
        n_act += __popc(act);
        n_tiles += __reduce_add_sync(0xffffffffu, (nd + 4 * kChunk - 1) / (4 * kChunk));  // a tile keeps to its shard
      }
      if (lane == 0) {
        stream_info[0] = n_act;
        stream_info[1] = n_tiles;
      }
    } else {
      // the keys the last row sees, in tiles of 128 from the first on; this CTA takes its part of the tiles
      const int seen = lane < 3 ? seen_by(lane == 0 ? row0 + nrows - 1 : row0 + (lane == 2 ? (n_sub - 1) * R : 0)) : 0;
      const int tiles = (__shfl_sync(0xffffffffu, seen, 0) + kNMax - 1) / kNMax;
      const int t0 = tiles * part_of_keys >> lg_split, t1 = tiles * (part_of_keys + 1) >> lg_split;
      if (lane == 0) {
        tab->need[0] = max(0, min(seen, t1 * kNMax) - t0 * kNMax);  // keys of this CTA's part
        tab->slot0[0] = t0 * kNMax;
        stream_info[0] = 1;
        stream_info[1] = t1 - t0;
      }
      if (lane == 1 || lane == 2) tab->first[lane - 1][0] = seen;
    }
  }
  WaitCtx<kWalk, kThreads / 32> wc;
  if constexpr (kWalk) wc.words = reinterpret_cast<volatile int*>(smem + kOffMisc);
  else wc.misc = smem_base + (uint32_t)kOffMisc;
  wc.status = pl.status;

  auto note = [&](int v) {
    if (lane == 0) wc.note(warp, v);
  };

  // Warp 9 sets the barriers up, a lane each, and has the first data on their way.  (A barrier that nobody else waits for it at, past
  // the requests, costs the softmax threads registers: partials of 4099 tokens in 16 shards 392 -> 418 us.)
  if (warp == 9) {
    if (lane < kBars) {  // one arrival, except by the threads of a sub-tile; TMA: one that announces the byte count, then the bytes
      const bool by_rows = lane < Q_FULL + 2 ? !q_boxes : lane >= P_FULL && lane < P_FULL + 4;
      mbar_init(bar(lane), by_rows ? 128u : 1u);
    }
    if (lane < kThreads / 32) wc.store(2 + lane, 0);
    if (lane == 0) wc.store(1, 0);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if constexpr (!kWalk) {
      if (lane == 0) {
        // The query rows and the first tiles of K and V (early, bit 0: K, bit 1: V; not what a gather in front of this grid
        // writes) are requested here, under the rest of the set-up.  (Query rows loaded by the softmax threads cost a CTA 2700
        // cycles before its first product: 2048 tokens 40.3 -> 38.5 us, 2 x 3001 tokens of head_dim 64 78.2 -> 76.7.)
        const int tiles = (seen_by(row0 + nrows - 1) + kNMax - 1) / kNMax;
        const int t0 = tiles * part_of_keys >> lg_split;
        if (tiles * (part_of_keys + 1) >> lg_split > t0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          auto request_q = [&](int s) {
            mbar_expect_tx(bar(Q_FULL + s), (uint32_t)kTileBytes);
            for (int half = 0; half < C::kHalves; ++half)
              tma_tile4(smem_base + (uint32_t)(kOffQ + s * kTileBytes + half * kHalfBytes), &tma.q, 64 * half, h0, row0 + s * R, b,
                        bar(Q_FULL + s));
          };
          auto request_kv = [&](const CUtensorMap* map, uint32_t dst, uint32_t fb) {
            mbar_expect_tx(fb, (uint32_t)kTileBytes);
            tma_tile4(dst, map, 0, t0 * kNMax, g, b, fb);
            if (C::kHalves == 2) tma_tile4(dst + (uint32_t)kHalfBytes, map, 64, t0 * kNMax, g, b, fb);
          };
          if (q_boxes) request_q(0);
          if (early & 1) request_kv(&tma.k, smem_base + kOffK, bar(K_FULL));
          if (q_boxes && n_sub == 2) request_q(1);
          if (early & 2) request_kv(&tma.v, smem_base + kOffV, bar(V_FULL));
        }
      }
      __syncwarp();
    }
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_base + (uint32_t)kOffMisc),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int n_act = stream_info[0];  // kWalk: shards of which the CTA sees something
  const int n_tiles = stream_info[1];
  // not kWalk: first key and number of keys of this CTA's part of the stream
  const int key0 = kWalk ? 0 : tab->slot0[0], n_keys = kWalk ? 0 : tab->need[0];
  // MMA tiles of four chunks; only the last one is narrower, or with kWalk the last one of every shard (see TileSeq)
  auto tile_chunks = [&](int i) { return min(4, (n_keys - kNMax * i + kChunk - 1) / kChunk); };

  // Once a wait has given up, later calls on the plan write nothing.  Warp 11 looks the word up during the set-up; the issuing
  // warp asks when the first logits are under way, the loaders when they have nothing left to do, and what is under way lands
  // before the CTA ends.  From then on the softmax warps find the abort flag raised.  (The load takes as long as the first data:
  // looked up by all before the set-up it costs 1000 cycles, joined to the barrier above 900, asked for before the first
  // logits 400 to 1300: 33 tokens, 64 / 8 heads, 6.7 -> 7.6 us.)
  auto goes_on = [&]() {
    wait_bar(wc, bar(CHECKED), 0u, 11);
    return wc.load(1) == 0;
  };
  auto landed = [&](uint32_t full, uint32_t parity) {  // what was requested, whatever the word says
    for (int i = 0; i < 1 << 14 && !mbar_try_wait(full, parity); ++i) {
    }
  };

  if (warp < 8) {
    // ------------------------------------------------------------------ softmax + epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    const int s = warp >> 2;  // sub-tile
    if (s < n_sub && n_tiles > 0 && !q_boxes) {
      if constexpr (kRope) {
        // q <- rotary_pos_emb(q, p): (lo, hi) = (x[i], x[i + 64]) -> (lo cos - hi sin, hi cos + lo sin) in fp32,
        // rounded once to bf16, then stored like the unrotated rows
        uint8_t* q_tile = smem + kOffQ + s * kTileBytes;
        const int c = tid & 7;
        auto turn_and_store = [&](int j, const float4 (&t)[4]) {
          __nv_bfloat162* lo = reinterpret_cast<__nv_bfloat162*>(&qv[2 * j]);
          __nv_bfloat162* hi = reinterpret_cast<__nv_bfloat162*>(&qv[2 * j + 1]);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 a = __bfloat1622float2(lo[e]), h = __bfloat1622float2(hi[e]);
            lo[e] = __floats2bfloat162_rn(a.x * t[e].x - h.x * t[e].y, a.y * t[e].z - h.y * t[e].w);
            hi[e] = __floats2bfloat162_rn(h.x * t[e].x + a.x * t[e].y, h.y * t[e].z + a.y * t[e].w);
          }
          const int r = (tid >> 3 & 15) + 16 * j;
          uint8_t* dst = q_tile + r * 128 + ((c ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(dst) = qv[2 * j];
          *reinterpret_cast<uint4*>(dst + kHalfBytes) = qv[2 * j + 1];
        };
        float4 cs2[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) cs2[j][e] = __ldg(rope_row[4 + j] + e);
#pragma unroll
        for (int j = 0; j < 4; ++j) turn_and_store(j, cs[j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) turn_and_store(4 + j, cs2[j]);
      } else {
        uint8_t* q_tile = smem + kOffQ + s * kTileBytes + (q_chunk >> 3) * kHalfBytes;
#pragma unroll
        for (int j = 0; j < kRowChunks; ++j) {
          const int r = q_row + kRowsPerPass * j;
          *reinterpret_cast<uint4*>(q_tile + r * 128 + (((q_chunk & 7) ^ (r & 7)) << 4)) = qv[j];
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> tensor-core reads
      mbar_arrive(bar(Q_FULL + s));
    }
    if (s < n_sub) {
      const int m = tid & 127;  // MMA row = TMEM lane
      const int sub_row0 = row0 + s * R;
      const int sub_nrows = min(R, nrows - s * R);
      const int slot_local = m >> lg;
      const bool row_ok = slot_local < sub_nrows;
      const int slot = sub_row0 + (row_ok ? slot_local : 0);
      const int head = h0 + (m & (Gp - 1));
      const int32_t* vis_row = vis + (size_t)(kWalk ? slot : 0) * P;
      const int32_t* vis_first = tab->first[s];  // shortest prefix of the sub-tile, per active shard (not kWalk: of all keys)
      // not kWalk: tiles that end at or before `unmasked` need no mask; how many of the CTA's keys this row sees is kept in
      // shared memory (unused columns of the shard table) for the others
      const int unmasked = kWalk ? 0 : min(vis_first[0] - key0, n_keys);
      volatile int* const my_seen = tab->kk + s * kM + m;
      if constexpr (!kWalk) *my_seen = row_ok ? seen_by(slot) - key0 : 0;
      const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
      uint32_t s_addr = lane_base + (uint32_t)(s * 128);  // kRing: the buffer of the current tile
      const uint32_t o_addr = kRing ? lane_base + C::kOCol + (uint32_t)(s * kD) : s_addr + C::kOCol;
      const float c = p.scale * 1.4426950408889634f;  // logits are kept in log2 units: x = s * scale * log2(e)
      const uint64_t c2 = pack2(c, c);
      float m_run = -INFINITY;   // reference max the accumulators are scaled by (may lag, see kRescaleBf16)
      float m_true = -INFINITY;  // exact running max
      float l_run = 0.f;         // sum of the weights; with !kLateMax and bf16 weights as the tensor core sees the largest
      float l_fix = 0.f;         // kLateMax: what that adds to it, see top_error
      // This row's prefix lengths in the current and the next three active shards (a tile spans at most four), fetched
      // as the stream moves on so that the loads are off the critical path.
      auto row_vis = [&](int j) { return (kWalk && j < n_act && row_ok) ? __ldg(vis_row + tab->kk[j]) : 0; };
      int vq0 = row_vis(0), vq1 = row_vis(1), vq2 = row_vis(2), vq3 = row_vis(3);
      ChunkCursor cur{};
      if (kWalk) cur.start(tab, n_act);
      int kk_open = -1;  // kWalk: the shard whose partial is being accumulated
      int n_flushed = 0;  // kWalk: partials written so far
      // kWalk: writes this warp's finished rows from TMEM, scaled.  kBoxes: through shared memory to the copy engine, a box per 64
      // columns; a box that would reach past the rows of the shard is left to the threads.  (Stores from the threads, 32 bytes
      // into each of 32 rows per instruction, keep a CTA's memory pipe busy for 3200 cycles, one copy per row takes 2200
      // cycles to issue.)  Otherwise every thread stores its own row.
      const int warp_row0 = sub_row0 + (((warp & 3) * 32) >> lg);
      const bool boxed = kBoxes && tma.o_valid && warp_row0 + (32 >> lg) <= sub_row0 + sub_nrows;
      const bool rows32 = (reinterpret_cast<uint64_t>(p.o_part) & 31) == 0;  // rows are multiples of 128 bytes
      auto store_rows = [&](float scale, bool have, int z, __nv_bfloat16* dst) {
        uint8_t* stage = smem + C::kOffStage + warp * C::kStageWarpBytes;
        if constexpr (kBoxes) {
          if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the previous rows have left
          __syncwarp();
        }
#pragma unroll
        for (int half = 0; half < C::kHalves; ++half) {
          uint32_t o[64];
          if (have) {
            CASCADE_TMEM_LD32(o_addr + (uint32_t)(half * 64), o, 0);
            CASCADE_TMEM_LD32(o_addr + (uint32_t)(half * 64 + 32), o, 32);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int j = 0; j < 64; ++j) o[j] = 0u;
          }
          auto packed = [&](int j) {
            uint4 val;
            val.x = pack_bf16x2(__uint_as_float(o[j]) * scale, __uint_as_float(o[j + 1]) * scale);
            val.y = pack_bf16x2(__uint_as_float(o[j + 2]) * scale, __uint_as_float(o[j + 3]) * scale);
            val.z = pack_bf16x2(__uint_as_float(o[j + 4]) * scale, __uint_as_float(o[j + 5]) * scale);
            val.w = pack_bf16x2(__uint_as_float(o[j + 6]) * scale, __uint_as_float(o[j + 7]) * scale);
            return val;
          };
          if (boxed) {
#pragma unroll
            for (int j = 0; j < 64; j += 8)
              *reinterpret_cast<uint4*>(stage + half * 4096 + lane * 128 + (((j >> 3) ^ (lane & 7)) << 4)) = packed(j);
          } else if (row_ok) {
#pragma unroll
            for (int j = 0; j < 64; j += 16) {
              const uint4 a = packed(j), b2 = packed(j + 8);
              __nv_bfloat16* to = dst + half * 64 + j;
              if (rows32) {
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(to), "r"(a.x), "r"(a.y), "r"(a.z),
                             "r"(a.w), "r"(b2.x), "r"(b2.y), "r"(b2.z), "r"(b2.w)
                             : "memory");
              } else {
                *reinterpret_cast<uint4*>(to) = a;
                *reinterpret_cast<uint4*>(to + 8) = b2;
              }
            }
          }
        }
        if (boxed) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // this thread's writes -> the copy engine's reads
          __syncwarp();
          if (lane == 0) {
#pragma unroll
            for (int half = 0; half < C::kHalves; ++half)
              tma_store4(&tma.o, half * 64, h0, warp_row0, z, smem_u32(stage + half * 4096));
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
        }
      };
      // kWalk: writes the finished partial of shard kk (this thread's row of u, and m, l) from TMEM and the running
      // statistics, then starts over.
      auto flush_shard = [&](int kk) {
        float o_scale = 0.f, m_out = -INFINITY, l_out = 0.f;
        if (l_run > 0.f) {
          o_scale = 1.f / l_run;
          l_out = l_run * ex2(m_run - m_true);
          m_out = m_true * 0.6931471805599453f;
        }
        if (wc.load(1)) return;  // nothing is written any more
        const int64_t stat = (((int64_t)b * P + kk) * pl.n_q + slot) * p.H + head;
        if (row_ok) {
          p.m_part[stat] = m_out;
          p.l_part[stat] = l_out;
        }
        store_rows(o_scale, true, b * P + kk, static_cast<__nv_bfloat16*>(p.o_part) + stat * kD);
        m_run = -INFINITY;
        m_true = -INFINITY;
        l_run = 0.f;
      };
      for (int i = 0; i < n_tiles; ++i) {
        // kWalk: a tile holds chunks of one shard only; the cursor stands at the tile's first chunk
        const int nch = kWalk ? min(4, cur.nc - cur.c) : tile_chunks(i);
        const bool opens = kWalk ? cur.c == 0 : i == 0;  // first tile of a shard (kWalk) or of the stream
        const int kk_tile = kWalk ? tab->kk[cur.j] : 0;
        // kWalk: mask bookkeeping for the tile's four chunks, done before the wait so that it costs nothing: a chunk of shard
        // j starting at key t0 needs the mask only if it reaches past the shortest prefix of the sub-tile; this row
        // then sees its first lc = vis - t0 columns.  Chunks a narrow last tile does not have count as fully masked.
        int lc[kWalk ? 4 : 1];
        uint32_t needm = 0;
        if constexpr (kWalk) {
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            if (ch < nch) {  // warp-uniform
              const int t0 = cur.c * kChunk;
              if (t0 + kChunk > vis_first[cur.j]) needm |= 1u << ch;
              lc[ch] = vq0 - t0;
              if (cur.advance(tab, n_act)) {
                vq0 = vq1;
                vq1 = vq2;
                vq2 = vq3;
                vq3 = row_vis(cur.j + 3);
              }
            } else {
              needm |= 1u << ch;
              lc[ch] = 0;
            }
          }
        }
        if constexpr (kWalk) {
          // The issuing warp commits O_RDY right after the last product of a shard, before it issues the logits of
          // this tile, so the previous shard's partial is written out while those logits are computed.  The first
          // product of this shard (which overwrites the accumulator) waits for this thread's arrival on P_FULL(i).
          if (opens) {
            if (i > 0) {
              // kRing: a parity tells PV(i-1) from PV(i-3) only once PV(i-2) is known to be in, which S_FULL(i) says
              if (kRing) wait_bar(wc, s_full(s, i), s_parity(i), 1, i);
              wait_bar(wc, bar(O_RDY + s), (uint32_t)((kRing ? i - 1 : n_flushed) & 1), 2, i);
              tc_fence_after();
              flush_shard(kk_open);
              ++n_flushed;
            }
            kk_open = kk_tile;
          }
        }
        wait_bar(wc, s_full(s, i), s_parity(i), 1, i);
        tc_fence_after();
        if constexpr (kRing) s_addr = lane_base + (uint32_t)((2 * i + s) % 3) * 128u;
        uint32_t sr[128];
        CASCADE_TMEM_LD32(s_addr, sr, 0);
        if (nch > 1) CASCADE_TMEM_LD32(s_addr + 32, sr, 32);
        if (nch > 2) CASCADE_TMEM_LD32(s_addr + 64, sr, 64);
        if (nch > 3) CASCADE_TMEM_LD32(s_addr + 96, sr, 96);
        tmem_wait_ld();
        // The mask is applied through a bit mask so that the compiler can move several bits at a time into predicates.
        if constexpr (!kWalk) {
          if (kNMax * (i + 1) > unmasked) {  // warp-uniform
            const int mine = min(*my_seen, n_keys) - kNMax * i;  // visible columns of the tile
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              const int lc_ch = mine - kChunk * ch;
              const uint32_t mk = lc_ch >= 32 ? 0xffffffffu : (lc_ch <= 0 ? 0u : ((1u << lc_ch) - 1u));
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (!((mk >> j) & 1u)) sr[32 * ch + j] = 0xff800000u;  // -inf
            }
          }
        } else if (needm != 0) {  // warp-uniform
#pragma unroll
          for (int ch = 0; ch < 4; ++ch) {
            if ((needm >> ch) & 1u) {  // warp-uniform
              const uint32_t mk = lc[ch] >= 32 ? 0xffffffffu : (lc[ch] <= 0 ? 0u : ((1u << lc[ch]) - 1u));
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (!((mk >> j) & 1u)) sr[32 * ch + j] = 0xff800000u;  // -inf
            }
          }
        }
        auto row_max = [&]() {  // raw logit
          float mx[4];
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            mx[q4] = __uint_as_float(sr[32 * q4]);
#pragma unroll
            for (int j = 1; j < 31; j += 2)
              mx[q4] = fmax3(mx[q4], __uint_as_float(sr[32 * q4 + j]), __uint_as_float(sr[32 * q4 + j + 1]));
            mx[q4] = fmaxf(mx[q4], __uint_as_float(sr[32 * q4 + 31]));
          }
          return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
        };
        // The reference the weights are scaled by is the maximum of the first tile, and stays that unless a later tile rises
        // far above it.  kLateMax: that shows in the weights, so the maximum of this tile is not needed before its
        // exponentials, and is taken while the products are under way (it was 320 of the 2200 cycles between the logits and
        // the weights; when it was introduced, 2048 tokens 47 -> 44 us, 4 x 8192 with rotary step 2.22 -> 2.06 ms).  Not with kWalk, where most tiles
        // open a shard (434 -> 471 us on 4099 tokens in 16 shards), nor with kRing, whose next logits are there already.
        float smax = 0.f, alpha = 1.f;
        bool changed = false;
        if constexpr (kLateMax) {
          if (opens) {
            smax = row_max();
            m_true = smax * c;
            // Finite also where the row sees nothing of the tile or only logits of -inf: the first finite logit then lies so far
            // above that its weight overflows, and the tile is done again with a reference of its own.
            m_run = fmaxf(m_true, -FLT_MAX);
          }
        } else {  // straight-line: branches here cost more than they save
          smax = row_max();
          m_true = fmaxf(m_true, smax * c);
          float m_new = m_run;
          if (m_run == -INFINITY || m_true > m_run + (kRing ? kRescaleTwoParts : kRescaleBf16)) m_new = m_true;
          alpha = (m_run == -INFINITY) ? 0.f : ex2(m_run - m_new);
          changed = m_new != m_run;
          m_run = m_new;
        }
        float neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
        uint64_t neg_m2 = pack2(neg_m, neg_m);
        uint64_t psum2 = pack2(0.f, 0.f);
        auto exp_chunk = [&](int ch) {
          uint32_t pk[16], pr[kRing ? 16 : 1];
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            float x0, x1;
            unpack2(ffma2(pack2(__uint_as_float(sr[32 * ch + j]), __uint_as_float(sr[32 * ch + j + 1])), c2, neg_m2), x0,
                    x1);
            const float p0 = ex2(x0), p1 = ex2(x1);
            psum2 = fadd2(psum2, pack2(p0, p1));
            if constexpr (kRing) {
              // the upper 16 bits, and what they leave out rounded to bf16: together within 2^-17 of the fp32 weight
              pk[j >> 1] = __byte_perm(__float_as_uint(p0), __float_as_uint(p1), 0x7632);
              pr[j >> 1] = pack_bf16x2(p0 - __uint_as_float(__float_as_uint(p0) & 0xffff0000u),
                                       p1 - __uint_as_float(__float_as_uint(p1) & 0xffff0000u));
            } else {
              pk[j >> 1] = pack_bf16x2(p0, p1);
            }
          }
          // P as the A operand of the PV product: lane = row, column kk holds keys 2 kk and 2 kk + 1
          CASCADE_TMEM_ST16(s_addr + (uint32_t)(16 * ch), pk);
          if constexpr (kRing) CASCADE_TMEM_ST16(s_addr + 64u + (uint32_t)(16 * ch), pr);
        };
        auto exp_tile = [&]() {
          if (nch == 4) {
            // The full tile is one straight-line block, so that the scheduler can run the MUFU instructions of one chunk
            // (8 issue cycles each) under the FMA / convert / store work of its neighbours; with a branch per chunk the
            // two parts ran back to back (1600 cycles per tile instead of the ~1130 the MUFU unit needs).
            exp_chunk(0);
            exp_chunk(1);
            exp_chunk(2);
            exp_chunk(3);
          } else {
#pragma unroll
            for (int ch = 0; ch < 3; ++ch)
              if (ch < nch) exp_chunk(ch);  // warp-uniform
          }
        };
        exp_tile();
        float psum0, psum1;
        unpack2(psum2, psum0, psum1);
        // The tensor core multiplies the weights after rounding them to bf16, while the sum above is taken before.
        // With the reference of another tile even the largest weight of a row has an arbitrary mantissa, so when one key
        // dominates a row its rounding error (up to 2^-9 relative) would go straight into O / l: 0.009 at |v| = 4.5.
        // The sum therefore takes the tile's largest weight as the tensor core sees it (same fma and ex2 as in the
        // loop above, so the same bits); the other weights' errors are small against l or average out.
        // (Not with kRing, whose weights keep 16 bits of mantissa.)
        auto top_error = [&]() {
          const float p_top = ex2(fmaf(smax, c, neg_m));
          return __uint_as_float(pack_bf16x2(0.f, p_top) & 0xffff0000u) - p_top;
        };
        // S_FULL(i) was committed after PV(i-1), so the output accumulator is quiescent until this thread's arrival on
        // P_FULL(i) below.  With kRing the logits run ahead of the products, and O_RDY says when PV(i-1) is in (it cannot
        // complete twice without this thread's arrival, so waiting only when needed keeps the parity).
        auto rescale = [&]() {  // this warp's 32 rows
          if constexpr (kRing) {
            wait_bar(wc, bar(O_RDY + s), (uint32_t)((i - 1) & 1), 2, i);
            tc_fence_after();
          }
          const float f = changed ? alpha : 1.f;
          if constexpr (kWalk) {
#pragma unroll
            for (int cc = 0; cc < kD / 32; ++cc) {
              uint32_t o[32];
              CASCADE_TMEM_LD32(o_addr + (uint32_t)(cc * 32), o, 0);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * f);
              CASCADE_TMEM_ST32(o_addr + (uint32_t)(cc * 32), o, 0);
            }
          } else {  // few registers: the tile's logits are still needed
#pragma unroll 1
            for (int cc = 0; cc < kD / 8; ++cc) {
              uint32_t o[8];
              CASCADE_TMEM_LD8(o_addr + (uint32_t)(cc * 8), o);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 8; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * f);
              CASCADE_TMEM_ST8(o_addr + (uint32_t)(cc * 8), o);
            }
          }
        };
        if constexpr (kLateMax) {
          if (!opens && __any_sync(0xffffffffu, !(psum0 + psum1 < kRescaleSum))) {
            smax = row_max();
            const float m_new = fmaxf(m_run, smax * c);
            alpha = (m_run == -INFINITY) ? 0.f : ex2(m_run - m_new);
            changed = true;
            m_run = m_new;
            neg_m = (m_run == -INFINITY) ? 0.f : -m_run;
            neg_m2 = pack2(neg_m, neg_m);
            l_run *= alpha;
            l_fix *= alpha;
            rescale();
            tmem_wait_st();  // the first weights, too: the second ones go to the same place
            psum2 = pack2(0.f, 0.f);
            exp_tile();
            unpack2(psum2, psum0, psum1);
          }
        } else {
          l_run = l_run * alpha + ((psum0 + psum1) + (kRing ? 0.f : top_error()));
          if (!opens && __any_sync(0xffffffffu, changed)) rescale();
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(p_full(s, i));
        if constexpr (kLateMax) {
          if (!opens) {
            smax = row_max();
            m_true = fmaxf(m_true, smax * c);
          }
          l_run += psum0 + psum1;
          l_fix += top_error();
        }
      }
      auto may_write = [&]() {  // asked after the last product; see goes_on
        return (n_tiles > 0 ? wc.load(1) : *reinterpret_cast<volatile const int32_t*>(wc.status)) == 0;
      };
      if (!kWalk && split > 1) {
        // ---- epilogue of a query tile whose keys were shared by the cluster: CTA r finishes columns r * cols .. of all
        // rows.  Every CTA sends it those columns of its accumulator and its row statistics (relative to its own m).
        const int lcols = (kD == 64 ? 6 : 7) - (31 - __clz(split)), cols = 1 << lcols, me = part_of_keys;
        const int pitch = cols * 4 + 16;  // bytes between received rows: spreads a warp's 16-byte stores over the banks
        const int row = s * kM + m;
        if (n_tiles > 0) {
          wait_bar(wc, bar(O_FULL + s), 0u, 3, n_tiles);
          tc_fence_after();
        }
        const bool out_ok = may_write() && row_ok;
        cluster_barrier();  // every product of the cluster is done: its Q, K and V tiles may be overwritten
        const uint32_t from_me = smem_base + (uint32_t)kOffQ;
        auto slot_of = [&](int sender, int receiver) { return sender < receiver ? sender : sender - 1; };
#pragma unroll
        for (int cc = 0; cc < kD / 32; ++cc) {
          uint32_t o[32];
          if (n_tiles > 0) {
            CASCADE_TMEM_LD32(o_addr + (uint32_t)(cc * 32), o, 0);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = 0u;
          }
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const int to = (cc * 32 + j) >> lcols;
            if (to != me)
              st_cluster(from_me + (uint32_t)((slot_of(me, to) * 2 * kM + row) * pitch + ((cc * 32 + j) & (cols - 1)) * 4), to,
                         o[j], o[j + 1], o[j + 2], o[j + 3]);
          }
        }
        const uint32_t stats = smem_base + (uint32_t)(kOffQ + (split - 1) * 2 * kM * pitch);  // [sender][row] (m, l)
        for (int to = 0; to < split; ++to)
          if (to != me)
            st_cluster(stats + (uint32_t)((slot_of(me, to) * 2 * kM + row) * 16), to, __float_as_uint(m_run),
                       __float_as_uint(l_run), __float_as_uint(l_fix), 0u);
        cluster_barrier();
        const uint8_t* got_stats = smem + kOffQ + (split - 1) * 2 * kM * pitch + row * 16;
        float f_of[7], m_all = m_run, l_all;  // the others' maxima, then their factors
#pragma unroll
        for (int i = 0; i < 7; ++i) {
          f_of[i] = i < split - 1 ? *reinterpret_cast<const float*>(got_stats + i * 2 * kM * 16) : -INFINITY;
          m_all = fmaxf(m_all, f_of[i]);
        }
        const float m_use = m_all == -INFINITY ? 0.f : m_all;
        const float f_me = ex2(m_run - m_use);
        l_all = l_run * f_me;
        float fix_all = l_fix * f_me;
#pragma unroll
        for (int i = 0; i < 7; ++i) {
          f_of[i] = ex2(f_of[i] - m_use);
          if (i < split - 1) {
            l_all += f_of[i] * *reinterpret_cast<const float*>(got_stats + i * 2 * kM * 16 + 4);
            if constexpr (kLateMax) fix_all += f_of[i] * *reinterpret_cast<const float*>(got_stats + i * 2 * kM * 16 + 8);
          }
        }
        const float inv = l_all > 0.f ? 1.f / (l_all + fix_all) : 0.f;
        __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(p.o_out) + (int64_t)b * p.os.batch + (int64_t)slot * p.os.token +
                             (int64_t)head * p.os.head + me * cols;
        for (int c0 = 0; c0 < cols; c0 += 8) {
          float acc[8];
          uint32_t o[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
          if (n_tiles > 0) {
            CASCADE_TMEM_LD8(o_addr + (uint32_t)(me * cols + c0), o);
            tmem_wait_ld();
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[j] = __uint_as_float(o[j]) * f_me;
#pragma unroll
          for (int i = 0; i < 7; ++i) {
            if (i < split - 1) {
              const float4* src = reinterpret_cast<const float4*>(smem + kOffQ + (i * 2 * kM + row) * pitch + c0 * 4);
              const float4 a = src[0], d = src[1];
              acc[0] = fmaf(a.x, f_of[i], acc[0]); acc[1] = fmaf(a.y, f_of[i], acc[1]);
              acc[2] = fmaf(a.z, f_of[i], acc[2]); acc[3] = fmaf(a.w, f_of[i], acc[3]);
              acc[4] = fmaf(d.x, f_of[i], acc[4]); acc[5] = fmaf(d.y, f_of[i], acc[5]);
              acc[6] = fmaf(d.z, f_of[i], acc[6]); acc[7] = fmaf(d.w, f_of[i], acc[7]);
            }
          }
          if (out_ok) {
            uint4 val;
            val.x = pack_bf16x2(acc[0] * inv, acc[1] * inv);
            val.y = pack_bf16x2(acc[2] * inv, acc[3] * inv);
            val.z = pack_bf16x2(acc[4] * inv, acc[5] * inv);
            val.w = pack_bf16x2(acc[6] * inv, acc[7] * inv);
            *reinterpret_cast<uint4*>(dst + c0) = val;
          }
        }
        if (out_ok && me == 0 && p.lse_out)
          p.lse_out[((int64_t)b * pl.n_q + slot) * p.H + head] =
              l_all > 0.f ? (m_use + log2f(l_all)) * 0.6931471805599453f : -INFINITY;
      } else {
      // ---- epilogue
      // Where this row goes is looked up before the wait for the last product, which hides the load.
      __nv_bfloat16* dst = nullptr;
      int64_t stat = 0;
      if (row_ok) {
        if (!kWalk && p.fused) {
          stat = ((int64_t)b * pl.n_q + slot) * p.H + head;
          dst = static_cast<__nv_bfloat16*>(p.o_out) + (int64_t)b * p.os.batch + (int64_t)slot * p.os.token +
                (int64_t)head * p.os.head;
        } else {
          // kWalk: the last shard the CTA saw anything of; its other shards were written on the way.  Otherwise there is
          // only one KV shard, and the row is a token.
          const int row = kWalk ? slot
                                : (int)CASCADE_CHECKED((int64_t)__ldg(pl.q_inv + (size_t)map * pl.n_q + slot), pl.n_q,
                                                       pl.status, 109);
          stat = (((int64_t)b * P + (kWalk ? max(kk_open, 0) : 0)) * pl.n_q + row) * p.H + head;
          dst = static_cast<__nv_bfloat16*>(p.o_part) + stat * kD;
        }
      }
      float o_scale = 0.f, m_out = -INFINITY, l_out = 0.f;
      if (n_tiles > 0) {
        wait_bar(wc, bar(O_FULL + s), 0u, 3, n_tiles);
        tc_fence_after();
        if (l_run > 0.f) {
          o_scale = 1.f / (l_run + l_fix);
          l_out = l_run * ex2(m_run - m_true);  // sum relative to the exact max
          m_out = m_true * 0.6931471805599453f;   // natural-log units
        }
      }
      const bool quiet = !may_write();
      if (quiet) dst = nullptr;
      if (dst) {
        if (p.fused) {
          if (p.lse_out) p.lse_out[stat] = l_out > 0.f ? m_out + logf(l_out) : -INFINITY;
        } else {
          p.m_part[stat] = m_out;
          p.l_part[stat] = l_out;
        }
      }
      if constexpr (kBoxes) {
        if (!quiet) store_rows(o_scale, n_tiles > 0, b * P + max(kk_open, 0), dst);
        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");  // the rows have left shared memory
      } else {
        // The products Q K^T of the CTA have completed, those of the other sub-tile among them: its last one is issued before this
        // sub-tile's last product with V, and a commit waits for all that was issued before it.  So the Q and K tiles in shared
        // memory are free (V may still be read, and is not touched): the thread stages its output row there (rows 16 bytes
        // further apart than they are long, which spreads a warp's accesses over all banks) and the warp stores whole rows, 512 bytes per instruction.  (A bulk copy per row took 2200 cycles to issue; boxes as
        // with kWalk are issued once here, and the first use of a tensor map costs more: 2048 tokens 43.6 -> 45.0 us.)
        uint8_t* stage = smem + C::kOffStage + (s * kM + m) * C::kStageRowBytes;
#pragma unroll
        for (int cc = 0; cc < kD / 32; ++cc) {
          uint32_t o[32];
          if (n_tiles > 0) {
            CASCADE_TMEM_LD32(o_addr + (uint32_t)(cc * 32), o, 0);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = 0u;
          }
#pragma unroll
          for (int j = 0; j < 32; j += 8) {
            uint4 val;
            val.x = pack_bf16x2(__uint_as_float(o[j]) * o_scale, __uint_as_float(o[j + 1]) * o_scale);
            val.y = pack_bf16x2(__uint_as_float(o[j + 2]) * o_scale, __uint_as_float(o[j + 3]) * o_scale);
            val.z = pack_bf16x2(__uint_as_float(o[j + 4]) * o_scale, __uint_as_float(o[j + 5]) * o_scale);
            val.w = pack_bf16x2(__uint_as_float(o[j + 6]) * o_scale, __uint_as_float(o[j + 7]) * o_scale);
            *reinterpret_cast<uint4*>(stage + cc * 64 + j * 2) = val;
          }
        }
        __syncwarp();
        const uint64_t dst_or_null = reinterpret_cast<uint64_t>(dst);  // null past the end of the sub-tile
        constexpr int kLanesPerRow = C::kRowBytes / 16, kRowsAtOnce = 32 / kLanesPerRow;
        const uint8_t* rows = smem + C::kOffStage + (s * kM + m - lane) * C::kStageRowBytes + (lane % kLanesPerRow) * 16;
#pragma unroll
        for (int r0 = 0; r0 < 32; r0 += kRowsAtOnce) {
          const int r = r0 + lane / kLanesPerRow;
          const uint64_t to = __shfl_sync(0xffffffffu, dst_or_null, r);
          const uint4 val = *reinterpret_cast<const uint4*>(rows + r * C::kStageRowBytes);
          if (to) *reinterpret_cast<uint4*>(to + (lane % kLanesPerRow) * 16) = val;
        }
      }
      }
      if constexpr (kWalk) {
        // the shards of which no row of the CTA sees anything were never walked: their partials are empty
        if (row_ok && may_write()) {
          int a = 0;
          for (int k = 0; k < P; ++k) {
            if (a < n_act && tab->kk[a] == k) {
              ++a;
              continue;
            }
            if (n_act == 0 && k == 0) continue;  // written by the epilogue above
            const int64_t st2 = (((int64_t)b * P + k) * pl.n_q + slot) * p.H + head;
            p.m_part[st2] = -INFINITY;
            p.l_part[st2] = 0.f;
            uint4* row = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.o_part) + st2 * kD);
#pragma unroll
            for (int j = 0; j < kRowChunks; ++j) row[j] = make_uint4(0u, 0u, 0u, 0u);
          }
        }
      }
      tc_fence_before();
    } else if (!kWalk && split > 1) {
      cluster_barrier();
      cluster_barrier();
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == 8) {
      // ---------------------------------------------------------------- MMA issuer
      // All 32 lanes run the loop (waits included) so that every address and descriptor is warp-uniform; the
      // tcgen05 instructions themselves are issued by one elected lane.
      const bool leader = elect_one();
      constexpr uint32_t idesc_pv = make_idesc(kM, kD, 0, 1);
      constexpr uint32_t hi_kmajor = desc_hi(1024);  // Q, K: 8-row groups 1024 bytes apart
      constexpr uint32_t hi_v = desc_hi(1024);       // V (MN-major): 8-key groups 1024 bytes apart
      const uint32_t q_lo0 = desc_lo(smem_base + kOffQ, 16);
      const uint32_t k_lo0 = desc_lo(smem_base + kOffK, 16);
      const uint32_t v_lo0 = desc_lo(smem_base + kOffV, kHalfBytes);  // the two 64-column halves of d
      if (n_tiles > 0) {
        auto s_col = [&](int s, int i) {  // logit buffer of sub-tile s, tile i
          return tmem + (uint32_t)((kRing ? (2 * i + s) % 3 : s) * 128);
        };
        auto issue_qk = [&](int s, int i, int n) {  // S_s = Q_s K(i)^T, n keys wide
          const uint32_t q_lo = q_lo0 + (uint32_t)(s * (kTileBytes >> 4));
          const uint32_t k_lo = k_lo0 + (uint32_t)((i % kKStages) * (kTileBytes >> 4));
          const uint32_t idesc_qk = make_idesc(kM, n, 0, 0);
          if (leader) {
#pragma unroll
            for (int ks = 0; ks < kD / 16; ++ks) {
              // 16 elements of head_dim = 32 bytes along the 128-byte row; elements 64.. live in the second half
              const uint32_t off = (uint32_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4);
              mma_ss(s_col(s, i), q_lo + off, k_lo + off, hi_kmajor, idesc_qk, ks > 0);
            }
            mma_commit(s_full(s, i));
          }
        };
        // O_s (+)= P_s V(i) over n keys; a tile that opens a shard (kWalk) or the stream starts the accumulator afresh
        auto issue_pv = [&](int s, int i, int n, bool opens) {
          const uint32_t v_lo = v_lo0 + (uint32_t)((i % kVStages) * (kTileBytes >> 4));
          const int ksteps = n >> 4;
          if (leader) {
#pragma unroll
            for (int ks = 0; ks < kNMax / 16; ++ks) {
              // A = P from TMEM: 16 keys = 8 columns; B = V (MN-major): 16 keys = 16 rows of 128 bytes
              if (ks < ksteps)
                mma_ts(tmem + C::kOCol + (uint32_t)(s * kD), s_col(s, i) + (uint32_t)(ks * 8),
                       v_lo + (uint32_t)(ks * (2048 >> 4)), hi_v, idesc_pv, !opens || ks > 0);
            }
            if constexpr (kRing) {  // the rest of P
#pragma unroll
              for (int ks = 0; ks < kNMax / 16; ++ks)
                if (ks < ksteps)
                  mma_ts(tmem + C::kOCol + (uint32_t)(s * kD), s_col(s, i) + (uint32_t)(64 + ks * 8),
                         v_lo + (uint32_t)(ks * (2048 >> 4)), hi_v, idesc_pv, true);
              mma_commit(bar(O_RDY + s));
            }
          }
        };
        TileSeq<kWalk> seq(tab, n_act, n_keys);
        bool opens_cur = true, opens_next = false;
        int n_cur = kChunk * seq.next(opens_cur), n_next = 0;
        // A wait that gives up ends the role: nothing more is issued, and no stage given back that may not be full (the loader
        // would have a second load counted on its barrier while the first is under way).
        bool fed = wait_bar(wc, bar(K_FULL), 0u, 7);
        for (int s = 0; s < n_sub; ++s) {
          fed = fed && wait_bar(wc, bar(Q_FULL + s), 0u, 6);
          tc_fence_after();
          if (fed) issue_qk(s, 0, n_cur);
        }
        if (fed && leader) mma_commit(bar(K_EMPTY));
        int n_run = fed ? n_tiles : 0;
        if constexpr (kRing) {
          // Order: QK_0(0) QK_1(0) QK_0(1), then per tile i: PV_0(i) QK_1(i+1) PV_1(i) QK_0(i+2).  QK_1(i+1) takes the
          // buffer PV_0(i) has read, QK_0(i+2) the one of PV_1(i); MMAs execute in issue order, so neither needs a
          // barrier.  K(j) is released after QK_1(j), the later of its two readers.
          const int last_sub = n_sub - 1;
          auto wait_k = [&](int i) {
            fed = fed && wait_bar(wc, bar(K_FULL + i % kKStages), (uint32_t)((i / kKStages) & 1), 7, i);
            tc_fence_after();
          };
          bool opens_2 = false;
          int n_2 = 0;
          if (n_tiles > 1) {
            n_next = kChunk * seq.next(opens_next);
            wait_k(1);
            if (fed) issue_qk(0, 1, n_next);
            if (fed && last_sub == 0 && leader) mma_commit(bar(K_EMPTY + 1 % kKStages));
          }
          if (!fed || !goes_on()) n_run = 0;
          for (int i = 0; i < n_run; ++i) {
            n_2 = i + 2 < n_run ? kChunk * seq.next(opens_2) : 0;
            fed = wait_bar(wc, bar(V_FULL + i % kVStages), (uint32_t)((i / kVStages) & 1), 4, i);
            for (int s = 0; s < n_sub && fed; ++s) {
              fed = wait_bar(wc, p_full(s, i), s_parity(i), 5, i);
              if (!fed) break;
              tc_fence_after();
              issue_pv(s, i, n_cur, opens_cur);
              if (i == n_run - 1 && leader) mma_commit(bar(O_FULL + s));
              if (s == last_sub && leader) mma_commit(bar(V_EMPTY + i % kVStages));
              if (s == 0 && n_sub == 2 && i + 1 < n_run) {
                issue_qk(1, i + 1, n_next);
                if (leader) mma_commit(bar(K_EMPTY + (i + 1) % kKStages));
              }
              if (s == last_sub && i + 2 < n_run) {
                wait_k(i + 2);
                if (!fed) break;
                issue_qk(0, i + 2, n_2);
                if (last_sub == 0 && leader) mma_commit(bar(K_EMPTY + (i + 2) % kKStages));
              }
            }
            if (!fed) break;
            n_cur = n_next;
            opens_cur = opens_next;
            n_next = n_2;
            opens_next = opens_2;
          }
        } else {
        if (!fed || !goes_on()) n_run = 0;
        for (int i = 0; i < n_run && fed; ++i) {
          const bool has_next = i + 1 < n_run;
          if (i > 0) {
            n_cur = n_next;
            opens_cur = opens_next;
          }
          n_next = has_next ? kChunk * seq.next(opens_next) : 0;
          fed = wait_bar(wc, bar(V_FULL + i % kVStages), (uint32_t)((i / kVStages) & 1), 4, i);
          for (int s = 0; s < n_sub && fed; ++s) {
            fed = wait_bar(wc, p_full(s, i), s_parity(i), 5, i);
            if (!fed) break;
            tc_fence_after();
            issue_pv(s, i, n_cur, opens_cur);
            if (!has_next && leader) mma_commit(bar(O_FULL + s));
            if (kWalk && has_next && opens_next && leader) mma_commit(bar(O_RDY + s));
            if (s == n_sub - 1 && leader) mma_commit(bar(V_EMPTY + i % kVStages));
            if (has_next) {
              if (s == 0) {
                fed = wait_bar(wc, bar(K_FULL + (i + 1) % kKStages), (uint32_t)(((i + 1) / kKStages) & 1), 7, i);
                if (!fed) break;
                tc_fence_after();
              }
              issue_qk(s, i + 1, n_next);
              if (s == n_sub - 1 && leader) mma_commit(bar(K_EMPTY + (i + 1) % kKStages));
            }
          }
        }
        }
        if (n_run == 0 || !fed) {
          // Everything issued so far, at the barrier of the second sub-tile: that of the first may have had its one arrival already,
          // when the wait for the other's last weights ran out, and would then say nothing of the products issued since.  (A
          // constant: as the barrier of the later sub-tile it cost all calls a hundredth, 268 tokens 8.9 -> 9.0 us.)
          if (leader) mma_commit(bar(O_FULL + 1));
          if (q_boxes)
            for (int s = 0; s < n_sub; ++s) landed(bar(Q_FULL + s), 0u);
          landed(bar(O_FULL + 1), 0u);
        }
      }
      __syncwarp();
    } else {
      // ---------------------------------------------------------------- loaders
      // Every barrier is served by one warp only, in tile order: a phase-parity wait cannot tell "one phase behind"
      // from "one phase ahead", so a warp must never skip a use of a stage.
      //   warp 9: the K tiles, warp 10: the V tiles (warp 11 has no work).
      const int lw = warp - 9;
      if (lw == 2) {
        if (lane == 0) {
          if (gave_up) wc.store(1, 1);
          mbar_arrive(bar(CHECKED));
        }
      } else if (n_tiles > 0) {
        const bool is_k = lw == 0;
        const CUtensorMap* map = is_k ? &tma.k : &tma.v;
        const int z = b * p.Hkv + g;  // kWalk: which [n_kv][head_dim] matrix of the shard-major copy
        const int n_stages = is_k ? kKStages : kVStages;
        const int full0 = is_k ? K_FULL : V_FULL, empty0 = is_k ? K_EMPTY : V_EMPTY;
        const uint32_t tiles_s = smem_base + (is_k ? kOffK : kOffV);
        const bool leader = elect_one();
        ChunkCursor cur{};
        if (kWalk) cur.start(tab, n_act);
        // The shard-major copies are written by the gather grid launched just before this one; when this grid was
        // launched as its programmatic dependent it may have started early, so wait here for that grid to complete
        // (a no-op otherwise).  Nothing else in this kernel reads what the gather grid writes.
        grid_wait();
        int n_issued = 0;
        for (int i = 0; i < n_tiles; ++i) {
          const int nch = kWalk ? min(4, cur.nc - cur.c) : tile_chunks(i);
          const int st = i % n_stages;
          note(8 * i + 1);
          // The first use of a stage waits for nothing, and must not: the products may have consumed a first tile that was
          // requested early before this warp gets here, and a wait for the phase before that would never end.
          if (i >= n_stages && !wait_bar(wc, bar(empty0 + st), (uint32_t)(((i / n_stages) & 1) ^ 1), is_k ? 9 : 10, i)) break;
          const uint32_t dst = tiles_s + (uint32_t)(st * kTileBytes), fb = bar(full0 + st);
          if constexpr (kWalk) {
            if (leader) mbar_expect_tx(fb, (uint32_t)(nch * C::kHalves * kChunkBytes));
            for (int ch = 0; ch < nch; ++ch) {
              // A chunk is 32 consecutive rows of the shard-major copy.  Rows past the shard's visible prefix belong
              // to later keys or, past the end of the matrix, are zero-filled: they are masked either way.
              const int slot = tab->slot0[cur.j] + cur.c * kChunk;
              if (leader) {
                tma_tile3(dst + (uint32_t)(ch * kChunkBytes), map, 0, slot, z, fb);
                if (C::kHalves == 2) tma_tile3(dst + (uint32_t)(kHalfBytes + ch * kChunkBytes), map, 64, slot, z, fb);
              }
              cur.advance(tab, n_act);
            }
          } else if (leader && !(i == 0 && ((early >> lw) & 1))) {
            // 128 rows at a time; rows past what any query sees lie outside the tensor map and are zero-filled, so that
            // whatever the unwritten tail of a cache holds stays out of the products
            mbar_expect_tx(fb, (uint32_t)kTileBytes);
            tma_tile4(dst, map, 0, key0 + kNMax * i, g, b, fb);
            if (C::kHalves == 2) tma_tile4(dst + (uint32_t)kHalfBytes, map, 64, key0 + kNMax * i, g, b, fb);
          }
          __syncwarp();
          n_issued = i + 1;
          note(8 * i + 2);
        }
        if (!goes_on())
          for (int i = max(0, n_issued - n_stages); i < n_issued; ++i) landed(bar(full0 + i % n_stages), (uint32_t)((i / n_stages) & 1));
      }
    }
    if (!kWalk && split > 1) {
      cluster_barrier();
      cluster_barrier();
    }
  }
  if (after_gather) grid_wait();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
}

}  // namespace tc

namespace {

// Shard-major K or V copy as a 3-D tensor [batch * kv_heads][n_kv][head_dim]; box = one chunk (32 rows) x 64 columns.
bool encode_sorted(CUtensorMap* map, const void* base, int d, int64_t n_kv, int64_t n_mats) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)n_kv, (cuuint64_t)n_mats};
  const cuuint64_t strides[2] = {(cuuint64_t)d * 2, (cuuint64_t)n_kv * d * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)tc::kChunk, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Number of SMs of the current device (queried once per device).
int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 148;
    cached[dev] = n;
  }
  return cached[dev];
}

}  // namespace

namespace {

// K or V rows in token order, [batch][kv_heads][rows][d] by strides; rows past `n_rows` read as zeros.
bool encode_rows(CUtensorMap* map, const TcRows& r, int d, int64_t n_rows, int64_t n_heads, int64_t batch) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)std::max<int64_t>(1, n_rows), (cuuint64_t)n_heads,
                              (cuuint64_t)batch};
  auto stride = [&](int64_t elems, int64_t extent) { return (cuuint64_t)(extent > 1 ? elems * 2 : d * 2); };
  const cuuint64_t strides[3] = {stride(r.strides.token, n_rows), stride(r.strides.head, n_heads),
                                 stride(r.strides.batch, batch)};
  const cuuint32_t box[4] = {64, (cuuint32_t)tc::kNMax, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(r.base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output rows [outer][rows][heads][d]; box = the rows of one warp (32 >> lg rows x 1 << lg heads), 64 columns.
bool encode_out(CUtensorMap* map, void* base, int d, int lg, int64_t heads, int64_t rows, int64_t outer, const Strides& st) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)heads, (cuuint64_t)rows, (cuuint64_t)outer};
  auto stride = [&](int64_t elems, int64_t extent) { return (cuuint64_t)(extent > 1 ? elems * 2 : d * 2); };
  const cuuint64_t strides[3] = {stride(st.head, heads), stride(st.token, rows), stride(st.batch, outer)};
  const cuuint32_t box[4] = {64, 1u << lg, 32u >> lg, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query rows [batch][tokens][heads][d]; box = a sub-tile (128 >> lg tokens x 1 << lg heads), 64 columns.
bool encode_queries(CUtensorMap* map, const AttnParams& p, int lg) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn || !tc_rows_loadable({p.q, p.qs}, p.plan.n_q, p.H, p.batch)) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)p.d, (cuuint64_t)p.H, (cuuint64_t)p.plan.n_q, (cuuint64_t)p.batch};
  auto stride = [&](int64_t elems, int64_t extent) { return (cuuint64_t)(extent > 1 ? elems * 2 : p.d * 2); };
  const cuuint64_t strides[3] = {stride(p.qs.head, p.H), stride(p.qs.token, p.plan.n_q), stride(p.qs.batch, p.batch)};
  const cuuint32_t box[4] = {64, 1u << lg, 128u >> lg, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(p.q), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct TcLaunch {
  int lg, tile_major, lg_split, early;
  bool after_gather;
  bool boxes;  // partials at head_dim 128
};

cudaError_t launch_kernel(const AttnParams& p, bool walk, const TcLaunch& l, int64_t n_tiles, const tc::TmaArgs& tma,
                          cudaStream_t stream) {
  auto kernel = p.d == 64 ? (walk ? tc::attn_tc_kernel<64, false, true, true> : tc::attn_tc_kernel<64, false, false, false>)
                : p.rope  ? tc::attn_tc_kernel<128, true, false, false>
                : !walk   ? tc::attn_tc_kernel<128, false, false, false>
                          : (l.boxes ? tc::attn_tc_kernel<128, false, true, true> : tc::attn_tc_kernel<128, false, true, false>);
  const int smem_bytes = p.d == 64 ? (walk ? tc::Cfg<64, true>::kSmemBytes : tc::Cfg<64, false>::kSmemBytes)
                                   : (l.boxes ? tc::Cfg<128, true>::kSmemBytes : tc::Cfg<128, false>::kSmemBytes);
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  if (e != cudaSuccess) return e;
  // (few CTAs if tile_major; a head group has a head, so n_hg and the batch fit the short axes as the entry points check)
  const unsigned n_hg = (unsigned)(p.H >> l.lg), batch = (unsigned)p.batch, tiles = (unsigned)n_tiles;
  const dim3 grid = l.tile_major ? dim3(n_hg << l.lg_split, batch, tiles) : dim3(tiles, n_hg, batch);
  TimedLaunch timed(stream);
  return launch_dependent(kernel, grid, tc::kThreads, smem_bytes, 1u << l.lg_split, !walk || l.after_gather, stream, p, l.lg,
                          l.tile_major, l.lg_split, l.early, (int)l.after_gather, tma);
}

// stack as many of the G heads of a KV head into one MMA tile as divide G (at most 8)
int stacked_log2(int G) {
  int lg = 0;
  while (lg < 3 && G % (2 << lg) == 0) ++lg;
  return lg;
}

}  // namespace

bool tc_rows_loadable(const TcRows& r, int64_t n_rows, int64_t n_heads, int64_t batch) {
  auto fine = [](int64_t stride, int64_t extent) { return extent <= 1 || (stride > 0 && stride < (int64_t)1 << 38); };
  return fine(r.strides.token, n_rows) && fine(r.strides.head, n_heads) && fine(r.strides.batch, batch);
}

// Estimated time in us of the partials of several shards at head_dim 64, see rows_time: a CTA takes 2 to 3.2 us a shard (by how
// many of its rows exist) and 1.5 us for every further 128 keys of it.  It is the wrong kernel for a query or KV shard of a few
// tokens: 130 tokens in 40 shards, 12 / 12 heads, 338 us and 99 on the ALUs; 500 tokens in 40 shards 345 and 238, with 16 / 4
// heads 176 and 317.
double tc_partials_time(const AttnParams& p) {
  const CutSize c(p);
  const int lg = stacked_log2(p.G);
  const double tiles = p.plan.n_qtiles[3 - lg], rows = p.plan.n_q / tiles;
  const double shard = 2 + 1.2 * rows / (256 >> lg) + 1.5 * (std::ceil(c.keys / 128) - 1);
  return std::ceil(tiles * (c.heads / (1 << lg)) / kEstimateSms) * (4 + c.shards * shard);
}

cudaError_t launch_attn_tc_partials(const AttnParams& p, const void* k_sorted, const void* v_sorted, cudaStream_t stream) {
  tc::TmaArgs tma = {};
  const int64_t n_mats = (int64_t)p.batch * p.Hkv;
  if (!encode_sorted(&tma.k, k_sorted, p.d, p.plan.n_kv, n_mats) ||
      !encode_sorted(&tma.v, v_sorted, p.d, p.plan.n_kv, n_mats)) {
    set_error("tensor-core attention: could not build the TMA descriptors of the shard-major K/V copies");
    return cudaErrorInvalidValue;
  }
  const int lg = stacked_log2(p.G);
  const int64_t n_q = p.plan.n_q;
  // Boxes: at head_dim 64 always (4099 tokens in 16 shards, 32 / 8 heads: 389 -> 361 us with the post-pass).  At head_dim 128, where
  // they cost the second K and V stages, with at least four heads a tile (a box is 32 rows of (slot, head), so it seldom
  // reaches past a shard), two sub-tiles in nearly every query tile, which hide each other's loads, and more than a chunk of
  // keys in a shard: 32 / 8 heads, 2000 tokens in 32 shards 289 -> 256 us, 4099 in 16 348 -> 336, 16 / 4 heads, 3000 in 30 269
  // -> 246.  Elsewhere they lose up to a quarter: 16 / 8 heads, 2000 tokens in 32 shards 199 and 226, 8 / 8 heads 178 and 222;
  // 32 / 4 heads, 1000 tokens in 31 shards 171 and 202, in 10 shards 72 and 78.
  const CutSize cut(p);
  const int64_t n_tiles = p.plan.n_qtiles[3 - lg];
  const bool boxes = p.d == 64 || (lg >= 2 && cut.keys >= 48 && cut.row_tiles(128 >> lg) >= 1.9 * cut.row_tiles(256 >> lg));
  tma.o_valid = boxes && encode_out(&tma.o, p.o_part, p.d, lg, p.H, n_q, (int64_t)p.batch * p.plan.n_kv_shards,
                                    {n_q * p.H * p.d, (int64_t)p.H * p.d, p.d});
  const int64_t n_ctas = n_tiles * (p.H >> lg) * p.batch;
  // few CTAs per SM: balance matters more than L2 locality
  const TcLaunch l = {lg, n_ctas <= 8 * (int64_t)sm_count(), 0, 0, true, boxes && tma.o_valid};
  return launch_kernel(p, true, l, n_tiles, tma, stream);
}

cudaError_t launch_attn_tc(const AttnParams& p, const TcRows& k, const TcRows& v, int64_t n_seen, bool k_gathered, bool v_gathered,
                           cudaStream_t stream) {
  tc::TmaArgs tma = {};
  if (!encode_rows(&tma.k, k, p.d, n_seen, p.Hkv, p.batch) || !encode_rows(&tma.v, v, p.d, n_seen, p.Hkv, p.batch)) {
    set_error("tensor-core attention: could not build the TMA descriptors of K and V");
    return cudaErrorInvalidValue;
  }
  const int lg = stacked_log2(p.G);
  tma.q_valid = !p.rope && encode_queries(&tma.q, p, lg);
  const int64_t tile_slots = 256 >> lg, n_qt = (p.plan.n_q + tile_slots - 1) / tile_slots;
  const int64_t n_ctas = n_qt * (p.H >> lg) * p.batch;
  // Few query tiles (a chunk of a chunked prefill, a short prompt) leave SMs idle: a cluster then shares the keys of each
  // tile, as far as its CTAs fit at once with one per SM (clusters of 2, 4 and 8: 148, 132 and 120 CTAs) and have three
  // 128-key tiles each, or two at head_dim 64 (500 tokens, 12 heads, in clusters of two 12.0 us, alone 12.9).  With two each
  // at head_dim 128 the exchange and, with a rotary step, query rows turned in every CTA cost more than they save: 500
  // tokens, 32 / 8 heads, 15.4 -> 14.1 us without, with the rotary step 22.5 -> 18.5; 8 / 8 heads, 1000 tokens, 22.2 -> 19.4
  // and 32.2 -> 26.9.  12 tiles in clusters of four take 32.8, alone 36.9.  The rule is the same with and without a rotary
  // step, so that both sum in the same order.  It counts the heads of the whole problem, see AttnParams.
  const int64_t rule_ctas = n_qt * ((int64_t)p.rule_kv_heads * p.G >> lg) * p.batch, key_tiles = (n_seen + 127) / 128;
  int lg_split = 0;
  if (p.fused) {
    const int64_t fit[4] = {148, 148, 132, 120};
    for (int i = 1; i < 4; ++i)
      if (rule_ctas << i <= fit[i] && key_tiles >= (p.d == 64 ? 2 : 3) << i) lg_split = i;
  }
  const TcLaunch l = {lg, n_ctas <= 8 * (int64_t)sm_count(), lg_split,
                      p.prefix_from_vis ? 0 : (k_gathered ? 0 : 1) | (v_gathered ? 0 : 2), k_gathered || v_gathered, false};
  return launch_kernel(p, false, l, n_qt, tma, stream);
}

}  // namespace cascade
