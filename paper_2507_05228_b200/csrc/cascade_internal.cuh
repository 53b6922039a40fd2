// Internal declarations shared by the translation units of the CUDA library (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "cascade.h"

namespace cascade {

constexpr int kNumTileSizes = 4;  // query-tile heights 32, 64, 128, 256

// The report of a wait that gave up, see WaitCtx: code, block, tile, and from word 8 on a progress word for each warp of the CTA.
constexpr int kMaxWaitWarps = 20, kStatusWords = 8 + kMaxWaitWarps;

// Device-side view of a plan.  All arrays have a leading n_maps dimension.
struct PlanDev {
  const int32_t* q_off;
  const int32_t* q_idx;
  const int32_t* q_inv;
  const int32_t* kv_off;
  const int32_t* kv_idx;
  const int32_t* kv_inv;
  const int32_t* kv_slot_shard;  // [n_kv]: the shard whose list holds this position of kv_idx
  const int32_t* vis;
  const uint8_t* pair_class;
  // Query tiles that never cross a shard boundary: {first slot, rows, shard, unused}; rows == 0 pads.
  // Ordered by decreasing work (longest visible prefix first) so late CTAs are the short ones.
  // One list per tile height: qtiles[i] holds tiles of up to (32 << i) slots.
  const int4* qtiles[kNumTileSizes];
  int32_t n_qtiles[kNumTileSizes];  // per map (padded to the maximum over maps)
  int32_t* status;      // device status word, 0 = fine; kStatusWords of them
  int32_t n_maps, n_q, n_kv, n_q_shards, n_kv_shards, q_pos_offset, causal;
};

struct Strides {
  int64_t batch, token, head;
};

struct AttnParams {
  PlanDev plan;
  const void* q;
  const void* k;
  const void* v;
  Strides qs, ks, vs;
  int32_t batch, H, Hkv, G, d;
  // KV heads of the whole problem: more than Hkv where a call computes a part of the heads at a time.  Rules that decide how
  // sums are split go by it, so that the parts get the same bits as one call would.
  int32_t rule_kv_heads;
  int32_t prefix_from_vis;  // the K/V rows have positions of their own: a query's prefix is the sum of its row of vis
  float scale;
  int32_t fused;  // 0: one job per KV shard, write (u, m, l); 1: walk all KV shards, write o (+lse)
  void* o_part;
  float* m_part;
  float* l_part;
  void* o_out;
  Strides os;
  float* lse_out;
  // Rotary step of the pre-pass fused into the staging of Q and K rows (the Pre-Pass algorithm): rows of the positional table,
  // rope[position * 64 + i] = (cos, sin) of position * theta_i; null = rows are used as given.  A query row sits at
  // position q_pos_offset + token, a key row at its token index.
  const float2* rope;
};

// Debug build (-DCASCADE_DEBUG, libcascade_b200_debug.so): every row index that a kernel reads out of a plan array
// before it forms an address is checked against the tensor it indexes; a bad one is recorded in the plan's status word
// (codes 101..; cascade_plan_device_status then fails) and replaced by row 0, so the access itself stays in bounds.
// The release build compiles the checks away.
#ifdef CASCADE_DEBUG
__device__ __forceinline__ int64_t cascade_checked_index(int64_t i, int64_t n, int32_t* status, int code) {
  if (i >= 0 && i < n) return i;
  atomicCAS(status, 0, code);
  return 0;
}
#define CASCADE_CHECKED(i, n, status, code) cascade_checked_index((i), (n), (status), (code))
#else
#define CASCADE_CHECKED(i, n, status, code) (i)
#endif

// What a decode step adds to the fused decode kernel (cascade_decode_step_rope); all zero for a plain decode.
constexpr int kMaxGivenVis = 256;
struct DecodeStep {
  const float2* rope;  // positional table, or null: no rotation, no append
  const __nv_bfloat16 *k_new, *v_new;
  Strides kns, vns;
  int32_t position;  // row of the caches that takes the new token
  int32_t n_vis;     // > 0: the prefix lengths of the plan for this position (n_maps * n_kv_shards of them) come along
  int32_t vis[kMaxGivenVis];
};

struct MergeParams {
  const void* o_part;
  const float* m_part;
  const float* l_part;
  const int32_t* row_scatter;
  int64_t row_scatter_batch_stride;
  void* o_out;
  Strides os;
  float* lse_out;
  int32_t batch, n_parts, n_rows, H, d;
};

// Post-pass that reads every part from the buffer of the party that computed it (cascade_merge_peers).
constexpr int kMaxMergeSources = 16;
struct MergePeersParams {
  const void* o_src[kMaxMergeSources];   // source s: [batch][parts[s]][n_src_rows][H][d]
  const float* m_src[kMaxMergeSources];  //           [batch][parts[s]][n_src_rows][H]
  const float* l_src[kMaxMergeSources];
  int32_t parts[kMaxMergeSources];
  int32_t n_src, n_src_rows;
  const int32_t* row_gather;  // [n_rows]: row of the source buffers that output row r combines; null = r
  void* o_out;
  Strides os;
  float* lse_out;
  int32_t batch, n_rows, H, d;
};

}  // namespace cascade

struct cascade_plan {
  cascade::PlanDev dev;
  std::vector<int32_t> q_off, q_idx, q_inv, kv_off, kv_idx, kv_inv, kv_slot_shard, vis;
  std::vector<int32_t> kv_pos;  // position of every K/V row; empty = the row's own index
  std::vector<uint8_t> pair_class;
  std::vector<int4> qtiles[cascade::kNumTileSizes];
  void* dev_blob = nullptr;
  size_t dev_blob_bytes = 0;
  int device = 0;                // the device that holds dev_blob
  bool dev_blob_pooled = false;  // dev_blob came from the device's plan pool
  // The device arrays vis and pair_class are made by a kernel (cascade_shard_plan, cascade_plan_advance); their host
  // copies are brought up to date only when something reads them (cascade_plan_get, cascade_plan_dense_mask)
  mutable bool host_vis_stale = false;
};

namespace cascade {

void set_error(const char* fmt, ...);
void count_launch(int n = 1);
// Kernel timing (cascade_kernel_timing_begin / _end): brackets a launch with events when recording is on.
void timing_mark(cudaStream_t stream, bool start);
bool timing_recording();  // true between cascade_kernel_timing_begin and _end
struct TimedLaunch {  // RAII: events around the launches issued while it lives
  cudaStream_t st;
  explicit TimedLaunch(cudaStream_t s) : st(s) { timing_mark(st, true); }
  ~TimedLaunch() { timing_mark(st, false); }
};

// Programmatic dependent launch: the blocks of a grid are set up while the last ones of the grid in front of it in the
// stream still run.  The kernels that are a whole call by themselves are launched so, and the attention kernel that follows
// a gather (measured, calls back to back: causal prefill of 2048 tokens 43.5 -> 41.5 us, head_dim 64 prefill 82.0 -> 79.7,
// decode step at 4096 tokens 10.25 -> 9.9; a pass over many short blocks gains nothing, and the chain gather -> partials ->
// merge lost 2 % with every kernel launched so).  In return such a kernel executes grid_wait() before it touches memory that
// others write: it returns when the grid in front has completed and its writes are visible.  Every block executes it before
// it ends, so that the completion of a grid implies that of all before it.  grid_go() lets a dependent start its set-up;
// a grid that is launched the plain way waits for the whole of its predecessor all the same.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launches in clusters of `cluster` blocks along x, as a programmatic dependent if asked to.  Never so while kernel timing
// is recording: the events around a launch must separate it from its neighbours.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, unsigned cluster, bool dependent,
                             cudaStream_t stream, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  cfg.attrs = attr;
  if (cluster > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = cluster;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  if (dependent && !timing_recording()) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  count_launch();
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// How a problem is cut, for the estimates by which a kernel is chosen.  They go by the heads of the whole problem, see
// AttnParams, and by the SMs of the GPU on which they were measured.
constexpr double kEstimateSms = 148;
struct CutSize {
  double heads, shards, q_shards, keys;  // (query head, sequence) pairs; KV shards, query shards; keys per KV shard
  double n_q, n_kv, first;               // first: position of the first query row
  bool causal;
  explicit CutSize(const AttnParams& p)
      : heads((double)p.rule_kv_heads * p.G * p.batch), shards(p.plan.n_kv_shards),
        q_shards(std::min(p.plan.n_q_shards, p.plan.n_q)), keys((double)p.plan.n_kv / p.plan.n_kv_shards), n_q(p.plan.n_q),
        n_kv(p.plan.n_kv), first(p.plan.q_pos_offset), causal(p.plan.causal != 0) {}
  // share of the keys that the query row at x n_q sees
  double seen_at(double x) const { return causal ? std::max(0.0, std::min(1.0, (first + x * n_q + 1) / n_kv)) : 1.0; }
  // the same for the last rows of tiles that do not cross shards, on average: rows ascend in a shard and spread over the sequence
  double seen_by_last(double tiles) const {
    const double per = std::max(1.0, tiles / q_shards), rows = n_q / q_shards;
    return seen_at((per + 1) / (2 * per) * rows / (rows + 1));
  }
  // tiles of `height` rows that do not cross shards (of equal size)
  double row_tiles(double height) const {
    const double least = std::floor(n_q / q_shards), longer = n_q - least * q_shards;
    return (q_shards - longer) * std::ceil(least / height) + longer * std::ceil((least + 1) / height);
  }
  // pieces of `width` keys in the visible prefix of a shard, on average
  double pieces(double seen, double width) const {
    const double all = std::ceil(keys / width);
    if (seen >= 1) return all;
    const double none = std::min(1.0, 2 * (1 - seen) / (keys + 1));
    return std::min(all, keys <= width ? 1 - none : seen * keys / width + 0.5);
  }
};
double rows_time(const AttnParams& p);         // attn_rows.cu
double tiles_time(const AttnParams& p);        // attn_simt.cu
double split_time(const AttnParams& p);        // attn_split.cu
double tc_partials_time(const AttnParams& p);  // attn_tc.cu, partials of several shards at head_dim 64

// Launchers; each returns a cudaError_t from the launch.
cudaError_t launch_attn_rows(const AttnParams& p, cascade_dtype_t dtype, cudaStream_t stream);
// the faster of attn_simt.cu and attn_rows.cu
cudaError_t launch_attn_simt(const AttnParams& p, cascade_dtype_t dtype, cudaStream_t stream);
// fp32, head_dim 64, at most 256 KV shards, on the tensor cores, and the scratch that it takes
cudaError_t launch_attn_split(const AttnParams& p, void* workspace, cudaStream_t stream);
size_t split_ws_bytes(const PlanDev& d, int batch, int Hkv);
// K or V rows [batch][kv_heads][rows][d] for the tensor-core kernel (strides in elements)
struct TcRows {
  const void* base;
  Strides strides;
};
bool tc_rows_loadable(const TcRows& r, int64_t n_rows, int64_t n_heads, int64_t batch);
// all keys of a query in one go, K and V in token order; rows from n_seen on are not looked at; k_gathered / v_gathered: the
// rows are written by a gather launched just before
cudaError_t launch_attn_tc(const AttnParams& p, const TcRows& k, const TcRows& v, int64_t n_seen, bool k_gathered,
                           bool v_gathered, cudaStream_t stream);
// the partials of every KV shard; k_sorted / v_sorted: shard-major copies, [batch][kv_head][n_kv][d] bf16
cudaError_t launch_attn_tc_partials(const AttnParams& p, const void* k_sorted, const void* v_sorted, cudaStream_t stream);
// Copies of K and V for the above, [batch][kv_head][n_kv][d]: shard-major, or with token_order as the rows are.
cudaError_t launch_gather_kv(const AttnParams& p, void* k_out, void* v_out, bool token_order, cudaStream_t stream);
// The same with the key rows turned (p.rope) on the way; null = not asked for.
struct RopeCopies {
  void *k_sorted, *k_tokens;  // keys in shard-major order, in token order
  void* v;                    // values, shard-major or in token order
  bool v_token_order;
  bool after_attention;  // made when the attention kernel in front is done, otherwise before it
};
cudaError_t launch_gather_kv_rope(const AttnParams& p, const RopeCopies& c, cudaStream_t stream);
cudaError_t launch_rope_table(int32_t n_positions, int32_t head_dim, double base, float2* table, cudaStream_t stream);
cudaError_t launch_rope_apply(cascade_dtype_t dtype, int32_t batch, int32_t n_rows, int32_t n_heads, int32_t head_dim,
                              const void* x, Strides xs, int32_t first_position, const float2* table, void* y, Strides ys,
                              cudaStream_t stream);
cudaError_t launch_decode(const AttnParams& p, cudaStream_t stream);
// decode of all shards with the post-pass in the same kernel; n_visible = keys the (longest) query row sees
cudaError_t launch_decode_fused(const AttnParams& p, const DecodeStep& step, int64_t n_visible, cudaStream_t stream);
// vis (n_vis values) and pair_class (n_cls) of a small plan written from the launch's own arguments
cudaError_t launch_plan_set(const PlanDev& d, const int32_t* vis, int n_vis, const uint8_t* pair_class, int n_cls,
                            cudaStream_t stream);
// number of keys of all shards that a query at position `pos` sees
int64_t visible_keys(const cascade_plan& pl, int map, int64_t pos);
// the fused decode of a checked call: cascade_attn_sharded, cascade_attn_decode_static
cudaError_t run_decode_fused(const cascade_plan& plan, const AttnParams& p, cudaStream_t stream);
// Fills a new plan's lists, inverses and (visible) vis and pair_class from the uploaded row lists, 16 or 32 bits an id.
cudaError_t launch_plan_fill(const PlanDev& d, const void* q_src, const void* kv_src, bool short_ids, bool visible,
                             cudaStream_t stream);
// vis and pair_class of a device plan recomputed for a new q_pos_offset (plans without kv_pos)
cudaError_t launch_plan_advance(const PlanDev& d, int32_t q_pos_offset, cudaStream_t stream);
cudaError_t launch_merge(const MergeParams& p, cascade_dtype_t dtype, cudaStream_t stream);
cudaError_t launch_merge_peers(const MergePeersParams& p, cascade_dtype_t dtype, cudaStream_t stream);

}  // namespace cascade
