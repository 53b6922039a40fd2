// cascade_plan_advance on the device: the visible-prefix lengths and pair classes of a plan for a new position of
// its first query row, recomputed from the plan's own index arrays (appendix "Cost Optimizations", Caching: the
// cache grows by one row per generated token, the shard lists do not change).  No host work and no upload per call;
// used for plans with more than a few hundred (row, shard) entries, where the host pass would cost more than a launch;
// cascade_shard_plan fills the device arrays of a new plan the same way, from the sorted row lists.
#include <string.h>

#include "cascade_internal.cuh"

namespace cascade {

namespace {

// Number of keys of shard k (positions ascending in kv_idx) at or before the position of query slot r of map mp.
template <typename T>
__device__ __forceinline__ int32_t visible_prefix(const PlanDev& d, const T* q_idx, const T* kv_idx, int32_t q_pos_offset,
                                                  int mp, int r, int k) {
  const int32_t* ko = d.kv_off + (size_t)mp * (d.n_kv_shards + 1);
  const int32_t begin = ko[k], len = ko[k + 1] - begin;
  if (!d.causal) return len;
  const int64_t pos = (int64_t)q_idx[(size_t)mp * d.n_q + r] + q_pos_offset;
  if (pos < 0) return 0;
  if (pos >= d.n_kv) return len;
  const T* list = kv_idx + (size_t)mp * d.n_kv + begin;
  // First entry greater than pos.  Each step reads seven entries at once and keeps an eighth of the range: what bounds
  // these kernels is the chain of dependent reads, 4 of them for 512 keys where halving makes 10.
  int lo = 0, n = len;
  while (n > 0) {
    const int step = n / 8 + 1;
    int below = 0;
#pragma unroll
    for (int i = 1; i < 8; ++i) {
      const int at = i * step - 1;
      below += at < n && (int32_t)list[lo + at] <= (int32_t)pos;
    }
    lo += below * step;
    n = min(n - below * step, step - 1);
  }
  return lo;
}

// The threads that visible_entry takes, a whole number of warps: one for a group of kWarpRows query slots (over all maps) and
// kWarpShards KV shards, then two threads for each pair of a query shard and a KV shard.
constexpr int kWarpShards = 4, kWarpRows = 32 / kWarpShards;
struct VisThreads {
  int64_t vis, all;
};
__host__ __device__ __forceinline__ VisThreads vis_threads(const PlanDev& d) {
  const int64_t vis = ((int64_t)d.n_maps * d.n_q + kWarpRows - 1) / kWarpRows *
                      ((d.n_kv_shards + kWarpShards - 1) / kWarpShards) * 32;
  return {vis, vis + ((int64_t)d.n_maps * d.n_q_shards * d.n_kv_shards * 2 + 31) / 32 * 32};
}

// Thread t's entry of vis[map][r][k] or, after those, its half of EMPTY / PARTIAL / FULL per (query shard, KV shard), from the
// prefix lengths of the shard's first and last row (rows ascend in position, so the first row has the shortest prefix and the
// last the longest; both are searched for again here, a thread each, so that one launch does everything: the launch is what
// costs).  Called by whole warps.  The lanes of a warp search few shards for neighbouring rows, so most of their reads are of
// the same lines, and write 16 bytes of a row.
// Measured back to back, 16 shards: 512 rows at 8192 keys 4.9 -> 3.3 us (halving, a thread per entry, shards first -> this), 1024
// at 16384 5.3 -> 3.7, 4096 at 4096 4.9 -> 5.0; 16384 rows at 32768 keys, 32 shards, 20.5 -> 11.6.  Sixteenths: 3.6, 4.1, 7.9
// and 16.0 with one shard a warp; eighths with one shard a warp 3.2, 3.6, 5.2 and 12.0, with eight 3.3, 3.7, 6.2 and 13.0.
template <typename T>
__device__ __forceinline__ void visible_entry(const PlanDev& d, const T* q_idx, const T* kv_idx, int32_t q_pos_offset, int64_t t,
                                              int64_t n_vis, int32_t* __restrict__ vis, uint8_t* __restrict__ pair_class) {
  const int J = d.n_q_shards, P = d.n_kv_shards;
  if (t < n_vis) {
    // 32-bit divisions: those of 64 bits take as long as a read
    const uint32_t warp = (uint32_t)(t / 32), across = (P + kWarpShards - 1) / kWarpShards;
    const int k = (int)(warp % across) * kWarpShards + (int)(t % kWarpShards);
    const int64_t row = (int64_t)(warp / across) * kWarpRows + t % 32 / kWarpShards;
    if (k < P && row < (int64_t)d.n_maps * d.n_q) {
      const int mp = d.n_maps == 1 ? 0 : (int)(row / d.n_q);
      vis[row * P + k] = visible_prefix(d, q_idx, kv_idx, q_pos_offset, mp, (int)(row - (int64_t)mp * d.n_q), k);
    }
    return;
  }
  const uint32_t e = (uint32_t)((t - n_vis) / 2);
  const bool last = t & 1, valid = e < (int64_t)d.n_maps * J * P;
  int seen = 0, len = 0;
  if (valid) {
    const int k = (int)(e % P), at = (int)(e / P), mp = at / J, j = at % J;
    const int32_t* qo = d.q_off + (size_t)mp * (J + 1);
    const int32_t* ko = d.kv_off + (size_t)mp * (P + 1);
    const int first = qo[j], end = qo[j + 1];
    if (end > first) len = ko[k + 1] - ko[k];
    if (len > 0) seen = visible_prefix(d, q_idx, kv_idx, q_pos_offset, mp, last ? end - 1 : first, k);
  }
  const int other = __shfl_xor_sync(0xffffffffu, seen, 1);  // (even lanes write: the last row's)
  if (valid && !last)
    pair_class[e] = other == 0 ? CASCADE_PAIR_EMPTY : (seen == len ? CASCADE_PAIR_FULL : CASCADE_PAIR_PARTIAL);
}

// One thread per entry, two per pair.  128 a block measured faster than 256 (3.6 against 4.2 us at 512 rows, 16 shards).
__global__ void plan_advance_kernel(PlanDev d, int32_t q_pos_offset, int32_t* __restrict__ vis,
                                    uint8_t* __restrict__ pair_class) {
  grid_go();
  grid_wait();
  const VisThreads n = vis_threads(d);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n.all; t += (int64_t)gridDim.x * blockDim.x)
    visible_entry(d, d.q_idx, d.kv_idx, q_pos_offset, t, n.vis, vis, pair_class);
}

// The arrays of a new plan that follow from its row lists kv_src and q_src (ids of T, as they were uploaded): the lists
// themselves, their inverses, the shard of every K/V slot and, unless the host has them (n_visible = 0), vis and pair_class.
// One thread per entry of each, those of visible_entry first.
template <typename T>
__global__ void plan_fill_kernel(PlanDev d, const T* __restrict__ q_src, const T* __restrict__ kv_src, int64_t n_vis,
                                 int64_t n_visible) {
  const int64_t n_q = (int64_t)d.n_maps * d.n_q, n_kv = (int64_t)d.n_maps * d.n_kv, n = n_visible + n_q + n_kv;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    if (t < n_visible) {
      visible_entry(d, q_src, kv_src, d.q_pos_offset, t, n_vis, const_cast<int32_t*>(d.vis),
                    const_cast<uint8_t*>(d.pair_class));
    } else if (t < n_visible + n_q) {
      const int64_t e = t - n_visible, first = e / d.n_q * d.n_q;  // entry, and the first entry of its map
      const int32_t row = q_src[e];
      const_cast<int32_t*>(d.q_idx)[e] = row;
      const_cast<int32_t*>(d.q_inv)[first + row] = (int32_t)(e - first);
    } else {
      const int64_t e = t - n_visible - n_q, mp = e / d.n_kv, first = mp * d.n_kv;
      const int32_t row = kv_src[e], slot = (int32_t)(e - first);
      const int32_t* off = d.kv_off + mp * (d.n_kv_shards + 1);
      int lo = 0, hi = d.n_kv_shards;  // last shard that starts at or before the slot
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= slot) lo = mid;
        else hi = mid;
      }
      const_cast<int32_t*>(d.kv_idx)[e] = row;
      const_cast<int32_t*>(d.kv_inv)[first + row] = slot;
      const_cast<int32_t*>(d.kv_slot_shard)[e] = lo;
    }
  }
}

// The same arrays of a plan with few entries, computed on the host and carried by the launch itself (two copies from pageable
// memory cost the caller 5 us, this 2 us).
struct PlanSetArgs {
  int32_t vis[kMaxGivenVis];
  uint8_t pair_class[kMaxGivenVis];
};
__global__ void __launch_bounds__(kMaxGivenVis) plan_set_kernel(const __grid_constant__ PlanSetArgs a, int n_vis, int n_cls,
                                                                int32_t* vis, uint8_t* pair_class) {
  grid_go();
  grid_wait();
  const int t = threadIdx.x;
  if (t < n_vis) vis[t] = a.vis[t];
  if (t < n_cls) pair_class[t] = a.pair_class[t];
}

}  // namespace

cudaError_t launch_plan_set(const PlanDev& d, const int32_t* vis, int n_vis, const uint8_t* pair_class, int n_cls,
                            cudaStream_t stream) {
  PlanSetArgs a;
  memcpy(a.vis, vis, (size_t)n_vis * 4);
  memcpy(a.pair_class, pair_class, (size_t)n_cls);
  return launch_dependent(plan_set_kernel, dim3(1), kMaxGivenVis, 0, 1, true, stream, a, n_vis, n_cls,
                          const_cast<int32_t*>(d.vis), const_cast<uint8_t*>(d.pair_class));
}

cudaError_t launch_plan_fill(const PlanDev& d, const void* q_src, const void* kv_src, bool short_ids, bool visible,
                             cudaStream_t stream) {
  const int64_t n_vis = vis_threads(d).vis;
  const int64_t n_visible = visible ? vis_threads(d).all : 0;
  const int64_t n = n_visible + (int64_t)d.n_maps * ((int64_t)d.n_q + d.n_kv);
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 8 * 1024);
  if (short_ids)
    plan_fill_kernel<<<blocks, threads, 0, stream>>>(d, static_cast<const uint16_t*>(q_src),
                                                     static_cast<const uint16_t*>(kv_src), n_vis, n_visible);
  else
    plan_fill_kernel<<<blocks, threads, 0, stream>>>(d, static_cast<const int32_t*>(q_src),
                                                     static_cast<const int32_t*>(kv_src), n_vis, n_visible);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_plan_advance(const PlanDev& d, int32_t q_pos_offset, cudaStream_t stream) {
  const int64_t n = vis_threads(d).all;
  const int threads = 128;  // spread over the SMs: 512 rows in 16 shards are 8704 threads
  const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 8 * 1024);
  // a dependent too: the chain plan -> attention of a 512-token chunk at 8192 keys 70.3 -> 68.8 us back to back
  return launch_dependent(plan_advance_kernel, dim3(blocks), threads, 0, 1, true, stream, d, q_pos_offset,
                          const_cast<int32_t*>(d.vis), const_cast<uint8_t*>(d.pair_class));
}

}  // namespace cascade
