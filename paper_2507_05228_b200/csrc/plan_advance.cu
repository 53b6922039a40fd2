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
  int lo = 0, hi = len;  // first entry greater than pos
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if ((int32_t)list[mid] <= (int32_t)pos) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Entry t of vis[map][r][k], or after those EMPTY / PARTIAL / FULL per (query shard, KV shard) from the prefix lengths of the
// shard's first and last row (rows ascend in position, so the first row has the shortest prefix and the last the longest;
// both are searched for again here, so that one launch does everything: the launch is what costs).
template <typename T>
__device__ __forceinline__ void visible_entry(const PlanDev& d, const T* q_idx, const T* kv_idx, int32_t q_pos_offset, int64_t t,
                                              int64_t n_vis, int32_t* __restrict__ vis, uint8_t* __restrict__ pair_class) {
  const int J = d.n_q_shards, P = d.n_kv_shards;
  const int64_t e = t < n_vis ? t : t - n_vis;
  const int k = (int)(e % P);
  const int64_t row = e / P;
  if (t < n_vis) {
    vis[t] = visible_prefix(d, q_idx, kv_idx, q_pos_offset, (int)(row / d.n_q), (int)(row % d.n_q), k);
    return;
  }
  const int mp = (int)(row / J), j = (int)(row % J);
  const int32_t* qo = d.q_off + (size_t)mp * (J + 1);
  const int32_t* ko = d.kv_off + (size_t)mp * (P + 1);
  const int len = ko[k + 1] - ko[k];
  uint8_t cls = CASCADE_PAIR_EMPTY;
  if (qo[j + 1] > qo[j] && len > 0) {
    const int lo = visible_prefix(d, q_idx, kv_idx, q_pos_offset, mp, qo[j], k);
    const int hi = visible_prefix(d, q_idx, kv_idx, q_pos_offset, mp, qo[j + 1] - 1, k);
    cls = hi == 0 ? CASCADE_PAIR_EMPTY : (lo == len ? CASCADE_PAIR_FULL : CASCADE_PAIR_PARTIAL);
  }
  pair_class[e] = cls;
}

// One thread per entry.
__global__ void plan_advance_kernel(PlanDev d, int32_t q_pos_offset, int32_t* __restrict__ vis,
                                    uint8_t* __restrict__ pair_class) {
  grid_go();
  grid_wait();
  const int64_t n_vis = (int64_t)d.n_maps * d.n_q * d.n_kv_shards;
  const int64_t n = n_vis + (int64_t)d.n_maps * d.n_q_shards * d.n_kv_shards;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    visible_entry(d, d.q_idx, d.kv_idx, q_pos_offset, t, n_vis, vis, pair_class);
}

// The arrays of a new plan that follow from its row lists kv_src and q_src (ids of T, as they were uploaded): the lists
// themselves, their inverses, the shard of every K/V slot and, unless the host has them (n_visible = 0), vis and pair_class.
// One thread per entry of each.
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
  const int64_t n_vis = (int64_t)d.n_maps * d.n_q * d.n_kv_shards;
  const int64_t n_visible = visible ? n_vis + (int64_t)d.n_maps * d.n_q_shards * d.n_kv_shards : 0;
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
  const int64_t n = (int64_t)d.n_maps * (d.n_q + d.n_q_shards) * d.n_kv_shards;
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 8 * 1024);
  // a dependent too: the chain plan -> attention of a 512-token chunk at 8192 keys 70.3 -> 68.8 us back to back
  return launch_dependent(plan_advance_kernel, dim3(blocks), threads, 0, 1, true, stream, d, q_pos_offset,
                          const_cast<int32_t*>(d.vis), const_cast<uint8_t*>(d.pair_class));
}

}  // namespace cascade
