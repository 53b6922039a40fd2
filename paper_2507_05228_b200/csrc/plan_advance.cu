// cascade_plan_advance on the device: the visible-prefix lengths and pair classes of a plan for a new position of
// its first query row, recomputed from the plan's own index arrays (appendix "Cost Optimizations", Caching: the
// cache grows by one row per generated token, the shard lists do not change).  No host work and no upload per call;
// used for plans with more than a few hundred (row, shard) entries, where the host pass would cost more than a launch;
// cascade_shard_plan fills the two arrays of a new plan the same way.
#include <string.h>

#include "cascade_internal.cuh"

namespace cascade {

namespace {

// Number of keys of shard k (positions ascending in kv_idx) at or before the position of query slot r of map mp.
__device__ __forceinline__ int32_t visible_prefix(const PlanDev& d, int32_t q_pos_offset, int mp, int r, int k) {
  const int32_t* ko = d.kv_off + (size_t)mp * (d.n_kv_shards + 1);
  const int32_t begin = ko[k], len = ko[k + 1] - begin;
  if (!d.causal) return len;
  const int64_t pos = (int64_t)d.q_idx[(size_t)mp * d.n_q + r] + q_pos_offset;
  if (pos < 0) return 0;
  if (pos >= d.n_kv) return len;
  const int32_t* list = d.kv_idx + (size_t)mp * d.n_kv + begin;
  int lo = 0, hi = len;  // first entry greater than pos
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (list[mid] <= (int32_t)pos) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// One thread per entry: first vis[map][r][k], then EMPTY / PARTIAL / FULL per (query shard, KV shard) from the prefix
// lengths of the shard's first and last row (rows ascend in position, so the first row has the shortest prefix and the
// last the longest; both are searched for again here, so that one launch does everything: the launch is what costs).
__global__ void plan_advance_kernel(PlanDev d, int32_t q_pos_offset, int32_t* __restrict__ vis,
                                    uint8_t* __restrict__ pair_class) {
  grid_go();
  grid_wait();
  const int J = d.n_q_shards, P = d.n_kv_shards;
  const int64_t n_vis = (int64_t)d.n_maps * d.n_q * P, n = n_vis + (int64_t)d.n_maps * J * P;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = t < n_vis ? t : t - n_vis;
    const int k = (int)(e % P);
    const int64_t row = e / P;
    if (t < n_vis) {
      vis[t] = visible_prefix(d, q_pos_offset, (int)(row / d.n_q), (int)(row % d.n_q), k);
      continue;
    }
    const int mp = (int)(row / J), j = (int)(row % J);
    const int32_t* qo = d.q_off + (size_t)mp * (J + 1);
    const int32_t* ko = d.kv_off + (size_t)mp * (P + 1);
    const int len = ko[k + 1] - ko[k];
    uint8_t cls = CASCADE_PAIR_EMPTY;
    if (qo[j + 1] > qo[j] && len > 0) {
      const int lo = visible_prefix(d, q_pos_offset, mp, qo[j], k);
      const int hi = visible_prefix(d, q_pos_offset, mp, qo[j + 1] - 1, k);
      cls = hi == 0 ? CASCADE_PAIR_EMPTY : (lo == len ? CASCADE_PAIR_FULL : CASCADE_PAIR_PARTIAL);
    }
    pair_class[e] = cls;
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

cudaError_t launch_plan_advance(const PlanDev& d, int32_t q_pos_offset, cudaStream_t stream) {
  const int64_t n = (int64_t)d.n_maps * (d.n_q + d.n_q_shards) * d.n_kv_shards;
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((n + threads - 1) / threads, 8 * 1024);
  // a dependent too: the chain plan -> attention of a 512-token chunk at 8192 keys 70.3 -> 68.8 us back to back
  return launch_dependent(plan_advance_kernel, dim3(blocks), threads, 0, 1, true, stream, d, q_pos_offset,
                          const_cast<int32_t*>(d.vis), const_cast<uint8_t*>(d.pair_class));
}

}  // namespace cascade
