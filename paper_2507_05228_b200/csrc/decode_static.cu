// Decode attention for callers that cannot provide or allocate scratch memory.
//
// cascade_attn_sharded asks for a caller-provided workspace for the decode step.  Some callers have none to give: an
// inference server whose cache manager has already claimed all free HBM, so a cudaMalloc at request time fails or fragments
// its pool; a latency-critical decode loop in which cudaMalloc / cudaFree would synchronise the whole device; a plug-in that
// is handed raw pointers and has no access to the host framework's allocator.  The fused decode kernel keeps the partials of
// the KV shards in distributed shared memory, so this entry point needs no scratch memory at all; the size limit of its
// interface (what a 16 MiB scratch array would hold) is kept.
#include <string.h>

#include "cascade_internal.cuh"

namespace cascade {
namespace {

constexpr size_t kScratchBytes = 16u << 20;  // the interface's limit: batch x KV shards x heads x 264 bytes

size_t round256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace
}  // namespace cascade

using namespace cascade;

extern "C" cascade_status_t cascade_attn_decode_static(const cascade_plan_t* plan, int32_t batch, int32_t n_heads,
                                                       int32_t n_kv_heads, float scale, const void* q,
                                                       cascade_strides_t q_strides, const void* k,
                                                       cascade_strides_t k_strides, const void* v,
                                                       cascade_strides_t v_strides, void* o_out,
                                                       cascade_strides_t o_strides, float* lse_out, void* stream) {
  constexpr int kHeadDim = 128;
  if (!plan || !q || !k || !v || !o_out) {
    set_error("cascade_attn_decode_static: null pointer");
    return CASCADE_ERR_INVALID_ARG;
  }
  if (!plan->dev_blob) {
    set_error("cascade_attn_decode_static: host-only plan");
    return CASCADE_ERR_INVALID_ARG;
  }
  if (batch < 1 || n_heads < 1 || n_kv_heads < 1 || (plan->dev.n_maps != 1 && plan->dev.n_maps != batch)) {
    set_error("cascade_attn_decode_static: bad batch or head counts");
    return CASCADE_ERR_INVALID_ARG;
  }
  if (!(scale > 0.f) || scale > 3.0e38f) {
    set_error("cascade_attn_decode_static: scale must be positive and finite");
    return CASCADE_ERR_INVALID_ARG;
  }
  const int G = n_kv_heads > 0 && n_heads % n_kv_heads == 0 ? n_heads / n_kv_heads : 0;
  if (plan->dev.n_q != 1 || !(G == 1 || G == 2 || G == 4 || G == 8)) {
    set_error("cascade_attn_decode_static: needs a plan with n_q == 1 and n_heads / n_kv_heads in {1,2,4,8} "
              "(bf16, head_dim 128)");
    return CASCADE_ERR_UNSUPPORTED;
  }
  auto misaligned = [](const void* p) { return ((uintptr_t)p & 15) != 0; };
  auto bad_strides = [](const cascade_strides_t& s) { return (s.batch % 8) || (s.token % 8) || (s.head % 8); };
  if (misaligned(q) || misaligned(k) || misaligned(v) || misaligned(o_out) || bad_strides(q_strides) ||
      bad_strides(k_strides) || bad_strides(v_strides) || bad_strides(o_strides)) {
    set_error("cascade_attn_decode_static: pointers and row strides must be 16-byte aligned");
    return CASCADE_ERR_INVALID_ARG;
  }
  if ((int64_t)batch > 65535) {
    set_error("cascade_attn_decode_static: batch exceeds 65535");
    return CASCADE_ERR_UNSUPPORTED;
  }
  const size_t rows = (size_t)batch * plan->dev.n_kv_shards * n_heads;  // one query row per sequence
  const size_t o_bytes = round256(rows * kHeadDim * sizeof(__nv_bfloat16));
  const size_t stat_bytes = round256(rows * sizeof(float));
  const size_t need = o_bytes + 2 * stat_bytes;
  if (need > kScratchBytes) {
    set_error("cascade_attn_decode_static: batch %d x %d KV shards x %d heads needs %zu bytes of scratch, the "
              "limit of this call is %zu; use cascade_attn_sharded with a workspace instead",
              batch, plan->dev.n_kv_shards, n_heads, need, kScratchBytes);
    return CASCADE_ERR_WORKSPACE;
  }
  AttnParams p;
  memset(&p, 0, sizeof(p));
  p.plan = plan->dev;
  p.q = q;
  p.k = k;
  p.v = v;
  p.qs = {q_strides.batch, q_strides.token, q_strides.head};
  p.ks = {k_strides.batch, k_strides.token, k_strides.head};
  p.vs = {v_strides.batch, v_strides.token, v_strides.head};
  p.batch = batch;
  p.H = n_heads;
  p.Hkv = n_kv_heads;
  p.G = G;
  p.d = kHeadDim;
  p.scale = scale;
  p.rule_kv_heads = n_kv_heads;
  p.fused = 1;
  p.o_out = o_out;
  p.os = {o_strides.batch, o_strides.token, o_strides.head};
  p.lse_out = lse_out;
  cudaError_t e = run_decode_fused(*plan, p, (cudaStream_t)stream);
  if (e != cudaSuccess) {
    set_error("cascade_attn_decode_static: decode launch: %s", cudaGetErrorString(e));
    return CASCADE_ERR_CUDA;
  }
  return CASCADE_OK;
}
