// moe_route: the router ahead of the plan step -- per token the k experts with the largest logits
// and the router weights softmax(logits) renormalised over those k (the router step of the MoE
// module of Section 2.1 of the paper; the paper does not fix the arithmetic, this is the
// softmax -> top-k -> renormalise form of the seeded workloads).
//
// One warp per token.  Each lane holds its share of the logits in registers as order-preserving
// unsigned keys (E <= 1024); k rounds pick the experts in order of decreasing logit, ties to the lower
// expert id, which is the order of decreasing softmax probability: one warp-wide integer maximum over
// the keys, one warp-wide minimum over the ids that hold it.  The weights need no sum over
// all E experts: exp(z_j - z_max) / sum over the chosen k of the same, the common denominator
// cancels.  No workspace, no context.
//
// Bound by instruction issue (8192 tokens x 256 experts: 8.4 MB of logits, 1.3 us at the HBM copy rate).  A lane holds
// 8 keys where E <= 256 and 32 beyond: a kernel that always walked 32 and found the maximum by five rounds
// of float and id shuffles took 41 us there and 6.7 us for one token; this one 14 us and 2.9 us.
#include "moe_dev.cuh"

namespace moe {

constexpr int kRouteMaxE = 1024;
constexpr int kRouteWarps = 8;

// unsigned order = float order (-0 counts as +0); 0 is below every float: "no candidate"
__device__ __forceinline__ unsigned float_key(float v) {
  const unsigned u = __float_as_uint(v + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned key) {
  return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key);
}

// kPer: keys per lane.  kVec: rows are 16-byte aligned and a lane loads four neighbouring logits at once.
template <int kPer, bool kVec>
__global__ void __launch_bounds__(kRouteWarps * 32) route_kernel(const float* __restrict__ logits, int T, int E, int k,
                                                                 int* __restrict__ ids, float* __restrict__ w) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kRouteWarps + warp;
  grid_dep_wait();
  if (t >= T) return;
  const float* z = logits + (size_t)t * E;
  unsigned key[kPer];                      // expert of key i: see id_of
  const auto id_of = [lane](int i) { return kVec ? 128 * (i / 4) + 4 * lane + i % 4 : lane + 32 * i; };
  if (kVec) {
#pragma unroll
    for (int i = 0; i < kPer; i += 4) {
      const int e = id_of(i);
      const float4 v = e < E ? *reinterpret_cast<const float4*>(z + e) : make_float4(0.f, 0.f, 0.f, 0.f);
      key[i] = e < E ? float_key(v.x) : 0u;
      key[i + 1] = e < E ? float_key(v.y) : 0u;
      key[i + 2] = e < E ? float_key(v.z) : 0u;
      key[i + 3] = e < E ? float_key(v.w) : 0u;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kPer; ++i) key[i] = id_of(i) < E ? float_key(z[id_of(i)]) : 0u;
  }
  unsigned my_key = 0;                     // lane j keeps the j-th pick (k <= 32)
  int my_id = 0;
  for (int j = 0; j < k; ++j) {
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) m = max(m, key[i]);
    m = __reduce_max_sync(0xffffffffu, m);
    unsigned id = 0xffffffffu;
#pragma unroll
    for (int i = kPer - 1; i >= 0; --i)
      if (key[i] == m) id = (unsigned)id_of(i);
    id = __reduce_min_sync(0xffffffffu, id);
#pragma unroll
    for (int i = 0; i < kPer; ++i)
      if ((unsigned)id_of(i) == id) key[i] = 0u;
    if (lane == j) { my_key = m; my_id = (int)id; }
  }
  const float zmax = key_float(__shfl_sync(0xffffffffu, my_key, 0));
  const float mine = lane < k ? expf(key_float(my_key) - zmax) : 0.f;
  float sum = 0.f;
  for (int j = 0; j < k; ++j) sum += __shfl_sync(0xffffffffu, mine, j);
  if (lane < k) {
    ids[(size_t)t * k + lane] = my_id;
    w[(size_t)t * k + lane] = mine / sum;
  }
}

}  // namespace moe

extern "C" int moe_route(const float* logits, int32_t n_tokens, int32_t n_experts, int32_t top_k,
                         int32_t* topk_ids, float* topk_w, void* stream) {
  using namespace moe;
  if (n_tokens < 0 || n_experts < 1 || n_experts > kRouteMaxE || top_k < 1 || top_k > 32 || top_k > n_experts)
    return MOE_EINVAL;
  if (n_tokens == 0) return MOE_OK;
  if (!logits || !topk_ids || !topk_w) return MOE_EINVAL;
  const int blocks = (n_tokens + kRouteWarps - 1) / kRouteWarps;
  const bool vec = n_experts % 4 == 0 && (reinterpret_cast<uintptr_t>(logits) & 15) == 0;
  const bool small = n_experts <= 256;
  auto* kernel = small ? (vec ? route_kernel<8, true> : route_kernel<8, false>)
                       : (vec ? route_kernel<32, true> : route_kernel<32, false>);
  return launch_after(kernel, blocks, kRouteWarps * 32, 0, static_cast<cudaStream_t>(stream), logits, n_tokens, n_experts, top_k,
                      topk_ids, topk_w) == cudaSuccess ? MOE_OK : MOE_ECUDA;
}
