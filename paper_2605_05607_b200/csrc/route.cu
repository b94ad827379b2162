// Routing of the MoE layer (paper Sec. II-A: the gate network selects topk experts per token); the
// gate logits themselves are computed in gate_gemm.cu.
//   topk_kernel : key = logit + bias; k largest keys per token ordered by
//                 (key descending, expert index ascending); gate weights over the k keys
#include "route.cuh"

#include <cuda_bf16.h>

namespace tcmoe {

template <int KPL>
__global__ void __launch_bounds__(256) topk_kernel(const float* __restrict__ logits, const float* __restrict__ bias,
                                                   long long bias_stride, int32_t* __restrict__ topk_idx,
                                                   float* __restrict__ topk_w, int T, int E, int k, int score_fn,
                                                   int32_t* status, uint32_t* clear, size_t clear_words) {
  grid_dependency_sync();
  // optional side job for the fused layer: zero the membership bitmasks of the layout builder that
  // runs next, so that no memset sits between this kernel and it
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < clear_words; i += (size_t)gridDim.x * blockDim.x)
    clear[i] = 0u;
  const int lane = threadIdx.x & 31;
  const int warps_per_block = blockDim.x >> 5;
  bool nonfinite = false;
  for (int t = blockIdx.x * warps_per_block + (threadIdx.x >> 5); t < T; t += gridDim.x * warps_per_block) {
    uint32_t my_e;
    float my_w;
    topk_token<KPL>(logits, bias, bias_stride, t, E, k, score_fn, lane, nonfinite, my_e, my_w);
    if (lane < k) {
      topk_idx[(size_t)t * k + lane] = (int32_t)my_e;
      topk_w[(size_t)t * k + lane] = my_w;
    }
  }
  if (__any_sync(0xFFFFFFFFu, nonfinite) && lane == 0) atomicOr(&status[ST_WARN], WARN_NONFINITE_LOGIT);
}

cudaError_t launch_topk(const Shape& s, const float* logits, const float* bias, int64_t bias_stride,
                        int32_t* topk_idx, float* topk_w, int32_t* status, cudaStream_t st, uint32_t* clear,
                        size_t clear_words) {
  if (s.T == 0) return cudaSuccess;
  const int warps = 8;
  int blocks = (s.T + warps - 1) / warps;
  const int cap = sm_count() * 8;
  if (blocks > cap) blocks = cap;
  const int kpl = (s.E + 31) / 32;
  ProfileScope prof(KID_TOPK, st);
#define TCMOE_TOPK(KPL)                                                                                      \
  launch_pdl(topk_kernel<KPL>, blocks, warps * 32, 0, st, logits, bias, (long long)bias_stride, topk_idx, topk_w, \
             s.T, s.E, s.k, s.score_fn, status, clear, clear_words)
  if (kpl <= 1) return TCMOE_TOPK(1);
  if (kpl <= 2) return TCMOE_TOPK(2);
  if (kpl <= 4) return TCMOE_TOPK(4);
  if (kpl <= 8) return TCMOE_TOPK(8);
  if (kpl <= 16) return TCMOE_TOPK(16);
  return TCMOE_TOPK(32);
#undef TCMOE_TOPK
}

}  // namespace tcmoe
