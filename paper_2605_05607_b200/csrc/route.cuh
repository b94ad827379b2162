// Top-k of one token by one warp (paper Sec. II-A: the gate network selects topk experts per token), shared by the top-k
// kernel and by the layout kernel of small batches.
#pragma once
#include "common.cuh"

namespace tcmoe {

// ------------------------------------------------------------------------------------------------
// Top-k: one warp per token.  Lane l holds experts l, l+32, ... (KPL of them) as order-preserving
// unsigned keys.  k rounds of: lane-local best -> warp max of the key -> warp min of the expert
// index among the lanes holding that key.  -0.0 is folded onto +0.0 and NaN onto -inf before
// ordering, so comparisons agree with IEEE "==" ties and never hang on NaN.
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t order_key(float v, bool& nonfinite) {
  uint32_t u = __float_as_uint(v);
  if ((u & 0x7F800000u) == 0x7F800000u) {
    nonfinite = true;
    if (u & 0x007FFFFFu) u = 0xFF800000u;  // NaN -> -inf
  }
  if ((u << 1) == 0) u = 0;                // -0.0 -> +0.0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_value(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o ^ 0x80000000u) : ~o);
}

// Lane j < k returns the j-th selected expert and its gate weight.
template <int KPL>
__device__ __forceinline__ void topk_token(const float* __restrict__ logits, const float* __restrict__ bias, long long bias_stride,
                                           int t, int E, int k, int score_fn, int lane, bool& nonfinite, uint32_t& my_e,
                                           float& my_w) {
  uint32_t key[KPL];
#pragma unroll
  for (int i = 0; i < KPL; ++i) {
    const int e = lane + 32 * i;
    if (e < E) {
      float v = __ldg(logits + (size_t)t * E + e);
      if (bias != nullptr) v = __fadd_rn(v, __ldg(bias + (size_t)t * bias_stride + e));
      key[i] = order_key(v, nonfinite);
    } else {
      key[i] = 0;  // below every real key (-inf maps to 0x007FFFFF)
    }
  }
  my_e = 0;              // lane j keeps the j-th selected expert and its key
  float my_key = 0.f;
  for (int j = 0; j < k; ++j) {
    uint32_t best = 0;
    int best_i = 0;
#pragma unroll
    for (int i = 0; i < KPL; ++i)
      if (key[i] > best) { best = key[i]; best_i = i; }  // strict: lowest i (lowest expert) wins ties
    const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, best);
    const uint32_t cand = (best == top) ? (uint32_t)(lane + 32 * best_i) : 0xFFFFFFFFu;
    const uint32_t win = __reduce_min_sync(0xFFFFFFFFu, cand);
    if ((int)(win & 31u) == lane) {
#pragma unroll
      for (int i = 0; i < KPL; ++i)
        if (i == (int)(win >> 5)) key[i] = 0;
    }
    if (lane == j) { my_e = win; my_key = key_value(top); }
  }
  // gate weights over the k selected keys (lanes 0..k-1)
  const float key0 = __shfl_sync(0xFFFFFFFFu, my_key, 0);
  float z = 0.f;
  if (lane < k) z = (score_fn == 0) ? expf(my_key - key0) : 1.f / (1.f + expf(-my_key));
  float sum = z;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, off);
  // Every lane divides, and a quotient of zero is a slow one: the other lanes take one of one (32768 tokens top-1 of 64 9.6 -> 8.4 us,
  // top-8 of 256 36.0 -> 35.0).
  my_w = (lane < k ? z : sum) / sum;
}

}  // namespace tcmoe
