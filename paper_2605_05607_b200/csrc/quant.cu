// bf16 -> E4M3 quantisation for the FP8 form of the expert FFN (paper Sec. V-A: the evaluated
// DeepSeek-V3 experts run FP8 GEMMs; format and scaling are this library's reading):
//   scale = fl32(max|v| / 448) over a row (activations) or over K for one (expert, output column)
//           (weights); 1 for an all-zero vector
//   code  = e4m3(fl32(v / scale)), round to nearest even, saturating at +-448
// Every step is a single fp32 operation, so a CPU restatement takes the same decisions.
#include "common.cuh"

#include <cuda_bf16.h>
#include <cuda_fp8.h>

namespace tcmoe {
namespace {

__device__ __forceinline__ uint8_t to_e4m3(float v, float scale) {
  return (uint8_t)__nv_cvt_float_to_fp8(__fdiv_rn(v, scale), __NV_SATFINITE, __NV_E4M3);
}
__device__ __forceinline__ float scale_of(float amax) { return amax == 0.f ? 1.f : __fdiv_rn(amax, 448.f); }

// Two codes at once, the low byte that of `a`.  fl32(v / scale) comes from the reciprocal, which the whole row shares, by
// Markstein's correction (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000 processor", IBM J. Res.
// Dev. 34, 1990): with inv = RN(1 / s) and q within an ulp of v / s, RN(q + (v - q s) * inv), the residual exact, is RN(v / s) as long
// as nothing leaves the normal range.  Values so small that the residual does round to code 0 either way.  (Taking the code
// where both ends of an error interval around v * inv agree was no faster than dividing: quotients of 8-bit significands
// tie exactly too often, and one lane's division stops its warp.)
__device__ __forceinline__ uint32_t to_e4m3_pair(float a, float b, float inv, float scale) {
  float qa = a * inv, qb = b * inv;
#pragma unroll
  for (int i = 0; i < 2; ++i) {   // the first step makes q faithful, the second is the one that rounds correctly
    qa = fmaf(fmaf(-qa, scale, a), inv, qa);
    qb = fmaf(fmaf(-qb, scale, b), inv, qb);
  }
  return __nv_cvt_float2_to_fp8x2(make_float2(copysignf(qa, a), copysignf(qb, b)),   // -0 stays -0
                                  __NV_SATFINITE, __NV_E4M3);
}
// WARPS warps per row (1, or the whole block of 4 for long rows; up to 2048 columns many rows take one warp each, few the block).  The row stays in registers between the maximum and the codes
// when it has at most KEEP vectors per lane; a longer one is read again.  cols % 8 == 0.  Bound by memory now, by the divisions
// before: 131072 rows of 1536 columns 152 -> 101 us (6.0 TB/s), 131072 of 4096 370 -> 281 (5.7 TB/s), 16384 of 4096, which stay in L2, 64 -> 37.
template <int KEEP, int WARPS>
__global__ void __launch_bounds__(WARPS == 1 ? 256 : WARPS * 32) quantize_rows_kernel(const uint4* __restrict__ src, uint2* __restrict__ dst,
                                                            float* __restrict__ scale, long long rows, int vec_per_row) {
  grid_dependency_sync();
  __shared__ float amax_s[WARPS];
  constexpr int LANES = WARPS * 32;
  const int lane = WARPS == 1 ? threadIdx.x & 31 : threadIdx.x;   // of the row's threads
  const long long rpb = blockDim.x / LANES;
  auto amax_of = [](const uint4& raw, float amax) {
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float2 f = __bfloat1622float2(p[q]);
      amax = fmaxf(amax, fmaxf(fabsf(f.x), fabsf(f.y)));
    }
    return amax;
  };
  for (long long r = blockIdx.x * rpb + (WARPS == 1 ? threadIdx.x >> 5 : 0); r < rows; r += (long long)gridDim.x * rpb) {
    const uint4* row = src + r * vec_per_row;
    uint4 keep[KEEP];
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < KEEP; ++i)
      keep[i] = lane + LANES * i < vec_per_row ? __ldg(row + lane + LANES * i) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int i = 0; i < KEEP; ++i) amax = amax_of(keep[i], amax);
#pragma unroll 1
    for (int v = lane + LANES * KEEP; v < vec_per_row; v += LANES) amax = amax_of(__ldg(row + v), amax);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, off));
    if (WARPS > 1) {
      __syncthreads();   // the last row's maxima have been read
      if ((lane & 31) == 0) amax_s[lane >> 5] = amax;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < WARPS; ++i) amax = fmaxf(amax, amax_s[i]);
    }
    const float sc = scale_of(amax);
    if (lane == 0) scale[r] = sc;
    uint2* out = dst + r * vec_per_row;
    if (!(sc >= 0x1p-80f && sc < 0x1p100f)) {   // the reciprocal or a residual could leave the normal range: divide
#pragma unroll 1
      for (int v = lane; v < vec_per_row; v += LANES) {
        const uint4 raw = __ldg(row + v);
        const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
        uint32_t w[2] = {0u, 0u};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 f = __bfloat1622float2(p[q]);
          w[q >> 1] |= ((uint32_t)to_e4m3(f.x, sc) | ((uint32_t)to_e4m3(f.y, sc) << 8)) << (16 * (q & 1));
        }
        out[v] = make_uint2(w[0], w[1]);
      }
      continue;
    }
    const float inv = __frcp_rn(sc);
    auto codes = [&](const uint4& raw) {
      const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
      uint32_t c[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 f = __bfloat1622float2(p[q]);
        c[q] = to_e4m3_pair(f.x, f.y, inv, sc);
      }
      return make_uint2(__byte_perm(c[0], c[1], 0x5410), __byte_perm(c[2], c[3], 0x5410));
    };
#pragma unroll
    for (int i = 0; i < KEEP; ++i)
      if (lane + LANES * i < vec_per_row) out[lane + LANES * i] = codes(keep[i]);
#pragma unroll 1
    for (int v = lane + LANES * KEEP; v < vec_per_row; v += LANES) out[v] = codes(__ldg(row + v));
  }
}

// Weights [E, K, N] (N contiguous) -> codes [E, N, K] (K contiguous) + scale [E, N].  One block
// per (expert, 32 output columns): pass 1 reduces max|w| over K per column, pass 2 quantises and
// transposes 32 x 32 tiles through shared memory.  A one-time preparation step.
__global__ void __launch_bounds__(256) quantize_weights_kernel(const __nv_bfloat16* __restrict__ w,
                                                               uint8_t* __restrict__ wq, float* __restrict__ scale,
                                                               int K, int N) {
  __shared__ float red[8][32];
  __shared__ float sc_s[32];
  __shared__ uint8_t tile[32][33];
  grid_dependency_sync();
  const int e = blockIdx.y, n0 = blockIdx.x * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // tx: column (pass 1 / tile load), ty: 0..7
  const __nv_bfloat16* we = w + (size_t)e * K * N;
  const int n = n0 + tx;
  float amax = 0.f;
  if (n < N)
    for (int k = ty; k < K; k += 8) amax = fmaxf(amax, fabsf(__bfloat162float(we[(size_t)k * N + n])));
  red[ty][tx] = amax;
  __syncthreads();
  if (ty == 0) {
    for (int i = 1; i < 8; ++i) amax = fmaxf(amax, red[i][tx]);
    const float sc = scale_of(amax);
    sc_s[tx] = sc;
    if (n < N) scale[(size_t)e * N + n] = sc;
  }
  __syncthreads();
  uint8_t* qe = wq + (size_t)e * N * K;
  for (int k0 = 0; k0 < K; k0 += 32) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {   // tile[k][n]
      const int k = k0 + ty + 8 * i;
      tile[ty + 8 * i][tx] = (k < K && n < N) ? to_e4m3(__bfloat162float(we[(size_t)k * N + n]), sc_s[tx]) : 0;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i) {   // write rows of [n][k0 .. k0+31]
      const int nn = n0 + ty + 8 * i, k = k0 + tx;
      if (nn < N && k < K) qe[(size_t)nn * K + k] = tile[tx][ty + 8 * i];
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_quantize_rows(const void* src, long long rows, int cols, void* dst, float* scale, cudaStream_t st) {
  if (rows <= 0 || cols <= 0) return cudaSuccess;
  const long long cap = (long long)sm_count() * 16;
  const uint4* in = static_cast<const uint4*>(src);
  uint2* out = static_cast<uint2*>(dst);
  auto grid = [&](long long n) { return (unsigned)(n > cap ? cap : n); };
  if (cols <= 512) return launch_pdl(quantize_rows_kernel<2, 1>, grid((rows + 7) / 8), 256, 0, st, in, out, scale, rows, cols / 8);
  // six vectors per lane where three do: 16384 rows of 768 columns 10.2 us, three 8.0
  if (cols <= 768) return launch_pdl(quantize_rows_kernel<3, 1>, grid((rows + 7) / 8), 256, 0, st, in, out, scale, rows, cols / 8);
  if (cols <= 1536) return launch_pdl(quantize_rows_kernel<6, 1>, grid((rows + 7) / 8), 256, 0, st, in, out, scale, rows, cols / 8);
  // us with a block / a warp per row: 16384 of 1544 columns 24.4 / 17.1, 4096 of 1792 6.8 / 5.7, 300 of 2048 2.2 / 2.6
  if (cols <= 2048 && rows >= 8ll * sm_count()) return launch_pdl(quantize_rows_kernel<8, 1>, grid((rows + 7) / 8), 256, 0, st, in, out, scale, rows, cols / 8);
  if (cols <= 4096) return launch_pdl(quantize_rows_kernel<4, 4>, grid(rows), 128, 0, st, in, out, scale, rows, cols / 8);
  return launch_pdl(quantize_rows_kernel<8, 4>, grid(rows), 128, 0, st, in, out, scale, rows, cols / 8);   // registers: 8192 columns
}

cudaError_t launch_quantize_weights(const void* w, int E, int K, int N, void* wq, float* scale, cudaStream_t st) {
  if (E <= 0 || K <= 0 || N <= 0) return cudaSuccess;
  return launch_pdl(quantize_weights_kernel, dim3((N + 31) / 32, E), 256, 0, st,
                    static_cast<const __nv_bfloat16*>(w), static_cast<uint8_t*>(wq), scale, K, N);
}

}  // namespace tcmoe
