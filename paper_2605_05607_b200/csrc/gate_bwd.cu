// Gradient that reaches the gate network (paper Sec. II-A: the gate picks the topk experts of a token and weighs
// their outputs; Sec. VI-A evaluates training).  The SELECTION is held fixed; the gate weights are functions of the
// router keys  key[t, e] = x[t] . w_gate[:, e] + bias[t, e]:
//     y[t] = sum_j w[t, j] * FFN_{e_j}(x[t]),   w[t, :] = softmax (or renormalised sigmoid) of key[t, e_0 .. e_{k-1}]
// With L = sum(dy * y):
//     g[t, j]    = w[t, j] * dL/dw[t, j] = w[t, j] * dy[t] . FFN_{e_j}(x[t])
//     dkey[t, j] = (g[t, j] - w[t, j] * sum_i g[t, i]) * c[t, j],     c = 1 (softmax),  1 - sigmoid(key[t, j]) (sigmoid)
//     dw_gate    = x^T . dlogits,    dx[t] += sum_j dkey[t, j] * w_gate[:, e_j]
// (dkey follows from the quotient rule with w_j = s_j / sum_i s_i; no division is left in either form.)
//
// The expert part of the backward pass (bwd.cu) has just produced, in the padded row space of its workspace,
// h (the recomputed SwiGLU output of every pair) and dH = (w * dy) . W2^T.  Their row-wise dot product is
//     h[r] . dH[r] = w_r * (h[r] . W2) . dy[t_r] = g  of the pair in row r,
// so dL/dw costs no GEMM; the backward SwiGLU epilogue, which holds both, leaves its sums over 64 columns each.  dw_gate is a weighted sum of each expert's rows of
// xs (also still in the workspace), dx gets k rows of the transposed gate weight per token.
//
// Sequence (one stream): sums of the row dots -> per-token key gradients -> partial sums of dw_gate per 128-row tile -> dw_gate (tiles in
// ascending order: deterministic, no atomics) and the transpose of w_gate -> dx update.
#include "common.cuh"

#include <cuda_bf16.h>

namespace tcmoe {
namespace {

// g_row[r] = h[r] . dH[r] for the rows in use (r < poff[E]): the partial sums that the recomputed GEMM-1 left per 64 columns
// (a pass over both buffers for it took 79 us on 65536 rows of f = 1536).
__global__ void __launch_bounds__(256) gate_rowdot_kernel(const float* __restrict__ row_dots, int parts, long long ld,
                                                          const int32_t* __restrict__ poff, float* __restrict__ g_row, int E) {
  grid_dependency_sync();
  const int rows = __ldg(poff + E);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int q = 0; q < parts; ++q) s += __ldcs(row_dots + (size_t)q * ld + r);
    g_row[r] = s;
  }
}

// Key gradients of a token's k pairs, one lane each (1 << shift lanes per token, k rounded up to a power of two, so that their number can pass
// 2^31 where that of the pairs does not); written per pair (dkey) and in place per padded row (g_row).  Latency of two dependent reads; a thread per token walked its slots one after the other (8192 tokens
// top-8 22 -> 5 us; the sums have the same order).
__global__ void __launch_bounds__(256) gate_route_bwd_kernel(const int32_t* __restrict__ topk_idx,
                                                             const float* __restrict__ topk_w,
                                                             const int32_t* __restrict__ pair_prow,
                                                             const float* __restrict__ logits,
                                                             const float* __restrict__ bias, long long bias_stride,
                                                             float* g_row, float* __restrict__ dkey, int T, int E, int k,
                                                             int sigmoid, int n_rows, int shift) {
  grid_dependency_sync();
  const long long at = (long long)blockIdx.x * blockDim.x + threadIdx.x, t = at >> shift;
  const int width = 1 << shift, j = (int)at & (width - 1);
  const bool slot = t < T && j < k;
  const size_t pair = (size_t)t * k + j;
  const int r = slot ? __ldg(pair_prow + pair) : -1;
  const bool live = r >= 0 && r < n_rows;
  const float g = live ? g_row[r] : 0.f;
  float dot = 0.f;   // ascending slots
  for (int i = 0; i < k; ++i) dot += __shfl_sync(0xFFFFFFFFu, g, i, width);
  float v = 0.f;
  if (live) {
    v = g - __ldg(topk_w + pair) * dot;
    if (sigmoid) {
      const int e = __ldg(topk_idx + pair);
      float key = __ldg(logits + (size_t)t * E + e);
      if (bias != nullptr) key += __ldg(bias + (size_t)t * bias_stride + e);
      v *= 1.f - 1.f / (1.f + __expf(-key));
    }
    g_row[r] = v;   // from here on g_row holds the key gradient of the pair in row r
  }
  if (slot) dkey[pair] = v;
}

// part[m, c] = sum over the rows r of 128-row tile m (ascending) of dkey_row[r] * xs[r, c]; tiles are those of the forward's
// row prefix, so a tile belongs to one expert.  Block: 128 threads x 8 columns.  Bound by the read of xs; one block per expert
// and column slab, as this was first, left a popular expert's thousands of rows to a single serial loop (skewed 128-expert
// layer, T = 3001: 721 us, now 42; T = 8192, d = 4096, top-8 without skew: 174, now 108; d = 2048, 64 experts: 290, now 50).
constexpr int DW_THREADS = 128, DW_ROWS = 128;
__global__ void __launch_bounds__(DW_THREADS) gate_dw_kernel(const uint4* __restrict__ xs, const float* __restrict__ dkey_row,
                                                             const int32_t* __restrict__ poff,
                                                             const int32_t* __restrict__ expert_counts,
                                                             const int32_t* __restrict__ mt_prefix, float* __restrict__ part,
                                                             int E, int d) {
  grid_dependency_sync();
  const int v = blockIdx.x * DW_THREADS + threadIdx.x;   // uint4 index inside the row
  const int vec_per_row = d >> 3;
  if (v >= vec_per_row) return;
  const int tiles = __ldg(mt_prefix + E);
  for (int m = blockIdx.y; m < tiles; m += gridDim.y) {
    int lo = 0, hi = E;   // mt_prefix[lo] <= m < mt_prefix[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (__ldg(mt_prefix + mid) <= m) lo = mid; else hi = mid;
    }
    const int first = (m - __ldg(mt_prefix + lo)) * DW_ROWS;
    const int r0 = __ldg(poff + lo) + first, n = min(DW_ROWS, __ldg(expert_counts + lo) - first);
    float acc[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[q] = 0.f;
    const uint4* col = xs + (size_t)r0 * vec_per_row + v;
#pragma unroll 8
    for (int i = 0; i < n; ++i) {
      const float g = __ldg(dkey_row + r0 + i);
      const uint4 xv = __ldcs(col + (size_t)i * vec_per_row);
      const __nv_bfloat162* px = reinterpret_cast<const __nv_bfloat162*>(&xv);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float2 f = __bfloat1622float2(px[q]);
        acc[2 * q] = fmaf(g, f.x, acc[2 * q]);
        acc[2 * q + 1] = fmaf(g, f.y, acc[2 * q + 1]);
      }
    }
    float4* out = reinterpret_cast<float4*>(part + (size_t)m * d + v * 8);
    out[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    out[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
}

// dw_gate[c, e] = sum over the tiles of expert e (ascending) of part[m, c]; wgt[e, c] = w_gate[c, e].  Both are transposes
// between [., d] and [d, E], 32 x 32 through shared memory.
__global__ void __launch_bounds__(256) gate_finish_kernel(const float* __restrict__ part, const int32_t* __restrict__ mt_prefix,
                                                          float* __restrict__ dw_gate, const float* __restrict__ w_gate,
                                                          float* __restrict__ wgt, int d, int E) {
  grid_dependency_sync();
  __shared__ float tile[2][32][33];
  const int c0 = blockIdx.x * 32, e0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;   // 8 rows per pass
  for (int i = ty; i < 32; i += 8) {
    const int c = c0 + i, e = e0 + tx;
    tile[0][i][tx] = (c < d && e < E) ? __ldg(w_gate + (size_t)c * E + e) : 0.f;
    float sum = 0.f;
    if (e0 + i < E && c0 + tx < d) {
      const int m1 = __ldg(mt_prefix + e0 + i + 1);
#pragma unroll 8
      for (int m = __ldg(mt_prefix + e0 + i); m < m1; ++m) sum += __ldcs(part + (size_t)m * d + c0 + tx);
    }
    tile[1][i][tx] = sum;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    if (e0 + i < E && c0 + tx < d) wgt[(size_t)(e0 + i) * d + c0 + tx] = tile[0][tx][i];
    if (c0 + i < d && e0 + tx < E) dw_gate[(size_t)(c0 + i) * E + e0 + tx] = tile[1][tx][i];
  }
}

// dx[t, :] += sum_j dkey[t, j] * wgt[e_j, :]; a warp per token, four columns per lane and step.  Few tokens are bound by the latency of the
// reads: FOUR has the rows of four slots in flight (48 registers per thread).  Many tokens hide it by their number: the plain loop
// takes 32 registers, so that the SM is full of warps.  Whole gate gradient, us, plain / four in flight: 320 tokens top-4 of d = 1896 52.7 /
// 45.6, 1000 top-8 of d = 4096 124 / 97, 1000 top-1 of d = 2048 44.0 / 44.3, 3001 top-4 of d = 2880 93 / 84, 4096 top-2 of d = 4096 100 / 96,
// 8192 top-8 of d = 2048 111 / 121, of d = 4096 240 / 237, 16384 top-4 of d = 1024 85 / 96.  Same sums, same order.
template <bool FOUR>
__global__ void __launch_bounds__(256) gate_dx_kernel(const int32_t* __restrict__ topk_idx, const float* __restrict__ dkey,
                                                      const float* __restrict__ wgt, __nv_bfloat16* dx, int T, int E,
                                                      int k, int d) {
  grid_dependency_sync();
  __shared__ int s_e[8][32];
  __shared__ float s_g[8][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  for (int t = blockIdx.x * wpb + wid; t < T; t += gridDim.x * wpb) {
    __syncwarp();
    if (lane < k) {
      const int e = __ldg(topk_idx + (size_t)t * k + lane);
      const bool in = e >= 0 && e < E;
      s_e[wid][lane] = in ? e : 0;
      s_g[wid][lane] = in ? __ldg(dkey + (size_t)t * k + lane) : 0.f;
    }
    __syncwarp();
    __nv_bfloat16* row = dx + (size_t)t * d;
    for (int c = lane * 4; c < d; c += 128) {
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      auto row_of = [&](int j) { return __ldg(reinterpret_cast<const float4*>(wgt + (size_t)s_e[wid][j] * d + c)); };
      auto add = [&](int j, const float4& wv) {
        const float g = s_g[wid][j];
        acc.x = fmaf(g, wv.x, acc.x);
        acc.y = fmaf(g, wv.y, acc.y);
        acc.z = fmaf(g, wv.z, acc.z);
        acc.w = fmaf(g, wv.w, acc.w);
      };
      if (FOUR) {
        for (int j = 0; j < k; j += 4) {
          float4 wv[4];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + q < k) wv[q] = row_of(j + q);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (j + q < k) add(j + q, wv[q]);
        }
      } else {
#pragma unroll 4
        for (int j = 0; j < k; ++j) add(j, row_of(j));
      }
      uint2 raw = *reinterpret_cast<const uint2*>(row + c);
      __nv_bfloat162* p2 = reinterpret_cast<__nv_bfloat162*>(&raw);
      const float2 lo = __bfloat1622float2(p2[0]), hi = __bfloat1622float2(p2[1]);
      p2[0] = __floats2bfloat162_rn(lo.x + acc.x, lo.y + acc.y);
      p2[1] = __floats2bfloat162_rn(hi.x + acc.z, hi.y + acc.w);
      *reinterpret_cast<uint2*>(row + c) = raw;
    }
  }
}

}  // namespace

cudaError_t launch_gate_backward(const Shape& s, const GateBwdArgs& a, cudaStream_t st) {
  cudaError_t err;
  if (s.T == 0) return cudaMemsetAsync(a.dw_gate, 0, (size_t)s.d * s.E * sizeof(float), st);
  const int n_rows = (int)bwd_row_capacity(s);
  ProfileScope prof(KID_GATE_BWD, st);
  const int cap = sm_count() * 8;
  int blocks = (n_rows + 255) / 256;
  if (blocks > cap) blocks = cap;
  if ((err = launch_pdl(gate_rowdot_kernel, blocks, 256, 0, st, a.row_dots, bwd_dot_parts(s), (long long)n_rows, a.poff, a.g_row,
                        s.E)) != cudaSuccess)
    return err;
  int shift = 0;
  while (1 << shift < s.k) ++shift;
  if ((err = launch_pdl(gate_route_bwd_kernel, (unsigned)((((long long)s.T << shift) + 255) / 256), 256, 0, st, a.topk_idx, a.topk_w, a.pair_prow,
                        a.logits, a.bias, (long long)a.bias_stride, a.g_row, a.dkey, s.T, s.E, s.k,
                        s.score_fn == 1 ? 1 : 0, n_rows, shift)) != cudaSuccess)
    return err;
  long long tiles = (long long)s.T * s.k / DW_ROWS + s.E;   // at most; the count is on the device
  if (tiles > 16384) tiles = 16384;
  if ((err = launch_pdl(gate_dw_kernel, dim3((s.d / 8 + DW_THREADS - 1) / DW_THREADS, (unsigned)tiles), DW_THREADS, 0, st,
                        static_cast<const uint4*>(a.xs), static_cast<const float*>(a.g_row), a.poff, a.expert_counts,
                        a.mt_prefix, a.part, s.E, s.d)) != cudaSuccess)
    return err;
  if ((err = launch_pdl(gate_finish_kernel, dim3((s.d + 31) / 32, (s.E + 31) / 32), 256, 0, st,
                        static_cast<const float*>(a.part), a.mt_prefix, a.dw_gate, a.w_gate, a.wgt, s.d, s.E)) != cudaSuccess)
    return err;
  blocks = (s.T + 7) / 8;
  // five blocks of the form with more registers fit an SM: it is taken while all of its blocks are resident
  const auto dx = blocks <= 5 * sm_count() ? gate_dx_kernel<true> : gate_dx_kernel<false>;
  if (blocks > cap) blocks = cap;
  return launch_pdl(dx, blocks, 256, 0, st, a.topk_idx, static_cast<const float*>(a.dkey),
                    static_cast<const float*>(a.wgt), static_cast<__nv_bfloat16*>(a.dx), s.T, s.E, s.k, s.d);
}

}  // namespace tcmoe
