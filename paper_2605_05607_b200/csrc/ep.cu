// Expert-parallel execution of the layer across GPUs (paper Sec. II-A: Dispatch sends each token to the
// GPUs hosting its experts, Combine brings the outputs back; Sec. III-D: one replica per destination, trimmed
// to that destination's targets; reduction of the outputs of one destination before they travel back).
// With the G expert groups placed on G GPUs, the data that crosses the links is exactly what the single-GPU
// path already builds: the dispatched buffer xg (one row per distinct (token, group)) on the way out, one
// pre-reduced row per (token, group) on the way back.  Two small kernels complete the picture:
//   ep_pack    for every dispatched row the trimmed target list: the token's experts that live in the row's
//              group (as indices local to the group) and their gate weights - the routing table the
//              receiving GPU runs its experts from (MOE_FLAG_SPARSE_TOPK form)
//   ep_finish  y[t] = sum over the groups t touched of the pre-reduced row that came back
// Everything between them (layout, expert FFN, in-group reduction) is the ordinary entry points applied to
// the received rows.
#include "common.cuh"

#include <cuda_bf16.h>

namespace tcmoe {
namespace {

// Thread per dispatched row n = (t, g): the token's slots that live in the group, in slot order, then -1 / 0.  The rows behind
// the last dispatched one (and a row whose table entry is no token) are unused.  Lists leave through shared memory, entry by
// entry, as whole lines.
constexpr int PACK_ROWS = 128, PACK_LD = PACK_ROWS + 4;   // + 4: eight entries of four rows fall into 32 banks
__global__ void __launch_bounds__(PACK_ROWS) ep_pack_kernel(const int32_t* __restrict__ topk_idx,
                                                            const float* __restrict__ topk_w,
                                                            const int32_t* __restrict__ disp_token,
                                                            const int32_t* __restrict__ group_offsets,
                                                            int32_t* __restrict__ send_idx, float* __restrict__ send_w, int T,
                                                            int k, int G, int m, int kk, int cap_rows) {
  extern __shared__ int32_t idx_s[];                      // [kk][PACK_LD]
  float* w_s = reinterpret_cast<float*>(idx_s + kk * PACK_LD);
  int32_t* goff_s = idx_s + 2 * kk * PACK_LD;             // [G + 1]
  grid_dependency_sync();
  const int tid = threadIdx.x;
  for (int i = tid; i <= G; i += PACK_ROWS) goff_s[i] = __ldg(group_offsets + i);
  __syncthreads();
  const int rows = min(goff_s[G], cap_rows);
  for (long long base = (long long)blockIdx.x * PACK_ROWS; base < cap_rows; base += (long long)gridDim.x * PACK_ROWS) {
    const long long n = base + tid;
    const int t = n < rows ? __ldg(disp_token + n) : -1;
    int pos = 0;
    if (t >= 0 && t < T) {
      int g = 0, hi = G;   // goff_s[g] <= n < goff_s[hi]
      while (hi - g > 1) {
        const int mid = (g + hi) >> 1;
        if (goff_s[mid] <= n) g = mid; else hi = mid;
      }
      for (int j = 0; j < k && pos < kk; ++j) {
        const int e = __ldg(topk_idx + (size_t)t * k + j) - g * m;   // m G = E: nothing outside [0, E) passes
        if (e < 0 || e >= m) continue;
        idx_s[pos * PACK_LD + tid] = e;
        w_s[pos * PACK_LD + tid] = __ldg(topk_w + (size_t)t * k + j);
        ++pos;
      }
    }
    for (; pos < kk; ++pos) {
      idx_s[pos * PACK_LD + tid] = -1;
      w_s[pos * PACK_LD + tid] = 0.f;
    }
    __syncthreads();
    const int entries = (int)min((long long)PACK_ROWS, cap_rows - base) * kk;
    for (int i = tid; i < entries; i += PACK_ROWS) {
      const int r = i / kk, q = i - r * kk;
      send_idx[(size_t)base * kk + i] = idx_s[q * PACK_LD + r];
      send_w[(size_t)base * kk + i] = w_s[q * PACK_LD + r];
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void add_row(float (&acc)[8], const uint4& raw) {
  const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(p[i]);
    acc[2 * i] += f.x;
    acc[2 * i + 1] += f.y;
  }
}
__device__ __forceinline__ uint4 round_row(const float (&acc)[8]) {
  uint4 out;
  __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(&out);
#pragma unroll
  for (int q = 0; q < 4; ++q) o[q] = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
  return out;
}

// Warp per (token, column part): fp32 sum over the groups, ascending g.  Lane g finds the row of group g once; with ROWS > 0 a token
// touches at most ROWS = min(k, G) groups (2 or 4) and their rows stay in registers, otherwise up to 32 groups' rows stay in the lanes
// (with more the later ones are looked up per column step).  Four loads are in flight per lane: four rows of a column, or two
// columns of two.  Bound by the read of the returned rows: 2050 tokens of d = 4096, top-8 of 8 groups 22 us, 8192 tokens of d = 2880, one
// group 15, two of 8 groups 20 (with the lookup in the column loop and one form for all: 23.5, 28 and 33).
constexpr int FINISH_BLOCKS = 5;   // resident per SM
template <int ROWS>
__global__ void __launch_bounds__(256, FINISH_BLOCKS) ep_finish_kernel(const uint4* __restrict__ back, uint4* __restrict__ y,
                                                           const int32_t* __restrict__ al,
                                                           const int32_t* __restrict__ group_offsets, int T, int G,
                                                           int vec_per_row, int parts, int vec_per_part) {
  grid_dependency_sync();
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  const unsigned units = (unsigned)T * parts;   // parts > 1 for a few thousand tokens only
  for (unsigned w = blockIdx.x * wpb + (threadIdx.x >> 5); w < units; w += gridDim.x * wpb) {
    const int t = w / parts, part = w % parts;
    const int v_begin = part * vec_per_part, v_end = min(vec_per_row, v_begin + vec_per_part);
    auto row_of = [&](int g) {
      if (g >= G) return -1;
      const int a = __ldg(al + (size_t)g * T + t);
      return a >= 0 ? __ldg(group_offsets + g) + a : -1;
    };
    uint4* out = y + (size_t)t * vec_per_row;
    if (ROWS > 0) {
      constexpr int R = ROWS > 0 ? ROWS : 1, COLS = 4 / R;
      int r[R];
#pragma unroll
      for (int q = 0; q < R; ++q) r[q] = -1;
      int n = 0;
      for (int g0 = 0; g0 < G; g0 += 32) {
        const int row = row_of(g0 + lane);
        for (unsigned live = __ballot_sync(0xFFFFFFFFu, row >= 0); live; live &= live - 1, ++n) {
          const int next = __shfl_sync(0xFFFFFFFFu, row, __ffs(live) - 1);
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (q == n) r[q] = next;
        }
      }
      for (int v = v_begin + lane; v < v_end; v += 32 * COLS) {
        uint4 buf[R][COLS];
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int u = 0; u < COLS; ++u)
            if (q < n && v + 32 * u < v_end) buf[q][u] = __ldcs(back + (size_t)r[q] * vec_per_row + v + 32 * u);
#pragma unroll
        for (int u = 0; u < COLS; ++u) {
          float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int q = 0; q < R; ++q)
            if (q < n) add_row(acc, buf[q][u]);
          if (v + 32 * u < v_end) out[v + 32 * u] = round_row(acc);
        }
      }
      continue;
    }
    const int first_row = row_of(lane);
    const unsigned first = __ballot_sync(0xFFFFFFFFu, first_row >= 0);
    for (int v0 = v_begin; v0 < v_end; v0 += 32) {   // whole warps: the row numbers are shuffled
      const int v = v0 + lane;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int g0 = 0; g0 < G; g0 += 32) {
        const int row = g0 == 0 ? first_row : row_of(g0 + lane);
        unsigned live = g0 == 0 ? first : __ballot_sync(0xFFFFFFFFu, row >= 0);
        while (live) {
          uint4 buf[4];
          int n = 0;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (live) {
              const int r = __shfl_sync(0xFFFFFFFFu, row, __ffs(live) - 1);
              live &= live - 1;
              n = q + 1;
              if (v < v_end) buf[q] = __ldcs(back + (size_t)r * vec_per_row + v);
            }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (q < n && v < v_end) add_row(acc, buf[q]);
        }
      }
      if (v < v_end) out[v] = round_row(acc);
    }
  }
}

}  // namespace

cudaError_t launch_ep_pack(const Shape& s, const int32_t* topk_idx, const float* topk_w, const Layout& L,
                           int32_t* send_idx, float* send_w, cudaStream_t st) {
  if (s.T == 0) return cudaSuccess;
  const int m = s.E / s.G, kk = s.k < m ? s.k : m;
  const int cap_rows = s.T * (s.k < s.G ? s.k : s.G);   // dispatched-row capacity
  const int blocks = min((cap_rows - 1) / PACK_ROWS + 1, sm_count() * 16);
  return launch_pdl(ep_pack_kernel, blocks, PACK_ROWS, ((size_t)2 * kk * PACK_LD + s.G + 1) * 4, st, topk_idx, topk_w, L.disp_token,
                    L.group_offsets, send_idx, send_w, s.T, s.k, s.G, m, kk, cap_rows);
}

cudaError_t launch_ep_finish(const Shape& s, const void* back, const Layout& L, void* y, cudaStream_t st) {
  if (s.T == 0) return cudaSuccess;
  const int vec = s.d / 8, parts = row_parts(s.T, vec);
  const int vec_per_part = ((vec + parts - 1) / parts + 31) & ~31;   // whole warp-strides per part
  long long blocks = ((long long)s.T * parts + 7) / 8;
  const long long cap = (long long)sm_count() * 2 * FINISH_BLOCKS;
  if (blocks > cap) blocks = cap;
  const int rows = min(s.k, s.G);
  return launch_pdl(rows <= 2 ? ep_finish_kernel<2> : rows <= 4 ? ep_finish_kernel<4> : ep_finish_kernel<0>, (unsigned)blocks, 256, 0, st,
                    static_cast<const uint4*>(back), static_cast<uint4*>(y), L.al, L.group_offsets, s.T, s.G, vec, parts,
                    vec_per_part);
}

}  // namespace tcmoe
