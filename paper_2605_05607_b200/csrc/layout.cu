// Dispatch layout, dispatch and combine (paper Sec. III-D: switch routing rule
// group = expert / experts_per_group, AL tables built by a running counter, MV translation;
// Sec. IV-B TID table; Sec. III-C un-weighted reduction in Combine).
//
// The hardware of the paper hands out layout rows in arrival order.  Here the order is fixed to
// ascending token index so that the layout is a pure function of topk_idx: membership bitmasks
// (one bit per (expert, token) and per (group, token)) are built with order-independent atomicOr,
// an exclusive popcount scan along each mask row gives every token its rank, and a fill pass
// turns ranks into the row tables.  No atomics touch the result arrays.
#include "combine.cuh"
#include "ptx.cuh"
#include "route.cuh"

#include <atomic>

namespace tcmoe {

// Mask and fill passes: a block takes one mask word of 32 tokens, its eight warps take turns in the slots and groups of these tokens.
// (With a thread per token a batch of 8192 tokens had 32 blocks, each walking 32 groups and 8 slots one latency after the other:
// 13 and 33 us; the four kernels of top-8 in 32 groups 37.6 -> 11.5 us.)
constexpr int WORD_WARPS = 8;

// ---- K2a: membership masks -------------------------------------------------------------------
__global__ void __launch_bounds__(WORD_WARPS * 32) build_masks_kernel(const int32_t* __restrict__ topk_idx, uint32_t* emask,
                                                          uint32_t* gmask, int T, int E, int k, int m, int W,
                                                          int32_t* status, int sparse) {
  grid_dependency_sync();
  const int lane = threadIdx.x & 31, word = blockIdx.x, t = word * 32 + lane;
  const bool live = t < T;
  for (int j = threadIdx.x >> 5; j < k; j += WORD_WARPS) {
    int e = live ? __ldg(topk_idx + (size_t)t * k + j) : -1;
    if (live && (e < 0 || e >= E)) {
      if (!(sparse && e == -1)) report_error(status, DEV_INDEX_OUT_OF_RANGE, KID_MASKS, t, e);   // -1: unused slot
      e = -1;
    }
    // lanes that picked the same expert (group) fold their bits into one atomicOr
    const unsigned same_e = __match_any_sync(0xFFFFFFFFu, e);
    if (e >= 0 && lane == __ffs(same_e) - 1) atomicOr(&emask[(size_t)e * W + word], same_e);
    const int g = (e >= 0) ? e / m : -1;
    const unsigned same_g = __match_any_sync(0xFFFFFFFFu, g);
    if (g >= 0 && lane == __ffs(same_g) - 1) atomicOr(&gmask[(size_t)g * W + word], same_g);
  }
}

// ---- K2b: exclusive popcount prefix along every mask row; row totals -> counts ------------------
__global__ void __launch_bounds__(256) scan_masks_kernel(const uint32_t* __restrict__ emask,
                                                         const uint32_t* __restrict__ gmask, int32_t* eprefix,
                                                         int32_t* gprefix, int32_t* expert_counts,
                                                         int32_t* group_counts, int E, int W) {
  grid_dependency_sync();
  __shared__ int warp_sum[8];
  __shared__ int running_s;
  const int row = blockIdx.x;
  const uint32_t* mask = (row < E) ? emask + (size_t)row * W : gmask + (size_t)(row - E) * W;
  int32_t* prefix = (row < E) ? eprefix + (size_t)row * W : gprefix + (size_t)(row - E) * W;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) running_s = 0;
  __syncthreads();
  for (int base = 0; base < W; base += 256) {
    const int i = base + threadIdx.x;
    const int c = (i < W) ? __popc(mask[i]) : 0;
    int incl = c;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, incl, off);
      if (lane >= off) incl += n;
    }
    if (lane == 31) warp_sum[wid] = incl;
    __syncthreads();
    int warp_base = 0;
    for (int w = 0; w < wid; ++w) warp_base += warp_sum[w];
    const int running = running_s;
    if (i < W) prefix[i] = running + warp_base + incl - c;
    __syncthreads();
    if (threadIdx.x == 255) running_s = running + warp_base + incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    if (row < E) expert_counts[row] = running_s;
    else group_counts[row - E] = running_s;
  }
}

// ---- K2c: offsets (exclusive scans over experts / groups) and the GEMM tile prefixes --------------
__global__ void __launch_bounds__(1024) offsets_kernel(const int32_t* __restrict__ expert_counts,
                                                       const int32_t* __restrict__ group_counts,
                                                       int32_t* expert_offsets, int32_t* group_offsets,
                                                       int32_t* mt_prefix, int32_t* mp_prefix, int E, int G) {
  grid_dependency_sync();
  __shared__ int sums[4][32];
  const int i = threadIdx.x;
  const int ce = (i < E) ? expert_counts[i] : 0;
  const int cg = (i < G) ? group_counts[i] : 0;
  int v[4] = {ce, cg, (ce + 127) >> 7, (ce + 255) >> 8};   // 128-row tiles (GEMM-1), 256-row CTA-pair tiles (GEMM-2)
  block_scan(v, sums);
  if (i < E) { expert_offsets[i + 1] = v[0]; mt_prefix[i + 1] = v[2]; mp_prefix[i + 1] = v[3]; }
  if (i < G) group_offsets[i + 1] = v[1];
  if (i == 0) { expert_offsets[0] = 0; group_offsets[0] = 0; mt_prefix[0] = 0; mp_prefix[0] = 0; }
}

// ---- K2d: ranks -> row tables ----------------------------------------------------------------
__global__ void __launch_bounds__(WORD_WARPS * 32) fill_layout_kernel(const int32_t* __restrict__ topk_idx, Layout L,
                                                          LayoutScratch sc, int T, int E, int k, int G, int m) {
  grid_dependency_sync();
  const int word = blockIdx.x, t = word * 32 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
  if (t >= T) return;
  const uint32_t below = (1u << (t & 31)) - 1u;
  for (int g = warp; g < G; g += WORD_WARPS) {
    const uint32_t bits = sc.gmask[(size_t)g * sc.W + word];
    int a = -1;
    if (bits >> (t & 31) & 1u) {
      a = sc.gprefix[(size_t)g * sc.W + word] + __popc(bits & below);
      L.disp_token[L.group_offsets[g] + a] = t;  // TID table entry of the allocated row
    }
    L.al[(size_t)g * T + t] = a;
  }
  for (int j = warp; j < k; j += WORD_WARPS) {
    const int e = __ldg(topk_idx + (size_t)t * k + j);
    if (e < 0 || e >= E) {          // unused slot (sparse top-k), or an index build_masks_kernel reported
      L.pair_row[(size_t)t * k + j] = -1;
      continue;
    }
    const int rank = sc.eprefix[(size_t)e * sc.W + word] + __popc(sc.emask[(size_t)e * sc.W + word] & below);
    const int r = L.expert_offsets[e] + rank;
    const int g = e / m;
    const uint32_t gbits = sc.gmask[(size_t)g * sc.W + word];
    const int a = sc.gprefix[(size_t)g * sc.W + word] + __popc(gbits & below);
    L.pair_row[(size_t)t * k + j] = r;
    L.row_pair[r] = t * k + j;
    L.row_src[r] = L.group_offsets[g] + a;
  }
}

// ---- K2 in one kernel ----------------------------------------------------------------------------
// The four passes above as one kernel of at most 8 thread blocks (a cluster), for small tables (layout_in_one): every block owns a
// contiguous range of tokens, builds its masks and their prefixes in shared memory, reads the other blocks' row totals through
// distributed shared memory and fills its tokens' entries.  The four launches are latency, not work: 12.2 us for 600 tokens of
// top-2 in 8 groups, 10.7 us for 3001 of top-4; in one kernel 4.9 and 8.2 us.
constexpr int ONE_THREADS = 1024, ONE_MAX_BLOCKS = 8, ONE_MAX_PAIRS = 32768, ONE_MAX_SMEM = 160 * 1024;
struct OneShape { int blocks, tokens, words; size_t smem; };   // tokens per block (a multiple of 32) and their mask words
OneShape one_shape(const Shape& s, bool topk) {
  OneShape o;
  o.blocks = 1;
  while (o.blocks < ONE_MAX_BLOCKS && o.blocks * (topk ? 32 : 256) < s.T) o.blocks *= 2;
  o.tokens = ((s.T + o.blocks - 1) / o.blocks + 31) & ~31;
  o.words = o.tokens / 32;
  const size_t rows = (size_t)s.E + s.G;
  o.smem = rows * (o.words + 1) * 4 + rows * (o.words + 1) * 2 + rows * 4 * 2 + 16 + (topk ? (size_t)o.tokens * s.k * 4 : 0);
  return o;
}

// With KPL > 0 the kernel first takes the top-k of its tokens (a warp each, E <= 32 KPL) and writes topk_idx / topk_w: for a batch
// of up to 512 tokens the top-k kernel is a launch's latency as well.
struct TopkArgs {
  const float *logits, *bias;
  long long bias_stride;
  float* topk_w;
  int score_fn;
};
template <int KPL>
__global__ void __launch_bounds__(ONE_THREADS) layout_one_kernel(int32_t* topk_idx, const TopkArgs tk, Layout L,
                                                                 int32_t* mt_prefix, int32_t* mp_prefix, int T, int E, int k,
                                                                 int G, int m, int TL, int W, int32_t* status, int sparse) {
  extern __shared__ uint32_t one_s[];
  __shared__ int warp_sum[4][32];
  const int rows = E + G, ld = W + 1;   // row e < E: expert e, row E + g: group g; a pad word against bank conflicts
  uint32_t* mask = one_s;                                                  // [rows][ld]
  int* total = reinterpret_cast<int*>(mask + (size_t)rows * ld);           // [rows] members among this block's tokens
  int* base = total + rows;                                                // [rows] table entry of the block's first member
  int* idx_s = base + rows;                                                // [TL][k] (KPL > 0): the selection of the block's tokens
  uint16_t* prefix = reinterpret_cast<uint16_t*>(idx_s + (KPL > 0 ? TL * k : 0));   // [rows][ld] members before the word
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int rank = blockIdx.x, blocks = gridDim.x;                         // the grid is one cluster
  const int t0 = rank * TL, tn = max(0, min(TL, T - t0));
  for (int i = tid; i < rows * ld; i += ONE_THREADS) mask[i] = 0u;
  grid_dependency_sync();
  if (KPL > 0) {
    bool nonfinite = false;
    for (int tl = wid; tl < tn; tl += ONE_THREADS / 32) {
      uint32_t e;
      float w;
      topk_token<KPL == 0 ? 1 : KPL>(tk.logits, tk.bias, tk.bias_stride, t0 + tl, E, k, tk.score_fn, lane, nonfinite, e, w);
      if (lane < k) {
        idx_s[tl * k + lane] = (int)e;
        topk_idx[(size_t)(t0 + tl) * k + lane] = (int32_t)e;
        tk.topk_w[(size_t)(t0 + tl) * k + lane] = w;
      }
    }
    if (__any_sync(0xFFFFFFFFu, nonfinite) && lane == 0) atomicOr(&status[ST_WARN], WARN_NONFINITE_LOGIT);
  }
  __syncthreads();
  for (int i = tid; i < tn * k; i += ONE_THREADS) {
    const int tl = i / k;
    const int e = KPL > 0 ? idx_s[i] : __ldg(topk_idx + (size_t)t0 * k + i);
    if (e < 0 || e >= E) {
      if (!(sparse && e == -1)) report_error(status, DEV_INDEX_OUT_OF_RANGE, KID_MASKS, t0 + tl, e);   // -1: unused slot
      continue;
    }
    atomicOr(&mask[e * ld + (tl >> 5)], 1u << (tl & 31));
    atomicOr(&mask[(E + e / m) * ld + (tl >> 5)], 1u << (tl & 31));
  }
  __syncthreads();
  for (int r = tid; r < rows; r += ONE_THREADS) {
    int n = 0;
    for (int w = 0; w < W; ++w) {
      prefix[r * ld + w] = (uint16_t)n;
      n += __popc(mask[r * ld + w]);
    }
    total[r] = n;
  }
  ptx::cluster_sync();
  // thread i: expert i and group i.  Members in the blocks before this one, and in all.
  int before[2] = {0, 0}, all[2] = {0, 0};
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (tid >= (j ? G : E)) continue;
    const uint32_t at = ptx::smem_u32(total + (j ? E + tid : tid));
    for (int b = 0; b < blocks; ++b) {
      const int n = ptx::ld_shared_cluster(ptx::mapa(at, b));
      if (b < rank) before[j] += n;
      all[j] += n;
    }
  }
  // exclusive scans over the experts / groups: rows, dispatched rows, 128-row tiles, 256-row tiles
  int v[4] = {all[0], all[1], (all[0] + 127) >> 7, (all[0] + 255) >> 8}, incl[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    incl[q] = v[q];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int n = __shfl_up_sync(0xFFFFFFFFu, incl[q], off);
      if (lane >= off) incl[q] += n;
    }
    if (lane == 31) warp_sum[q][wid] = incl[q];
  }
  __syncthreads();
  if (wid < 4) {
    int n = warp_sum[wid][lane];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int u = __shfl_up_sync(0xFFFFFFFFu, n, off);
      if (lane >= off) n += u;
    }
    warp_sum[wid][lane] = n;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (wid > 0) incl[q] += warp_sum[q][wid - 1];
  if (tid < E) base[tid] = incl[0] - v[0] + before[0];
  if (tid < G) base[E + tid] = incl[1] - v[1] + before[1];
  __shared__ int goff_s[1024];                                             // first dispatched row of a group
  if (tid < G) goff_s[tid] = incl[1] - v[1];
  if (rank == 0) {
    if (tid < E) {
      L.expert_counts[tid] = all[0];
      L.expert_offsets[tid + 1] = incl[0];
      mt_prefix[tid + 1] = incl[2];
      mp_prefix[tid + 1] = incl[3];
    }
    if (tid < G) {
      L.group_counts[tid] = all[1];
      L.group_offsets[tid + 1] = incl[1];
    }
    if (tid == 0) { L.expert_offsets[0] = 0; L.group_offsets[0] = 0; mt_prefix[0] = 0; mp_prefix[0] = 0; }
  }
  __syncthreads();
  ptx::cluster_arrive();   // this block has read the others' totals
  auto rank_of = [&](int r, int tl) {
    return (int)prefix[r * ld + (tl >> 5)] + __popc(mask[r * ld + (tl >> 5)] & ((1u << (tl & 31)) - 1u));
  };
  for (int i = tid; i < G * TL; i += ONE_THREADS) {
    const int g = i / TL, tl = i - g * TL;
    if (tl >= tn) continue;
    int a = -1;
    if (mask[(E + g) * ld + (tl >> 5)] >> (tl & 31) & 1u) {
      const int row = base[E + g] + rank_of(E + g, tl);
      a = row - goff_s[g];
      L.disp_token[row] = t0 + tl;   // TID table entry of the allocated row
    }
    L.al[(size_t)g * T + t0 + tl] = a;
  }
  for (int i = tid; i < tn * k; i += ONE_THREADS) {
    const int tl = i / k, p = t0 * k + i;
    const int e = KPL > 0 ? idx_s[i] : __ldg(topk_idx + p);
    if (e < 0 || e >= E) {           // unused slot (sparse top-k), or an index reported above
      L.pair_row[p] = -1;
      continue;
    }
    const int r = base[e] + rank_of(e, tl), g = E + e / m;
    L.pair_row[p] = r;
    L.row_pair[r] = p;
    L.row_src[r] = base[g] + rank_of(g, tl);
  }
  __syncwarp();
  ptx::cluster_wait();     // no block leaves while another may still read its totals
}

// Eight blocks write the G x T table of allocated rows and the T x k ones, so the one kernel is the better form while there are few
// entries: microseconds of both, fitted to 1 to 32768 tokens, top-1 to top-32, 1 to 1024 groups (a warp of the four kernels walks every
// eighth slot and group).  Four kernels / one, us: 32768 tokens top-1, 1 group 12.2 / 15.1, 104 groups 16.3 / 143; 12000 top-2, 4 groups
// 9.0 / 12.6; 4096 top-8, 32 groups 11.0 / 16.5; 5000 top-6, 16 groups 9.8 / 15.2; 3001 top-4, 8 groups 10.7 / 8.2; 2050 top-8, 8 groups
// 11.1 / 9.3; 1777 top-4, 8 groups 10.3 / 6.5; 600 top-2, 8 groups 12.2 / 4.9.
bool layout_in_one(const Shape& s) {
  if (s.T <= 0 || (long long)s.T * s.k > ONE_MAX_PAIRS || one_shape(s, false).smem > ONE_MAX_SMEM) return false;
  const double one = 5.0 + s.T * (4.2 + 1.7 * s.k + 0.62 * s.G) / 16384, four = 9.0 + (s.k + 7) / 8 + 0.45 * ((s.G + 7) / 8) + 3.2e-5 * s.T * s.k;
  return one < four;
}

template <int KPL>
static cudaError_t launch_layout_one(const Shape& s, int32_t* topk_idx, const TopkArgs& tk, const Layout& L,
                                     const LayoutScratch& sc, int32_t* status, cudaStream_t st) {
  static std::atomic<bool> attr_set[MAX_DEVICES];   // per device; setting the attribute twice is harmless
  const int dev = current_device();
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(layout_one_kernel<KPL>, cudaFuncAttributeMaxDynamicSharedMemorySize, ONE_MAX_SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  const OneShape o = one_shape(s, KPL > 0);
  return launch_pdl_cluster(o.blocks, layout_one_kernel<KPL>, o.blocks, ONE_THREADS, o.smem, st, topk_idx, tk, L, sc.mt_prefix,
                            sc.mp_prefix, s.T, s.E, s.k, s.G, s.E / s.G, o.tokens, o.words, status, (s.flags & 4) ? 1 : 0);
}

// up to 512 tokens (at most two per warp) of up to 256 experts
bool topk_in_layout(const Shape& s) { return s.T <= 512 && s.E <= 256 && layout_in_one(s) && one_shape(s, true).smem <= ONE_MAX_SMEM; }

cudaError_t launch_topk_layout(const Shape& s, const float* logits, const float* bias, int64_t bias_stride, int32_t* topk_idx,
                               float* topk_w, const Layout& L, const LayoutScratch& sc, int32_t* status, cudaStream_t st) {
  const TopkArgs tk{logits, bias, (long long)bias_stride, topk_w, s.score_fn};
  ProfileScope prof(KID_TOPK_LAYOUT, st);
  if (s.E <= 32) return launch_layout_one<1>(s, topk_idx, tk, L, sc, status, st);
  if (s.E <= 64) return launch_layout_one<2>(s, topk_idx, tk, L, sc, status, st);
  if (s.E <= 128) return launch_layout_one<4>(s, topk_idx, tk, L, sc, status, st);
  return launch_layout_one<8>(s, topk_idx, tk, L, sc, status, st);
}

// exclusive prefixes of 128-row tiles and 256-row pair tiles per expert, from the counts alone
__global__ void __launch_bounds__(1024) tile_prefix_kernel(const int32_t* __restrict__ expert_counts,
                                                           int32_t* mt_prefix, int32_t* mp_prefix, int E) {
  grid_dependency_sync();
  __shared__ int sums[2][32];
  const int i = threadIdx.x;
  const int c = (i < E) ? expert_counts[i] : 0;
  int v[2] = {(c + 127) >> 7, (c + 255) >> 8};
  block_scan(v, sums);
  if (i < E) { mt_prefix[i + 1] = v[0]; mp_prefix[i + 1] = v[1]; }
  if (i == 0) { mt_prefix[0] = 0; mp_prefix[0] = 0; }
}

cudaError_t launch_tile_prefix(const Shape& s, const int32_t* expert_counts, int32_t* mt_prefix, int32_t* mp_prefix,
                               cudaStream_t st) {
  return launch_pdl(tile_prefix_kernel, 1, 1024, 0, st, expert_counts, mt_prefix, mp_prefix, s.E);
}

cudaError_t launch_layout(const Shape& s, const int32_t* topk_idx, const Layout& L, const LayoutScratch& sc,
                          int32_t* status, cudaStream_t st, bool masks_cleared) {
  const int m = s.E / s.G;
  cudaError_t err;
  if (layout_in_one(s)) return launch_layout_one<0>(s, const_cast<int32_t*>(topk_idx), TopkArgs{}, L, sc, status, st);
  if (!masks_cleared &&
      (err = cudaMemsetAsync(sc.emask, 0, sizeof(uint32_t) * (size_t)(s.E + s.G) * sc.W, st)) != cudaSuccess)
    return err;  // emask and gmask are adjacent
  const int words = (s.T + 31) / 32;
  if (s.T > 0 && (err = launch_pdl(build_masks_kernel, words, WORD_WARPS * 32, 0, st, topk_idx, sc.emask, sc.gmask, s.T, s.E, s.k,
                                   m, sc.W, status, (s.flags & 4) ? 1 : 0)) != cudaSuccess)
    return err;
  if ((err = launch_pdl(scan_masks_kernel, s.E + s.G, 256, 0, st, sc.emask, sc.gmask, sc.eprefix, sc.gprefix,
                        L.expert_counts, L.group_counts, s.E, sc.W)) != cudaSuccess)
    return err;
  if ((err = launch_pdl(offsets_kernel, 1, 1024, 0, st, L.expert_counts, L.group_counts, L.expert_offsets,
                        L.group_offsets, sc.mt_prefix, sc.mp_prefix, s.E, s.G)) != cudaSuccess)
    return err;
  if (s.T > 0) return launch_pdl(fill_layout_kernel, words, WORD_WARPS * 32, 0, st, topk_idx, L, sc, s.T, s.E, s.k, s.G, m);
  return cudaSuccess;
}

// ---- K3: dispatch ------------------------------------------------------------------------------
// Token-centric: a warp reads (its part of) row x[t] once (16-byte vectors) and writes one copy per distinct
// group the token touches - the single-HBM image of "send once, the switch replicates per port".  With few tokens
// a row is split over `parts` warps (see combine_kernel).
__global__ void __launch_bounds__(256) dispatch_kernel(const uint4* __restrict__ x, uint4* __restrict__ xg,
                                                       const int32_t* __restrict__ al,
                                                       const int32_t* __restrict__ group_offsets, int T, int G,
                                                       int vec_per_row, int parts, int vec_per_part) {
  grid_dependency_sync();
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  const long long units = (long long)T * parts;
  for (long long u = (long long)blockIdx.x * wpb + (threadIdx.x >> 5); u < units; u += (long long)gridDim.x * wpb) {
    const int t = (int)(u / parts), part = (int)(u % parts);
    const int v_lo = part * vec_per_part, v_hi = min(vec_per_row, v_lo + vec_per_part);
    const uint4* src = x + (size_t)t * vec_per_row;
    for (int g0 = 0; g0 < G; g0 += 32) {
      const int g = g0 + lane;
      int dst_row = -1;
      if (g < G) {
        const int a = __ldg(al + (size_t)g * T + t);
        if (a >= 0) dst_row = __ldg(group_offsets + g) + a;
      }
      unsigned live = __ballot_sync(0xFFFFFFFFu, dst_row >= 0);
      if (!live) continue;
      for (int v0 = v_lo; v0 < v_hi; v0 += 128) {
        uint4 buf[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int v = v0 + q * 32 + lane;
          if (v < v_hi) buf[q] = __ldcs(src + v);
        }
        for (unsigned rem = live; rem; rem &= rem - 1) {
          const int row = __shfl_sync(0xFFFFFFFFu, dst_row, __ffs(rem) - 1);
          uint4* dst = xg + (size_t)row * vec_per_row;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int v = v0 + q * 32 + lane;
            if (v < v_hi) __stcs(dst + v, buf[q]);
          }
        }
      }
    }
  }
}

cudaError_t launch_dispatch(const Shape& s, const void* x, const Layout& L, void* xg, cudaStream_t st) {
  if (s.T == 0) return cudaSuccess;
  const int vec = s.d / 8;
  const int parts = row_parts(s.T, vec);
  const int vec_per_part = ((vec + parts - 1) / parts + 127) & ~127;   // whole 128-vector steps per part
  long long blocks = ((long long)s.T * parts + 7) / 8;
  const long long cap = (long long)sm_count() * 8;
  if (blocks > cap) blocks = cap;
  ProfileScope prof(KID_DISPATCH, st);
  return launch_pdl(dispatch_kernel, (unsigned)blocks, 256, 0, st, static_cast<const uint4*>(x), static_cast<uint4*>(xg),
                    L.al, L.group_offsets, s.T, s.G, vec, parts, vec_per_part);
}

// ---- K3b: dispatch into the per-expert layout tensors ----------------------------------------------
// xs[r, :] = src[gather_idx[r] / gather_div, :] for every expert-sorted row r: the dense per-expert buffers that
// the destination's memory manager fills in the paper (Sec. III-D: one AL sub-table per local expert), which is
// what lets GEMM-1 read its rows as plain TMA tiles.  One warp per row, 16-byte vectors; the number of rows in
// use is read from the device (expert_offsets[E]).
__global__ void __launch_bounds__(256) permute_rows_kernel(const uint4* __restrict__ src, uint4* __restrict__ xs,
                                                           const int32_t* __restrict__ gather_idx, int gather_div,
                                                           const int32_t* __restrict__ expert_offsets, int E,
                                                           int src_rows, int vec_per_row, int32_t* status) {
  grid_dependency_sync();
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  const int rows = __ldg(expert_offsets + E);
  for (int r = blockIdx.x * wpb + (threadIdx.x >> 5); r < rows; r += gridDim.x * wpb) {
    int idx = __ldg(gather_idx + r);
    if (gather_div > 1) idx /= gather_div;
    uint4* dst = xs + (size_t)r * vec_per_row;
    if (idx < 0 || idx >= src_rows) {   // a table entry that is no row of the source: reported, the row zero-filled
      if (lane == 0) report_error(status, DEV_INDEX_OUT_OF_RANGE, KID_DISPATCH, r, idx);
      for (int v = lane; v < vec_per_row; v += 32) dst[v] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const uint4* from = src + (size_t)idx * vec_per_row;
    for (int v0 = 0; v0 < vec_per_row; v0 += 128) {
      uint4 buf[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int v = v0 + q * 32 + lane;
        if (v < vec_per_row) buf[q] = __ldg(from + v);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int v = v0 + q * 32 + lane;
        if (v < vec_per_row) dst[v] = buf[q];
      }
    }
  }
}

cudaError_t launch_permute_rows(const Shape& s, const void* src, int src_rows, const int32_t* gather_idx,
                                int gather_div, const int32_t* expert_offsets, void* xs, int32_t* status,
                                cudaStream_t st) {
  if (s.T == 0) return cudaSuccess;
  long long blocks = ((long long)s.T * s.k + 7) / 8;
  const long long cap = (long long)sm_count() * 8;
  if (blocks > cap) blocks = cap;
  ProfileScope prof(KID_DISPATCH, st);
  return launch_pdl(permute_rows_kernel, (unsigned)blocks, 256, 0, st, static_cast<const uint4*>(src),
                    static_cast<uint4*>(xs), gather_idx, gather_div, expert_offsets, s.E, src_rows, s.d / 8, status);
}

// ---- K5: combine -----------------------------------------------------------------------------
// One warp per (token, column part); the per-token work is combine_token() (combine.cuh).  With few tokens a row
// is split over `parts` warps so that enough loads are in flight to reach the memory bandwidth (one warp per token
// leaves a 4096-token batch at a third of it).
template <int BATCH, int COLS, bool EARLY>
__global__ void __launch_bounds__(256, 3) combine_kernel(const CombineArgs c, int parts, int vec_per_part) {
  if (!EARLY) grid_dependency_sync();
  __shared__ int s_row[8][32];   // per warp: expert-sorted row of the slot at sorted position p
  __shared__ int s_dst[8][32];   // dispatched row (t, g) of that slot's group
  __shared__ float s_w[8][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  const long long units = (long long)c.T * parts;
  for (long long u = (long long)blockIdx.x * wpb + wid; u < units; u += (long long)gridDim.x * wpb) {
    const int t = (int)(u / parts), part = (int)(u % parts);
    combine_token<false, BATCH, COLS, EARLY>(c, t, lane, s_row[wid], s_dst[wid], s_w[wid], part * vec_per_part,
                                (part + 1) * vec_per_part);
  }
  if (EARLY) grid_dependency_sync();   // warps without a token
}

// parts of a row so that about 32 warps per SM exist even for small batches (at most 8, at least 4 vectors per lane)
int row_parts(int T, int vec_per_row) {
  int parts = 1;
  while (parts < 8 && (long long)T * parts < 32ll * sm_count() * 2 && vec_per_row / (parts * 2) >= 128) parts *= 2;
  return parts;
}

cudaError_t launch_combine(const Shape& s, const void* o, const Layout& L, const int32_t* topk_idx,
                           const float* topk_w, void* pg, void* y, int32_t* status, cudaStream_t st, bool early) {
  return launch_combine_rows(s, o, L, topk_idx, topk_w, pg, y, s.T * s.k, status, st, early);
}

// n_rows: rows of `o` (L.pair_row entries outside [0, n_rows) are reported and skipped).  early: the kernel before this one is the library's
// own GEMM that writes o, so the tables are older than it (it waited for the kernel before it and then let this one start): every warp
// orders its first token's slots before it waits.  Layer of 256 tokens, 8 experts of 512 x 1024 30.5 -> 29.3 us.
cudaError_t launch_combine_rows(const Shape& s, const void* o, const Layout& L, const int32_t* topk_idx,
                                const float* topk_w, void* pg, void* y, int n_rows, int32_t* status, cudaStream_t st, bool early) {
  if (s.T == 0) return cudaSuccess;
  const int vec = s.d / 8;
  const int parts = row_parts(s.T, vec);
  const int vec_per_part = ((vec + parts - 1) / parts + 31) & ~31;   // whole warp-strides per part
  long long blocks = ((long long)s.T * parts + 7) / 8;
  const long long cap = (long long)sm_count() * 8;
  if (blocks > cap) blocks = cap;
  ProfileScope prof(KID_COMBINE, st);
  CombineArgs c{static_cast<const uint4*>(o), static_cast<uint4*>(y), static_cast<uint4*>(pg), topk_idx, topk_w,
                L.pair_row, L.al, L.group_offsets, s.T, s.E, s.k, s.E / s.G, vec, (s.flags & 1) ? 1 : 0,
                n_rows, status};
  // parts that are no multiple of four warp strides: two columns at a time, so that the last step is not half empty (2050 tokens of
  // d = 2880 with group sums, 192 columns each: 11.8 -> 10.4 us, 10.7 with single columns)
  auto launch = [&](auto plain, auto before_wait) {
    return launch_pdl(early ? before_wait : plain, (unsigned)blocks, 256, 0, st, c, parts, vec_per_part);
  };
  if (s.k <= 2 && vec_per_part % 128 != 0) return launch(combine_kernel<2, 2, false>, combine_kernel<2, 2, true>);
  if (s.k <= 2) return launch(combine_kernel<2, 4, false>, combine_kernel<2, 4, true>);
  if (s.k <= 4) return launch(combine_kernel<4, 4, false>, combine_kernel<4, 4, true>);
  return launch(combine_kernel<8, 4, false>, combine_kernel<8, 4, true>);
}

// Last step of the layer when Combine ran inside GEMM-2's epilogue: the fp32 token accumulators
// become the bf16 output, 8 elements per thread.
__global__ void __launch_bounds__(256) round_rows_kernel(const float4* __restrict__ acc, uint4* __restrict__ y,
                                                         size_t n_vec) {
  grid_dependency_sync();
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_vec; i += stride) {
    const float4 a = __ldcs(acc + 2 * i), b = __ldcs(acc + 2 * i + 1);
    uint4 q;
    __nv_bfloat162 v;
    v = __floats2bfloat162_rn(a.x, a.y); q.x = *reinterpret_cast<uint32_t*>(&v);
    v = __floats2bfloat162_rn(a.z, a.w); q.y = *reinterpret_cast<uint32_t*>(&v);
    v = __floats2bfloat162_rn(b.x, b.y); q.z = *reinterpret_cast<uint32_t*>(&v);
    v = __floats2bfloat162_rn(b.z, b.w); q.w = *reinterpret_cast<uint32_t*>(&v);
    y[i] = q;
  }
}

cudaError_t launch_round_rows(const Shape& s, const float* acc, void* y, cudaStream_t st) {
  const size_t n_vec = (size_t)s.T * s.d / 8;
  if (n_vec == 0) return cudaSuccess;
  size_t blocks = (n_vec + 255) / 256;
  const size_t cap = (size_t)sm_count() * 16;
  if (blocks > cap) blocks = cap;
  ProfileScope prof(KID_COMBINE, st);
  return launch_pdl(round_rows_kernel, (unsigned)blocks, 256, 0, st, reinterpret_cast<const float4*>(acc),
                    static_cast<uint4*>(y), n_vec);
}

}  // namespace tcmoe
