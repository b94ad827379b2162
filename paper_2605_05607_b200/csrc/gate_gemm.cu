// Gate logits on the tensor cores (paper Sec. II-A: the gate network that selects the experts):
//     logits[T, E] = x[T, d] (bf16) * w_gate[d, E] (fp32), fp32 result.
//
// x is bf16, so every product x * w is exact once w is written as hi + mid + lo with three bf16
// terms (8 + 8 + 8 mantissa bits cover fp32's 24): three bf16 UMMAs per k-step into fp32
// accumulators in TMEM (the fp32 ALUs would need 2 T d E flop: 120 GFLOP, 3.7 ms for the
// DeepSeek-V3-shaped layer).
//
// A task is a 128-token x GN-expert tile and the whole of K.  x comes by TMA.  For few tokens sixteen warps (groups that take
// turns) read the fp32 block of w_gate, split it and write the three terms straight into the swizzled MN-major operand tiles:
// no split copy of the weight in memory and no launch for it.  For many tokens every task would split the same blocks again,
// so a kernel before this one writes the terms to the workspace once and they come by TMA too (PRE).
// What bounds it: for few tokens the walk along K, one k-block of 64 after the other, so tiles are
// narrow (a short k-block, and E / GN thread blocks share the work); for many tokens shared-memory
// bandwidth (the UMMAs read the rows of x once per 256 columns), so tiles are wide and two row tiles may share
// a weight block.  Up to 128 experts the three terms are summed apart, as one wide B of 3 GN columns: an
// UMMA takes about 70 cycles for any N up to 128.  More experts keep one running sum (TMEM columns).
// K is never divided over thread blocks, although that would be faster still for a decode batch (9 us
// at T = 64, d = 4096, E = 128): a logit is the same sum in the same order whatever the tile, and a
// different order moves it by up to 1e-4, enough to change the selection of a token whose k-th and next
// key nearly tie.
#include "ffn_common.cuh"

#include <atomic>

namespace tcmoe {
namespace {

using namespace ffn;

constexpr int A_BYTES = BM * BK * 2;            // 16 KiB of x
constexpr int RING_BYTES = 192 * 1024;
constexpr int MAX_STAGES = 8;
constexpr int NUM_BARS = 2 * MAX_STAGES + 1;
constexpr int SMEM_BYTES = 1024 + RING_BYTES + A_BYTES + NUM_BARS * 8 + 64;   // + A_BYTES: see a_bytes
// Warps that split the weight and store the logits; a TMA warp and an UMMA warp follow.  Only stored with PRE: few warps leave
// room for the next kernel's blocks to start early.
__host__ __device__ constexpr int work_warps(bool pre) { return pre ? 4 : 16; }
__host__ __device__ constexpr int threads(bool pre) { return (work_warps(pre) + 2) * 32; }
constexpr int PRE_MIN_TOKENS = 512;             // fewer tokens never take a split copy of the weight: no workspace for it
constexpr double PRE_US = 3.0;                  // its launch
constexpr int STAGE_OUT = 32 * 33;              // floats of a warp's transpose buffer, in the ring
static_assert(16 * STAGE_OUT * 4 <= RING_BYTES, "buffers of all warps");

struct GateParams {
  const float* w;     // [d, E]
  float* logits;      // [T, E]
  int T, d, E, KB, n_tiles;
  int m_sub;          // row tiles per task, 1 or 2: they share the split weight block
  int a_bytes;        // bytes of x per row tile and stage: fewer rows than the tile has are loaded when T is small (the UMMA then
                      // reads whatever follows; only rows >= T depend on it)
  int32_t* status;
};

// ROWS_M: rows of a tile, 64 or 128.  APART: hi, mid and lo sums in accumulators of their own, added at the end; otherwise one
// running sum.  PRE: the three terms come by TMA from the copy that split_gate_kernel made (map_w); the split warps only store.
template <int GN, int GROUPS, int ROWS_M, bool APART, bool PRE>
__global__ void __launch_bounds__(threads(PRE), 1)
gate_umma_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const GateParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RING_BYTES + A_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
  int* abort_s = reinterpret_cast<int*>(tmem_slot + 1);

  const uint32_t smem_base = ptx::smem_u32(smem);
  const uint32_t bar_base = ptx::smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (MAX_STAGES + s); };
  const uint32_t done_bar = bar_base + 8u * (2 * MAX_STAGES);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row0 = (blockIdx.x / p.n_tiles) * p.m_sub * ROWS_M, n0 = (blockIdx.x % p.n_tiles) * GN;
  const int n_sub = p.m_sub > 1 && row0 + ROWS_M < p.T ? 2 : 1;           // row tiles of this task that have rows
  // a stage: hi | mid | lo columns of the weight block side by side in 64-column slabs of 8 KiB, then the x tiles
  constexpr int WARPS = work_warps(PRE), TMA_WARP = WARPS, MMA_WARP = WARPS + 1;
  constexpr int GROUP_WARPS = WARPS / GROUPS;
  constexpr int B_BYTES = (3 * GN + 63) / 64 * 8192;
  // A group that has filled block i knows that block i - n_stages was consumed.  Its next one, i + GROUPS, needs
  // i + GROUPS - 2 n_stages consumed for its parity wait to mean the right phase: no more groups than stages.
  static_assert(GROUPS <= RING_BYTES / (B_BYTES + 2 * A_BYTES) && GROUPS <= MAX_STAGES, "more groups than stages");
  const int stage_bytes = B_BYTES + p.m_sub * p.a_bytes, n_stages = min(MAX_STAGES, RING_BYTES / stage_bytes);
  const int ncols = min(GN, (p.E - n0 + 31) & ~31);                   // expert columns of this tile, zero beyond E

  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_STAGES; ++s) {
      ptx::mbar_init(full_bar(s), PRE ? 1 : GROUP_WARPS + 1);   // one group of split warps + the TMA thread (expect_tx)
      ptx::mbar_init(empty_bar(s), 1);
    }
    ptx::mbar_init(done_bar, 1);
    ptx::fence_mbar_init();
  }
  if (warp == TMA_WARP && lane == 0) {
    ptx::prefetch_tensormap(&map_x);
    if (PRE) ptx::prefetch_tensormap(&map_w);
  }
  if (warp == MMA_WARP) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::tmem_relinquish();
  }
  grid_dependency_sync();   // nothing above touches global data
  if (threadIdx.x == 0) *abort_s = p.status[ST_ABORT];
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  volatile int* abort_flag = abort_s;
  const volatile int* global_abort = p.status + ST_ABORT;
  auto timeout = [&](int detail) {
    report_error(p.status, DEV_TIMEOUT, KID_GATE, detail, blockIdx.x);
    p.status[ST_ABORT] = 1;
    *abort_flag = 1;
  };

  if (warp < WARPS) {
    // ================================ weight block -> three bf16 terms ================================
    // Thread: 8 columns (one 16-byte piece of a swizzle row) of CHUNKS rows of K.  Group g takes every GROUPS-th
    // k-block and keeps DEPTH of its blocks on the way in registers.
    constexpr int PIECES = GN / 8, ROWS = GROUP_WARPS * 32 / PIECES, CHUNKS = BK / ROWS;
    constexpr int DEPTH = CHUNKS >= 4 ? 1 : 4 / CHUNKS;
    static_assert(CHUNKS * ROWS == BK, "whole passes");
    const int group = warp / GROUP_WARPS, tid = threadIdx.x % (GROUP_WARPS * 32);
    const int piece = tid % PIECES, krow = tid / PIECES;
    const int col = n0 + piece * 8;
    const bool vec = (p.E & 3) == 0;                                      // 16-byte vectors, each inside the row or beyond it
    float w[DEPTH][CHUNKS][8];
    auto load = [&](int kb, float (&v)[CHUNKS][8]) {
      const float* src = p.w + (size_t)(kb * BK + krow) * p.E + col;
      if (vec && kb * BK + BK <= p.d) {
#pragma unroll
        for (int c = 0; c < CHUNKS; ++c) {
          const float4* q = reinterpret_cast<const float4*>(src + (size_t)(c * ROWS) * p.E);
          const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 a = col < p.E ? __ldg(q) : zero, b = col + 4 < p.E ? __ldg(q + 1) : zero;
          v[c][0] = a.x; v[c][1] = a.y; v[c][2] = a.z; v[c][3] = a.w;
          v[c][4] = b.x; v[c][5] = b.y; v[c][6] = b.z; v[c][7] = b.w;
        }
      } else {
#pragma unroll
        for (int c = 0; c < CHUNKS; ++c)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            v[c][i] = (kb * BK + c * ROWS + krow < p.d && col + i < p.E) ? __ldg(src + (size_t)(c * ROWS) * p.E + i) : 0.f;
      }
    };
    int s = 0, ph = 1;
    auto advance = [&](int n) {
      for (s += n; s >= n_stages; s -= n_stages) ph ^= 1;
    };
    advance(group);
    auto block = [&](int kb, float (&v)[CHUNKS][8]) {
      if (!ptx::mbar_wait_warp(empty_bar(s), ph, abort_flag, global_abort)) { timeout(2); return false; }
      const uint32_t dst0 = smem_base + s * stage_bytes;
#pragma unroll
      for (int c = 0; c < CHUNKS; ++c) {
        const int k = c * ROWS + krow;
        uint32_t q[3][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float a = v[c][2 * i], b = v[c][2 * i + 1];
#pragma unroll
          for (int t = 0; t < 3; ++t) {   // the remainders are exact
            const __nv_bfloat162 r = __floats2bfloat162_rn(a, b);
            const uint32_t u = *reinterpret_cast<const uint32_t*>(&r);
            q[t][i] = u;
            a = __fsub_rn(a, __uint_as_float(u << 16));
            b = __fsub_rn(b, __uint_as_float(u & 0xFFFF0000u));
          }
        }
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const int at = t * PIECES + piece;   // 16-byte piece of the 3 GN columns
          ptx::st_shared_v4(dst0 + (at >> 3) * 8192 + k * 128 + (((at & 7) ^ (k & 7)) << 4), q[t][0], q[t][1], q[t][2], q[t][3]);
        }
      }
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(full_bar(s));
      if (kb + GROUPS * DEPTH < p.KB) load(kb + GROUPS * DEPTH, v);
      advance(GROUPS);
      return true;
    };
    bool ok = !*abort_flag;
#pragma unroll
    for (int i = 0; i < DEPTH; ++i)
      if (!PRE && ok && group + GROUPS * i < p.KB) load(group + GROUPS * i, w[i]);
    for (int kb = group; !PRE && ok && kb < p.KB; kb += GROUPS * DEPTH) {
#pragma unroll
      for (int i = 0; i < DEPTH; ++i)
        if (ok && kb + GROUPS * i < p.KB) ok = block(kb + GROUPS * i, w[i]);
    }
    // ================================ epilogue ================================
    if (!*abort_flag) {
      if (!ptx::mbar_wait_warp<true>(done_bar, 0, abort_flag, global_abort)) {
        timeout(1);
      } else {
        ptx::tc_fence_after();
        // warp w: TMEM lanes 32 (w % 4) .. + 31, every (warps / 4)-th 32-column block from w / 4 on.  A 64-row accumulator has row
        // 16 q + i in lane 32 q + i (i < 16).
        const int lrow = ROWS_M == 64 ? (lane < 16 ? (warp & 3) * 16 + lane : p.T) : (warp & 3) * 32 + lane;
        constexpr int PARTS = GN > 32 ? GN / 32 : 1;   // of 32 columns (16-column tiles: the upper half is not used)
        for (int u = warp >> 2; u < n_sub * PARTS; u += WARPS / 4) {
          const int i = u / PARTS, c = (u % PARTS) * 32;
          const int row = row0 + i * ROWS_M + lrow;
          if (c >= ncols) continue;
          const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + c;
          uint32_t acc[32];
          if (APART) {   // logits = (hi + mid) + lo
            uint32_t other[32];
            ptx::tmem_ld32(taddr + (i * 3) * GN, acc);
#pragma unroll
            for (int t = 1; t < 3; ++t) {
              ptx::tmem_ld32(taddr + (i * 3 + t) * GN, other);
              ptx::tmem_ld_wait_on(acc);
              ptx::tmem_ld_wait_on(other);
#pragma unroll
              for (int v = 0; v < 32; ++v)
                acc[v] = __float_as_uint(__fadd_rn(__uint_as_float(acc[v]), __uint_as_float(other[v])));
            }
          } else {
            ptx::tmem_ld32(taddr + i * GN, acc);
            ptx::tmem_ld_wait_on(acc);
          }
          if (vec) {
            if (row >= p.T) continue;
            float* out = p.logits + (size_t)row * p.E + n0 + c;
#pragma unroll
            for (int v = 0; v < 8; ++v)
              if (c + v * 4 < GN && n0 + c + v * 4 < p.E)
                *reinterpret_cast<uint4*>(out + v * 4) = make_uint4(acc[v * 4], acc[v * 4 + 1], acc[v * 4 + 2], acc[v * 4 + 3]);
          } else {
            // Rows that start anywhere.  A lane that stores its own row by the element makes 32 pieces of each store, which bounds the
            // kernel for short K; so 32 rows go through the ring, which nothing fills or reads any more, and leave a row per store:
            // route of 16384 tokens, d = 256, 129 experts 36.0 -> 23.5 us, d = 7168, 250 experts 164 -> 149, 12288, 256, 66: 22.9 -> 15.0.
            float* st = reinterpret_cast<float*>(smem) + warp * STAGE_OUT;
#pragma unroll
            for (int v = 0; v < 32; ++v) st[lane * 33 + v] = __uint_as_float(acc[v]);
            __syncwarp();
            const int first = row0 + i * ROWS_M + (warp & 3) * (ROWS_M / 4), rows = min(ROWS_M / 4, p.T - first);
            if (c + lane < GN && n0 + c + lane < p.E) {
              float* out = p.logits + (size_t)first * p.E + n0 + c + lane;
#pragma unroll 8
              for (int r = 0; r < rows; ++r) out[(size_t)r * p.E] = st[r * 33 + lane];
            }
            __syncwarp();
          }
        }
        ptx::tc_fence_before();
      }
    }
  } else if (warp == TMA_WARP) {
    // ================================ TMA producer (rows of x; PRE: the weight's terms) ================================
    if (lane == 0 && !*abort_flag) {
      int s = 0, ph = 1;
      for (int kb = 0; kb < p.KB; ++kb) {
        if (!ptx::mbar_wait(empty_bar(s), ph, abort_flag, global_abort)) { timeout(3); break; }
        ptx::mbar_arrive_expect_tx(full_bar(s), n_sub * p.a_bytes + (PRE ? B_BYTES : 0));
        for (int i = 0; i < n_sub; ++i)
          ptx::tma_load_2d(smem_base + s * stage_bytes + B_BYTES + i * p.a_bytes, &map_x, full_bar(s), kb * BK, row0 + i * ROWS_M);
        if (PRE) {
          static_assert(!PRE || GN % 64 == 0, "a slab of 64 columns holds one term");
#pragma unroll
          for (int c = 0; c < B_BYTES / 8192; ++c)
            ptx::tma_load_3d(smem_base + s * stage_bytes + c * 8192, &map_w, full_bar(s), n0 + c * 64 % GN, kb * BK, c * 64 / GN);
        }
        if (++s == n_stages) { s = 0; ph ^= 1; }
      }
    }
  } else {
    // ================================ UMMA issuer ================================
    if (!*abort_flag) {
      const bool elected = ptx::elect_one();
      const uint32_t base = __shfl_sync(0xFFFFFFFFu, smem_base, 0), tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
      const uint64_t a_desc = desc_at(desc_base(16, 1024), base + B_BYTES), b_desc = desc_at(desc_base(BK * 128, 1024), base);
      auto idesc = [](int n) {
        return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(ROWS_M >> 4) << 24);
      };
      const uint32_t stage16 = stage_bytes >> 4, a16 = p.a_bytes >> 4;
      bool ok = true;
      int s = 0, ph = 0;
      // For few tokens the loop is bound by its own instructions, 530 cycles per k-block, half of them to issue the UMMAs.  The vote
      // makes the exit uniform for the compiler, and a known number of row tiles leaves the descriptors in uniform registers: moe_route of
      // (T, d, E), us, 1, 4096, 8: 21.7 -> 18.3; 5, 5744, 64: 29.5 -> 24.9; 128, 7168, 256: 50.3 -> 40.2.
      for (int kb = 0; kb < p.KB; ++kb) {
        if (__any_sync(0xFFFFFFFFu, !ptx::mbar_wait(full_bar(s), ph, abort_flag, global_abort))) { timeout(4); ok = false; break; }
        ptx::tc_fence_after();
        if (elected) {
          for (int i = 0; i < (GN <= 32 ? 1 : n_sub); ++i) {   // (up to 32 columns: one row tile)
            const uint64_t ad = a_desc + (s * stage16 + i * a16), bd = b_desc + s * stage16;
            if (APART) {   // the terms as one wide B
              constexpr int N1 = 3 * GN < 256 ? 3 * GN : 256, N2 = 3 * GN - N1;
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) {
                const uint32_t d = tmem + i * 3 * GN;
                ptx::umma_bf16(d, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * 128), idesc(N1), (kb | k) > 0);
                if (N2 > 0)
                  ptx::umma_bf16(d + N1, ad + (uint64_t)(k * 2), bd + (uint64_t)(N1 / 64 * 512 + k * 128), idesc(N2), (kb | k) > 0);
              }
            } else {
#pragma unroll
              for (int t = 0; t < 3; ++t)
#pragma unroll
                for (int k = 0; k < BK / 16; ++k)
                  ptx::umma_bf16(tmem + i * GN, ad + (uint64_t)(k * 2), bd + (uint64_t)((t * GN / 64) * 512 + (t * GN % 64) / 8 + k * 128), idesc(GN),
                                 (kb | k | t) > 0);
            }
          }
          ptx::umma_commit(empty_bar(s));
        }
        if (++s == n_stages) { s = 0; ph ^= 1; }
      }
      if (ok && elected) ptx::umma_commit(done_bar);
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    for (int i = 0; i < 64; ++i) __nanosleep(1000);   // abort path: let bulk copies in flight land
  }
  __syncthreads();
  if (warp == MMA_WARP) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, 512);
  }
}

// w_gate fp32 [d, E] -> bf16 [3, d, cols]: hi, mid, lo terms, zero in the padding columns
__global__ void __launch_bounds__(256) split_gate_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ out, int d, int E,
                                                         int cols) {
  grid_dependency_sync();
  const size_t n = (size_t)d * cols;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int row = (int)(i / cols), col = (int)(i % cols);
    float v = col < E ? __ldg(w + (size_t)row * E + col) : 0.f;
#pragma unroll
    for (int t = 0; t < 3; ++t) {   // the remainders are exact
      const __nv_bfloat16 r = __float2bfloat16_rn(v);
      out[t * n + i] = r;
      v = __fsub_rn(v, __bfloat162float(r));
    }
  }
}

// Tile width, rows of a tile, row tiles per task and where the terms of the weight come from: the cheapest by a model in
// microseconds that is fitted to this kernel: tasks go in rounds of one per SM, a round costs `start` and a time per k-block of
// 64; rows of w_gate whose length is no multiple of 4 are read by the element, which the forms that split inside the GEMM pay in
// every k-block (16384 tokens, d = 7168: 256 experts 178 us, 250 experts 236).  The split copy costs a launch.
// Tiles of 64 rows halve what a UMMA reads of x, which counts where twelve of them make a k-block (running sum: 128 tokens
// of d = 7168, 256 experts 66 -> 48 us); with the terms apart they change nothing.
// moe_route of (T, d, E), us, without the split copy / with this table: 16384, 2880, 65: 61.4 / 50.4; 16384, 2880, 128: 53.0 / 49.4;
// 32768, 2880, 96: 102 / 92; 8192, 7168, 256: 115 / 85; 32768, 7168, 250: 459 / 335; 4097, 7168, 258: 194 / 90 (the last two
// 315 -> 291 and 98 -> 91 in a replayed graph since ragged rows of logits leave whole).
// Up to 128 experts tiles of 16 columns where the SMs take them in as many rounds: a block has half the weight to split and less to
// move through shared memory per k-block, moe_route of (T, d, E), us, 32 / 16 columns: 64, 4096, 128 23.5 / 20.6; 300, 4096, 65 30.2 / 24.5;
// 872, 6832, 16 35.8 / 27.8; 1669, 3520, 64 23.9 / 19.4; 200, 256, 64 7.0 / 6.3.  With more than 64 experts a hundred blocks of them get in each
// other's way, 2.4 us whatever K (1659, 256, 128: 9.8 / 10.0, 1915 tokens 9.8 / 12.1; of d = 1024 13.7 / 13.9, 13.8 / 16.0, of d = 4096 28.8 / 24.3,
// 28.7 / 26.7).
struct GatePlan { int gn, bm, m_sub; bool pre; };
GatePlan plan_gate(int T, int d, int E) {
  struct Cost { double start, kb, kb_ragged; };
  constexpr Cost NO = {1e9, 0, 0};
  static const struct { GatePlan form; Cost running, apart; } forms[] = {
      {{32, 64, 1, false}, {4, 0.37, 0.38}, NO},
      {{64, 64, 1, false}, {4, 0.43, 0.63}, NO},
      {{16, 128, 1, false}, NO, {4.8, 0.24, 0.27}},
      {{32, 128, 1, false}, {4.3, 0.455, 0.46}, {4.5, 0.318, 0.345}},
      {{64, 128, 1, false}, {4.8, 0.525, 0.66}, NO},
      {{64, 128, 2, false}, {7, 0.83, 0.87}, {8, 0.63, 0.68}},
      {{64, 128, 1, true}, NO, {4.8, 0.33, 0.33}},
      {{128, 128, 1, true}, {4.8, 0.58, 0.58}, {6, 0.49, 0.49}},
      {{128, 128, 2, true}, {9, 1.04, 1.04}, NO}};
  GatePlan best{};
  double best_us = 1e30;
  for (const auto& f : forms) {
    if (f.form.pre && T < PRE_MIN_TOKENS) continue;
    const Cost& c = E <= 128 ? f.apart : f.running;
    const int rows = f.form.m_sub * f.form.bm, sms = sm_count();
    const long long tasks = (long long)((T + rows - 1) / rows) * ((E + f.form.gn - 1) / f.form.gn);
    const double round = c.start + ((d + BK - 1) / BK) * (E % 4 == 0 ? c.kb : c.kb_ragged);
    const double crowd = f.form.gn == 16 && E > 64 && tasks > 100 ? 2.4 : 0.0;
    const double us = (double)((tasks + sms - 1) / sms) * round + (f.form.pre ? PRE_US : 0.0) + crowd;
    if (us < best_us) { best_us = us; best = f.form; }
  }
  return best;
}

template <int GN, int GROUPS, int ROWS_M, bool APART, bool PRE = false>
cudaError_t launch_width(const GateParams& p, int grid, const CUtensorMap& m_x, const CUtensorMap& m_w, cudaStream_t st) {
  // per device; several host threads may get here at once: setting the attribute twice is harmless
  static std::atomic<bool> attr_set[MAX_DEVICES];
  const int dev = current_device();
  const auto kernel = gate_umma_kernel<GN, GROUPS, ROWS_M, APART, PRE>;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  return launch_pdl(kernel, grid, threads(PRE), SMEM_BYTES, st, m_x, m_w, p);
}

}  // namespace

size_t gate_split_bytes(const Shape& s) {
  return s.T < PRE_MIN_TOKENS ? 0 : (size_t)3 * s.d * ((s.E + 63) & ~63) * 2;
}

cudaError_t launch_gate_logits(const Shape& s, const void* x, const float* w_gate, float* logits, void* wsplit, int32_t* status,
                               cudaStream_t st) {
  if (s.T == 0) return cudaSuccess;
  const bool apart = s.E <= 128;
  const GatePlan plan = plan_gate(s.T, s.d, s.E);
  const int a_rows = s.T < plan.bm ? (s.T + 7) & ~7 : plan.bm;
  CUtensorMap m_x, m_w{};
  {
    cuuint64_t dims[2] = {(cuuint64_t)s.d, (cuuint64_t)s.T};
    cuuint64_t strides[1] = {(cuuint64_t)s.d * 2};
    cuuint32_t box[2] = {BK, (cuuint32_t)a_rows};
    if (!ffn::encode_tiled(&m_x, false, 2, x, dims, strides, box)) return cudaErrorInvalidValue;
  }
  ProfileScope prof(KID_GATE, st);
  if (plan.pre) {
    const int cols = (s.E + 63) & ~63;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)s.d, 3};
    cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)cols * s.d * 2};
    cuuint32_t box[3] = {64, BK, 1};
    if (!ffn::encode_tiled(&m_w, false, 3, wsplit, dims, strides, box)) return cudaErrorInvalidValue;
    size_t blocks = ((size_t)s.d * cols + 255) / 256;
    if (blocks > (size_t)sm_count() * 8) blocks = (size_t)sm_count() * 8;
    cudaError_t err = launch_pdl(split_gate_kernel, (unsigned)blocks, 256, 0, st, w_gate, static_cast<__nv_bfloat16*>(wsplit), s.d,
                                 s.E, cols);
    if (err != cudaSuccess) return err;
  }
  GateParams p;
  p.w = w_gate;
  p.logits = logits;
  p.T = s.T;
  p.d = s.d;
  p.E = s.E;
  p.KB = (s.d + BK - 1) / BK;
  p.n_tiles = (s.E + plan.gn - 1) / plan.gn;
  p.m_sub = plan.m_sub;
  p.a_bytes = a_rows * BK * 2;
  p.status = status;
  const int grid = ((s.T + p.m_sub * plan.bm - 1) / (p.m_sub * plan.bm)) * p.n_tiles;
  if (plan.pre) {
    if (!apart) return launch_width<128, 1, 128, false, true>(p, grid, m_x, m_w, st);
    if (plan.gn == 64) return launch_width<64, 1, 128, true, true>(p, grid, m_x, m_w, st);
    return launch_width<128, 1, 128, true, true>(p, grid, m_x, m_w, st);
  }
  if (apart) {
    if (plan.gn == 16) return launch_width<16, 4, 128, true>(p, grid, m_x, m_x, st);
    if (plan.gn == 32) return launch_width<32, 4, 128, true>(p, grid, m_x, m_x, st);
    return launch_width<64, 2, 128, true>(p, grid, m_x, m_x, st);
  }
  if (plan.bm == 64 && plan.gn == 32) return launch_width<32, 4, 64, false>(p, grid, m_x, m_x, st);
  if (plan.bm == 64) return launch_width<64, 2, 64, false>(p, grid, m_x, m_x, st);
  if (plan.gn == 32) return launch_width<32, 4, 128, false>(p, grid, m_x, m_x, st);
  return launch_width<64, 2, 128, false>(p, grid, m_x, m_x, st);
}

}  // namespace tcmoe
