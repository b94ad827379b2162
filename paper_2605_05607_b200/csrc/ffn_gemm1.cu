// GEMM-1 of the expert FFN with the SwiGLU epilogue (paper Sec. II-A "GEMM-1"; Sec. IV: the
// dispatch gather is the GEMM's prologue, tiles of 128 tokens):
//     h[r, n] = silu(a_r . W1[e][:, n]) * (a_r . W3[e][:, n]),   a_r = src[gather_idx[r] / gather_div]
//
// A rows are GATHERED (they are arbitrary rows of the dispatched buffer, or of x itself in the
// fused layer) by cp.async into the 128-byte swizzled K-major layout the UMMA descriptor expects;
// B = two 64-column slabs of W1 and the same two of W3 loaded by TMA side by side, so that ONE
// 128 x 256 x 16 UMMA yields both products (accumulator columns [0,128) = a.W1, [128,256) = a.W3).
//
// One persistent CTA per SM (tcgen05 cta_group::1) walks tile tasks decoded from the device-side
// tile prefix, so no routing-dependent quantity visits the host.  Warp roles: epilogue
// (TMEM -> registers -> SwiGLU -> global), one TMA producer, one UMMA issuer and TMEM owner, four gather
// producers.  Accumulators are double-buffered in TMEM (2 x 256 columns): the epilogue of tile i
// overlaps the main loop of tile i+1.  Every wait is bounded.
//
// Pipeline: 4 stages, each an A tile (16 KiB, gathered) and a B tile (32 KiB, TMA) behind one
// full / one empty barrier.  The gather threads never wait for their own copies: after issuing the
// cp.async copies of a stage each thread posts cp.async.mbarrier.arrive.noinc on the stage's full
// barrier, so the barrier completes exactly when the last row has landed (and the TMA bytes are
// in), independent of how far the issuing threads have moved on.  An earlier form published a
// stage only when the copies of two later stages had been issued (commit groups, wait, proxy
// fence, arrive): the publication then trailed the tensor pipe by one stage and the kernel ran
// 8-11 % (K = 4096) to 30 % (K = 7168, rows gathered from DRAM) slower; deeper or split A / B
// rings on that form recovered only part of it and cost a second wait per k-block.
//
// CTA-pair (cta_group::2) variants of this kernel were measured and not kept.  With lagged
// publication they lost by 20-60 %; with self-arriving copies (the peer CTA's arrivals relayed to the
// leader's barrier by one thread, with a RELAXED cluster-scope arrive: a releasing one waits for the
// copies the SM has in flight and held the kernel at 0.83 us per stage) the paired form reaches the
// same UMMA rate as this kernel and then loses 4 % to the padding of 256-row tiles.  TMA
// tile::gather4 as the gather engine sustains only one 4-row instruction per ~40 ns.
#include "ffn_common.cuh"

#include <atomic>

namespace tcmoe {
namespace ffn {
namespace {

constexpr int RING_BYTES = 192 * 1024;       // 4 stages of A + a 256-column B, more of narrower ones
constexpr int MAX_STAGES = 12;            // 64 rows x 64 columns: 16 KiB
constexpr int NUM_BARS = 2 * MAX_STAGES + 4;
// Four epilogue warps, one per row quarter, or eight (two per quarter, half of the columns each) where a tile's epilogue takes longer than its
// main loop (512 cycles per 128 bytes of K) or is most of a layer's last round: see launch_width.
__host__ __device__ constexpr int epi_warps(bool eight) { return eight ? 8 : 4; }
constexpr int EPI_WARPS_MAX = 8;
constexpr int STAGE_OUT_WARP = 32 * 64;      // epilogue transpose buffer of one warp: 32 rows x 32 columns, swizzled
constexpr int TABLE_BYTES = (2 * (MAX_E + 1) * 4 + 15) & ~15;
constexpr int COLSCALE_WARP = UMMA_N / 2 * 4;   // FP8: one warp's copy of the scales of its columns (half of the accumulator's with eight warps)
constexpr int SMEM_BYTES =
    1024 + RING_BYTES + NUM_BARS * 8 + 64 + TABLE_BYTES + EPI_WARPS_MAX * (STAGE_OUT_WARP + COLSCALE_WARP);
constexpr int GATHER_THREADS = 128;
__host__ __device__ constexpr int threads(bool eight) { return (epi_warps(eight) + 2) * 32 + GATHER_THREADS; }
// The producers (TMA thread, 128 gather threads) wait for a free stage with a suspend-time hint: parked in hardware
// instead of polling.  At the board's power limit the layer's time follows energy: GEMM-1 alone in a loop on the
// DeepSeek-V3 shape 15.78 -> 15.50 ms with the hint (two alternations, same box), a single cold launch 13.41 -> 13.48.
// The UMMA thread's wait for a full stage is on the critical path and keeps the plain form (hinting it too gives the
// gain back).
constexpr uint32_t FEED_HINT = 1000;
constexpr int SWAP_ROWS = 96;   // see `swapped`

// FP8 = true: A rows and weights are E4M3 codes, a stage holds 128 elements of K (the same 128
// bytes per row), W1 / W3 come K-major from [E, N, K] as two 128-row boxes, and the epilogue applies
// a_scale[source row] * b_scale[e, n] before the SwiGLU; h is written as bf16 either way.
//
// PLAIN = true turns the kernel into a single-CTA form of GEMM-2 (Sec. II-A "GEMM-2", gate weight in the
// epilogue, Sec. III-C): the "gather" reads the rows of h in place (gather_idx = NULL), both halves of
// the 256-column B tile come from the one weight map (map_w1), the epilogue writes
// o[r, n] = w_r * acc[r, n] for 256 columns.  Used instead of the CTA-pair kernel when experts are small
// (128-row tiles pad far less than 256-row pair tiles when most experts hold fewer than 128 rows).
//
// NARROW = true: tiles of a quarter (PLAIN: 64 columns) or half the width (64 columns of W1 and of W3), for layers with fewer
// full-width tiles than SMs: one decoded token reads two wide experts' weights through 32 full-width tiles of GEMM-2.  The
// sums are the same, element by element.
//
// FEW = true (narrow tiles only): tiles of 64 rows, for layers of at most 64 rows in all.  A stage is then a third smaller and
// the ring holds more of the weights in flight (96 KiB instead of 64 in GEMM-2), which is what bounds a CTA that streams a column
// slab of one expert: GEMM-2 of one token, top-2 of d = 4096, f = 14336, 58 -> 46 us (4.1 -> 5.1 TB/s).
template <bool FP8, bool PLAIN, bool NARROW, bool FEW, bool EIGHT>
__global__ void __launch_bounds__(threads(EIGHT), 1)
ffn_gemm1_kernel(const __grid_constant__ CUtensorMap map_w1, const __grid_constant__ CUtensorMap map_w3,
                 const GemmParams p) {
  constexpr int BN = !NARROW ? UMMA_N : PLAIN ? 64 : 128;   // accumulator columns of a tile
  constexpr int BN_OUT = PLAIN ? BN : BN / 2;               // output columns
  constexpr int HALF = BN > 64 ? BN / 2 : BN;               // columns from each of the two weight maps (BN = 64: one)
  constexpr int ROWS = FEW ? 64 : BM;                       // rows of a tile
  constexpr int WROWS = ROWS / 4;                           // rows of an epilogue warp: TMEM lanes 32 q .. 32 q + WROWS - 1
  constexpr int EPI_WARPS = epi_warps(EIGHT), TMA_WARP = EPI_WARPS, MMA_WARP = EPI_WARPS + 1, GATHER_WARP = EPI_WARPS + 2;
  constexpr int WCOLS = BN_OUT / (EPI_WARPS / 4);           // output columns of an epilogue warp
  constexpr int SCALES = UMMA_N / (EPI_WARPS / 4);          // FP8: floats of its column scales
  static_assert(NARROW || !FEW, "64-row tiles come with narrow ones");
  constexpr int A_BYTES = ROWS * BK * 2;
  constexpr int B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;   // B: 64-column slabs of 8 KiB
  constexpr int NSTAGE = RING_BYTES / STAGE_BYTES;
  static_assert(NSTAGE <= MAX_STAGES, "barriers");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RING_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
  int* abort_s = reinterpret_cast<int*>(tmem_slot + 1);
  int* tp_s = reinterpret_cast<int*>(tmem_slot + 16);
  int* eoff_s = tp_s + (MAX_E + 1);
  const uint32_t stage_base = ptx::smem_u32(tp_s) + TABLE_BYTES;   // 16-byte aligned
  float* colscale_base = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(tp_s) + TABLE_BYTES + EPI_WARPS_MAX * STAGE_OUT_WARP);

  const uint32_t smem_base = ptx::smem_u32(smem);
  const uint32_t bar_base = ptx::smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (MAX_STAGES + s); };
  auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * MAX_STAGES + b); };
  auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * MAX_STAGES + 2 + b); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      ptx::mbar_init(full_bar(s), GATHER_THREADS + 1);   // every gather thread's copies + the TMA thread (expect_tx)
      ptx::mbar_init(empty_bar(s), 1);                   // tcgen05.commit
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(tfull_bar(b), 1);      // tcgen05.commit
      ptx::mbar_init(tempty_bar(b), EPI_WARPS);   // one lane per epilogue warp
    }
    ptx::fence_mbar_init();
  }
  if (warp == TMA_WARP && lane == 0) {
    ptx::prefetch_tensormap(&map_w1);
    ptx::prefetch_tensormap(&map_w3);
  }
  if (warp == MMA_WARP) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
    ptx::tmem_relinquish();
  }
  // GEMM-2 reads nothing of the kernel before it but the rows (and their scales): its tables and weights were there before that kernel
  // started, which in turn let this one start only after its own wait.  So the weights of the first stages are fetched while the
  // other thread blocks of that kernel finish, and only the warps that touch rows wait.
  if (!PLAIN) grid_dependency_sync();   // nothing above touches global data
  for (int i = threadIdx.x; i <= p.E; i += blockDim.x) {
    tp_s[i] = __ldcg(p.tile_prefix + i);
    eoff_s[i] = __ldcg(p.expert_offsets + i);
  }
  if (threadIdx.x == 0) *abort_s = p.status[ST_ABORT];
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int total = tp_s[p.E] * p.n_tiles;
  constexpr int BK_ELEMS = FP8 ? 2 * BK : BK;   // K elements per stage: 128 bytes per row either way
  const int KB = (p.K + BK_ELEMS - 1) / BK_ELEMS;
  volatile int* abort_flag = abort_s;
  const volatile int* global_abort = p.status + ST_ABORT;

  auto timeout = [&](int detail) {
    report_error(p.status, DEV_TIMEOUT, PLAIN ? KID_GEMM2 : KID_GEMM1, detail, blockIdx.x);
    p.status[ST_ABORT] = 1;
    *abort_flag = 1;
  };
  // An expert of at most 96 rows exchanges the operands: the tile's weight columns are the M side (two UMMAs of 128), its rows, rounded
  // up to 16, the N side.  A layer of such experts streams weights at the board's power limit, and an UMMA of 128 rows, most of
  // them padding, over 256 columns costs energy (and copies of zero rows) for the padding too.  Same sums, same bits.
  // Layers in a loop, us, rows per expert in brackets: 64 tokens, top-8 of 128 x 4096 x 1536 (4) 766 -> 722, 128 tokens, 256 x 7168 x 2048
  // in 8 bits (4) 1930 -> 1733, 1777 skewed tokens, 128 x 2880 x 2880 946 -> 894, 1200, 128 x 2880 x 2880 in 8 bits (75) 706 -> 686,
  // 500 top-4 of 32 x 4096 x 1536 (62) 253 -> 249, 800 top-8 of 64 x 2048 x 2048 (100) 343 -> 344; up to 64 rows only: 1200 in 8 bits 703;
  // up to 128: 800 tokens 350.  The last tile of a larger expert keeps the plain form: a CTA that is done with it earlier leaves the
  // company of those that read the same weights (32768 tokens, 256 x 7168 x 2048: 23100 -> 25900).
  auto swapped = [&](const Tile& t) { return !NARROW && t.rows <= SWAP_ROWS && t.row0 == eoff_s[t.e]; };
  auto tile_of = [&](int w) { return decode_tile(w, tp_s, eoff_s, p.E, p.n_tiles, BN_OUT, BM, 0); };

  if (warp < EPI_WARPS) {
    // ================================ epilogue ================================
    if (PLAIN) grid_dependency_sync();
    const int quarter = warp & 3, half = warp >> 2;   // TMEM lanes this warp owns, and which half of their columns with eight warps
    int tl = 0;
    for (int w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x, ++tl) {
      const Tile t = tile_of(w);
      const int buf = tl & 1;
      if (!ptx::mbar_wait_warp<true>(tfull_bar(buf), (tl >> 1) & 1, abort_flag, global_abort)) { timeout(1); break; }
      ptx::tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN);
      // A thread owns one accumulator row; 32 threads storing 16 bytes each to 32 different rows would cost 32 memory transactions per
      // instruction.  The warp transposes 32 output columns at a time through shared memory (64-byte rows, pieces swizzled by row pair:
      // conflict-free both ways) and stores 64-byte row segments, 8 rows per instruction.
      const uint32_t stage = stage_base + (uint32_t)(warp * STAGE_OUT_WARP);
      const int srow = lane >> 2, piece = lane & 3;
      auto put = [&](int v, uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3) {   // columns 8 v .. + 7 of this thread's row
        ptx::st_shared_v4(stage + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4), q0, q1, q2, q3);
      };
      auto send = [&](int at) {   // 32 staged columns, from column `at` of the tile on, to the rows of out
        __syncwarp();
        const int col = t.n0 + at + piece * 8;
        if (col < p.N) {
#pragma unroll
          for (int i = 0; i < WROWS / 8; ++i) {
            const int r = i * 8 + srow;   // row of this warp's
            if (quarter * WROWS + r < t.rows)
              *reinterpret_cast<uint4*>(p.out + (size_t)(t.row0 + quarter * WROWS + r) * (size_t)p.out_ld + col) =
                  ptx::ld_shared_v4(stage + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4));
          }
        }
        __syncwarp();
      };
      if (swapped(t)) {
        // lane = output column of a half tile (GEMM-1: the same column of W1 and of W3), TMEM column = row
        const int c = quarter * 32 + lane, odd = lane & 1;
        const size_t sc = (size_t)t.e * p.N + t.n0 + c;
        float sa = 1.f, sb = 1.f;   // FP8: column scales
        if (FP8) {
          const int hi = PLAIN ? HALF : 0;
          sa = t.n0 + c < p.N ? __ldg(p.b_scale + sc) : 0.f;
          sb = t.n0 + hi + c < p.N ? __ldg((PLAIN ? p.b_scale : p.b_scale2) + sc + hi) : 0.f;
        }
#pragma unroll 1
        for (int r0 = half * 16; r0 < t.rows; r0 += EPI_WARPS * 4) {   // the warps of a quarter take turns
          const int mine = r0 + (lane & 15);
          float rs = 1.f;   // scale of this lane's row of the 16
          if (mine < t.rows) {
            const size_t grow = (size_t)t.row0 + mine;
            if (PLAIN) {
              if (p.topk_w != nullptr) rs = __ldg(p.topk_w + __ldg(p.row_pair + grow));
              if (FP8) rs *= __ldg(p.a_scale + grow);
            } else if (FP8) {
              int idx = __ldg(p.gather_idx + grow);
              if (p.gather_div > 1) idx /= p.gather_div;
              rs = (idx >= 0 && idx < p.a_rows) ? __ldg(p.a_scale + idx) : 0.f;
            }
          }
          uint32_t a[16], b[16];
          ptx::tmem_ld16(taddr + r0, a);
          ptx::tmem_ld16(taddr + HALF + r0, b);
          ptx::tmem_ld_wait_on(a, b);
          // two rows at a time: neighbouring lanes swap, and each stores two columns of one of the rows
          auto put = [&](float v0, float v1, int r, int col) {
            const float got = __shfl_xor_sync(0xFFFFFFFFu, odd ? v0 : v1, 1);
            const int row = r0 + r + odd, at = col - odd;
            if (row < t.rows && at < p.N)
              *reinterpret_cast<uint32_t*>(p.out + (size_t)(t.row0 + row) * (size_t)p.out_ld + at) = odd ? pack2(got, v1) : pack2(v0, got);
          };
#pragma unroll
          for (int r = 0; r < 16; r += 2) {
            const float w0 = __shfl_sync(0xFFFFFFFFu, rs, r), w1 = __shfl_sync(0xFFFFFFFFu, rs, r + 1);
            float a0 = __uint_as_float(a[r]), a1 = __uint_as_float(a[r + 1]), b0 = __uint_as_float(b[r]), b1 = __uint_as_float(b[r + 1]);
            if (PLAIN) {
              put(w0 * (FP8 ? a0 * sa : a0), w1 * (FP8 ? a1 * sa : a1), r, t.n0 + c);
              put(w0 * (FP8 ? b0 * sb : b0), w1 * (FP8 ? b1 * sb : b1), r, t.n0 + HALF + c);
            } else {
              if (FP8) { a0 *= w0 * sa; b0 *= w0 * sb; a1 *= w1 * sa; b1 *= w1 * sb; }
              put(silu_mul(a0, b0), silu_mul(a1, b1), r, t.n0 + c);
            }
          }
        }
      } else if (PLAIN) {
        // ---- GEMM-2 form: o = (gate weight x row scale) * acc * column scale
        const int lrow = quarter * WROWS + lane;
        float wr = 1.f;
        if (lane < WROWS && lrow < t.rows) {
          const size_t grow = (size_t)t.row0 + lrow;
          if (p.topk_w != nullptr) wr = __ldg(p.topk_w + __ldg(p.row_pair + grow));
          if (FP8) wr *= __ldg(p.a_scale + grow);
        }
        float* sb_col = colscale_base + warp * SCALES;   // scales of this warp's columns (0 beyond N)
        if (FP8) {
          const int n0 = t.n0 + half * WCOLS;
          const float* g = p.b_scale + (size_t)t.e * p.N + n0;
#pragma unroll
          for (int i = 0; i < WCOLS / 32; ++i) {
            const int n = lane + 32 * i;
            sb_col[n] = (n0 + n < p.N) ? __ldg(g + n) : 0.f;
          }
          __syncwarp();
        }
#pragma unroll 1
        for (int c = 0; c < WCOLS / 32; ++c) {
          uint32_t acc[32];
          ptx::tmem_ld32(taddr + half * WCOLS + c * 32, acc);
          ptx::tmem_ld_wait_on(acc);
          if (FP8) {
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(__uint_as_float(acc[j]) * sb_col[c * 32 + j]);
          }
#pragma unroll
          for (int v = 0; v < 4; ++v)
            put(v, pack2(wr * __uint_as_float(acc[v * 8]), wr * __uint_as_float(acc[v * 8 + 1])),
                pack2(wr * __uint_as_float(acc[v * 8 + 2]), wr * __uint_as_float(acc[v * 8 + 3])),
                pack2(wr * __uint_as_float(acc[v * 8 + 4]), wr * __uint_as_float(acc[v * 8 + 5])),
                pack2(wr * __uint_as_float(acc[v * 8 + 6]), wr * __uint_as_float(acc[v * 8 + 7])));
          send(half * WCOLS + c * 32);
        }
      } else {
        // ---- GEMM-1 form: SwiGLU of the W1 / W3 halves
        float sa = 1.f;   // FP8: scale of this thread's row (the gather source row)
        float* s1 = colscale_base + warp * SCALES;   // the W1 / W3 scales of this warp's columns (0 beyond N)
        float* s3 = s1 + WCOLS;
        if (FP8) {
          const int lrow = quarter * WROWS + lane, n0 = t.n0 + half * WCOLS;
          if (lane < WROWS && lrow < t.rows) {
            int idx = __ldg(p.gather_idx + t.row0 + lrow);
            if (p.gather_div > 1) idx /= p.gather_div;
            sa = (idx >= 0 && idx < p.a_rows) ? __ldg(p.a_scale + idx) : 0.f;
          }
          const size_t g = (size_t)t.e * p.N + n0;
#pragma unroll
          for (int i = 0; i < WCOLS / 32; ++i) {
            const int n = lane + 32 * i;
            const bool in = n0 + n < p.N;
            s1[n] = in ? (__ldg(p.b_scale + g + n)) : 0.f;
            s3[n] = in ? (__ldg(p.b_scale2 + g + n)) : 0.f;
          }
          __syncwarp();
        }
#pragma unroll 1
        for (int c = 0; c < WCOLS / 32; ++c) {
          uint32_t a1[32], a3[32];
          ptx::tmem_ld32(taddr + half * WCOLS + c * 32, a1);
          ptx::tmem_ld32(taddr + BN_OUT + half * WCOLS + c * 32, a3);
          ptx::tmem_ld_wait_on(a1, a3);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            uint32_t q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int j = v * 8 + 2 * i;
              float u0 = __uint_as_float(a1[j]), u1 = __uint_as_float(a1[j + 1]);
              float g0 = __uint_as_float(a3[j]), g1 = __uint_as_float(a3[j + 1]);
              if (FP8) {
                const int n = c * 32 + j;
                u0 *= sa * s1[n];
                g0 *= sa * s3[n];
                u1 *= sa * s1[n + 1];
                g1 *= sa * s3[n + 1];
              }
              q[i] = pack2(silu_mul(u0, g0), silu_mul(u1, g1));
            }
            put(v, q[0], q[1], q[2], q[3]);
          }
          send(half * WCOLS + c * 32);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(tempty_bar(buf));
    }
  } else if (warp == TMA_WARP) {
    // ================================ TMA producer (weights) ================================
    if (lane == 0) {
      uint32_t it = 0;
      for (int w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x) {
        const Tile t = tile_of(w);
        bool ok = true;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % NSTAGE;
          if (!ptx::mbar_wait<false, FEED_HINT>(empty_bar(s), ((it / NSTAGE) & 1) ^ 1, abort_flag, global_abort)) {
            timeout(2); ok = false; break;
          }
          const uint32_t sb = smem_base + s * STAGE_BYTES + A_BYTES;
          ptx::mbar_arrive_expect_tx(full_bar(s), B_BYTES);
          const int k0 = kb * BK_ELEMS;
          const CUtensorMap* hi_map = PLAIN ? &map_w1 : &map_w3;   // second half of the accumulator columns
          const int hi_n = PLAIN ? t.n0 + HALF : t.n0;
          if (FP8) {   // K-major boxes of HALF output columns x 128 bytes of K
            ptx::tma_load_3d(sb, &map_w1, full_bar(s), k0, t.n0, t.e);
            if (BN > HALF) ptx::tma_load_3d(sb + HALF * 128, hi_map, full_bar(s), k0, hi_n, t.e);
          } else {     // MN-major slabs of 64 output columns x 64 rows of K
#pragma unroll
            for (int c = 0; c < BN / 64; ++c) {
              const bool hi = c * 64 >= HALF;
              ptx::tma_load_3d(sb + c * 8192, hi ? hi_map : &map_w1, full_bar(s), (hi ? hi_n - HALF : t.n0) + c * 64, k0, t.e);
            }
          }
        }
        if (!ok) break;
      }
    }
  } else if (warp == MMA_WARP) {
    // ================================ UMMA issuer ================================
    // the warp walks the loop, one elected lane issues (see ptx::elect_one)
    const bool elected = ptx::elect_one();
    const uint32_t base = __shfl_sync(0xFFFFFFFFu, smem_base, 0), tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
    const uint64_t a_desc = desc_at(desc_base(16, 1024), base);
    const uint64_t b_desc = desc_at(FP8 ? desc_base(16, 1024) : desc_base(BK * 128, 1024), base + A_BYTES);   // K-major : MN-major
    constexpr uint32_t IDESC = FP8 ? idesc_e4m3(ROWS, BN) : idesc_bf16(ROWS, BN);
    constexpr int B_STEP = FP8 ? 2 : 128;   // 32 bytes of K per UMMA (16 bf16 / 32 E4M3): +32 B inside the swizzle row, or +2 atoms
    int s = 0, tl = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int w = blockIdx.x; ok && w < total && !*abort_flag; w += gridDim.x, ++tl) {
      const int buf = tl & 1;
      if (!ptx::mbar_wait(tempty_bar(buf), ((tl >> 1) & 1) ^ 1, abort_flag, global_abort)) { timeout(3); break; }
      ptx::tc_fence_after();
      const uint32_t d_tmem = tmem + (uint32_t)(buf * BN);
      // one k-block after the other; an elected lane runs `issue` on the stage's operands
      auto walk = [&](auto issue) {
        for (int kb = 0; kb < KB; ++kb) {
          if (!ptx::mbar_wait(full_bar(s), ph, abort_flag, global_abort)) { timeout(4); return false; }
          ptx::tc_fence_after();
          if (elected) {
            issue(a_desc + (uint64_t)(s * (STAGE_BYTES >> 4)), b_desc + (uint64_t)(s * (STAGE_BYTES >> 4)), kb);
            ptx::umma_commit(empty_bar(s));   // free the stage when these UMMAs have read it
          }
          if (++s == NSTAGE) { s = 0; ph ^= 1u; }
        }
        return true;
      };
      auto mma = [](uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, bool acc) {
        if (FP8) ptx::umma_f8(d, ad, bd, idesc, acc);
        else ptx::umma_bf16(d, ad, bd, idesc, acc);
      };
      const Tile t = tile_of(w);
      if (swapped(t)) {
        const uint32_t idesc = idesc_swapped(FP8, (t.rows + 15) & ~15);
        ok = walk([&](uint64_t ad, uint64_t bd, int kb) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h)
              mma(d_tmem + h * HALF, bd + (uint64_t)(k * B_STEP + h * (HALF * 128 >> 4)), ad + (uint64_t)(k * 2), idesc, (kb | k) != 0);
        });
      } else {
        ok = walk([&](uint64_t ad, uint64_t bd, int kb) {
#pragma unroll
          for (int k = 0; k < 4; ++k) mma(d_tmem, ad + (uint64_t)(k * 2), bd + (uint64_t)(k * B_STEP), IDESC, (kb | k) != 0);
        });
      }
      if (ok && elected) ptx::umma_commit(tfull_bar(buf));   // accumulator complete
    }
  } else {
    // ================================ A gather producers ================================
    if (PLAIN) grid_dependency_sync();
    const int gt = threadIdx.x - GATHER_WARP * 32;   // 0..127
    if (PLAIN && gt == 0 && *global_abort) *abort_flag = 1;   // set by the kernel before
    const int chunk = gt & 7;             // 16-byte chunk of the 128-byte K row
    const int rbase = gt >> 3;            // rows rbase + 16 j
    uint32_t it = 0;
    for (int w = blockIdx.x; w < total && !*abort_flag; w += gridDim.x) {
      const Tile t = tile_of(w);
      constexpr int ELEM = FP8 ? 1 : 2;   // bytes per element of the source rows
      const uint8_t* src[ROWS / 16];
      const uint8_t* base = static_cast<const uint8_t*>(p.a_src);
      uint32_t live = 0;
      const bool swap = swapped(t);
      const int pieces = (t.rows + 15) / 16;
#pragma unroll
      for (int j = 0; j < ROWS / 16; ++j) {
        const int lr = rbase + 16 * j;
        src[j] = base;
        if (lr < t.rows) {
          int idx = t.row0 + lr;   // PLAIN: the rows of h in place
          if (!PLAIN) {
            idx = __ldg(p.gather_idx + idx);
            if (p.gather_div > 1) idx /= p.gather_div;
            if (idx < 0 || idx >= p.a_rows) {   // a table entry that is no row of the source: zero-filled
              report_error(p.status, DEV_INDEX_OUT_OF_RANGE, KID_GEMM1, t.row0 + lr, idx);
              continue;
            }
          }
          src[j] = base + (size_t)idx * p.a_ld * ELEM;
          live |= 1u << j;
        }
      }
      bool ok = true;
      for (int kb = 0; kb < KB; ++kb, ++it) {
        const int s = it % NSTAGE;
        if (!ptx::mbar_wait<false, FEED_HINT>(empty_bar(s), ((it / NSTAGE) & 1) ^ 1, abort_flag, global_abort)) {
          timeout(5); ok = false; break;
        }
        const uint32_t sa = smem_base + s * STAGE_BYTES;
        const int col = kb * 128 + chunk * 16;   // byte offset inside the source row
        const bool kin = col < p.K * ELEM;
        auto copy = [&](int j) {
          const int lr = rbase + 16 * j;
          const uint32_t dst = sa + lr * 128 + ((chunk ^ (lr & 7)) << 4);
          const bool on = kin && ((live >> j) & 1u);
          ptx::cp_async_16(dst, on ? (const void*)(src[j] + col) : (const void*)base, on ? 16u : 0u);
        };
        if (!swap) {   // (one loop with a bound for both: a quarter less for full tiles, 32768 tokens 23100 -> 29000 us)
#pragma unroll
          for (int j = 0; j < ROWS / 16; ++j) copy(j);
        } else {
#pragma unroll
          for (int j = 0; j < SWAP_ROWS / 16 && j < ROWS / 16; ++j)   // (ROWS = 64: not reached)
            if (j < pieces) copy(j);
        }
        // one arrival on the stage's full barrier once the copies above have landed; the thread
        // itself goes straight on to the next stage
        ptx::cp_async_arrive_noinc(full_bar(s));
      }
      if (!ok) break;
    }
    ptx::cp_async_wait_all();   // nothing may still be in flight towards shared memory at exit
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // abort path only: give bulk copies still in flight time to land before the CTA retires
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  __syncthreads();
  if (warp == MMA_WARP) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem_base, 512);
  }
}

}  // namespace

namespace {
template <bool FP8, bool PLAIN, bool NARROW, bool FEW, bool EIGHT>
cudaError_t launch_form(const GemmParams& p, const CUtensorMap& m_a, const CUtensorMap& m_b, bool overlap, cudaStream_t st) {
  // per device; several host threads may get here at once: setting the attribute twice is harmless
  static std::atomic<bool> attr_set[MAX_DEVICES];
  const int dev = current_device();
  const auto kernel = ffn_gemm1_kernel<FP8, PLAIN, NARROW, FEW, EIGHT>;
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  ProfileScope prof(PLAIN ? KID_GEMM2 : KID_GEMM1, st);
  return launch_kernel(overlap, 0, kernel, sm_count(), threads(EIGHT), SMEM_BYTES, st, m_a, m_b, p);
}

template <bool FP8, bool PLAIN>
cudaError_t launch_width(const GemmParams& p, const CUtensorMap& m_a, const CUtensorMap& m_b, bool narrow, bool few, bool overlap,
                         cudaStream_t st) {
  // Eight epilogue warps for full-width tiles with a K walk of up to 24 blocks, and for narrow tiles of 128 rows whatever their K: such layers
  // have one round of tiles or two, so the epilogue is not hidden.  Layers, us, four / eight in the full-width tiles, K walk of GEMM-1 in
  // brackets: 10181 tokens top-1 of 8 x 656 x 4512 in 8 bits (6) 236 / 230, 529 top-4 of 16 x 608 x 1392 (10; GEMM-2 22) 50.8 / 49.7, 4000 top-4 of
  // 32 x 1504 x 2048 (24) 377.7 / 378.5, of 2048 x 2048 (32) 461.5 / 463.4, 16384 top-8 of 128 x 4096 x 1536 in 8 bits (32) 3099 / 3106, 32768 top-8 of
  // 256 x 7168 x 2048 (112) 21320 / 21440; narrow tiles, by the K of GEMM-1 and GEMM-2: 256 top-2 of 8 (512, 1024) 28.1 / 27.2, 36 top-2 of 8
  // (4160, 1008) 64.9 / 64.2, 200 (7168, 2048) 85.1 / 84.9, 100 (6144, 4096) 79.2 / 79.1, 90 (3072, 8192) 73.9 / 73.7, 65 (4096, 14336) 117.1 / 118.2, in
  // 8 bits 90.1 / 91.7; but of 64 rows (1 token, 8 x 4096 x 14336) 143 / 145.
  if (!narrow && p.K * (FP8 ? 1 : 2) > 24 * 128) return launch_form<FP8, PLAIN, false, false, false>(p, m_a, m_b, overlap, st);
  if (!narrow) return launch_form<FP8, PLAIN, false, false, true>(p, m_a, m_b, overlap, st);
  return few ? launch_form<FP8, PLAIN, true, true, false>(p, m_a, m_b, overlap, st) : launch_form<FP8, PLAIN, true, false, true>(p, m_a, m_b, overlap, st);
}
}  // namespace

// narrow: 64 output columns per tile instead of 128 (GEMM-1) or 256 (GEMM-2); p.n_tiles is set here.  The FP8 weight maps then
// have boxes of 64 columns (make_weight_map_fp8).  few: no expert has more than 64 rows (used by narrow tiles only).
//
// rows: pairs of the layer, the unused slots of a sparse table among them (how many are used is known on the device only).  A long GEMM
// starts when the kernel before it has drained, so that its thread blocks are placed on an empty GPU, in order, and not one by one as SMs
// become free.  Blocks that share a weight tile then probably sit closer together (what the times show; where a block sits was not looked
// at), and less of the board's power goes into moving operands.  Layers, overlapped / drained, us:
// 32768 tokens, top-8 of 256 x 7168 x 2048 22750 / 21620; 16384 skewed 12970 / 12570; 8192 top-4 of 64 x 7168 x 4096 in 8 bits
// 3490 / 3310; 16384 top-4 of 32 x 2048 x 2048 1581 / 1563; 2048 top-4 of 32 x 4096 x 4096 (2^37 products per matrix) 1072 / 1072;
// 4096 skewed, top-8 of 32 x 2048 x 1024 (2^36) 465 / 467.  At the line both are alike, so a sparse table that is counted as longer than it
// is loses nothing there; one of 16384 rows that uses 2 of 8 slots counts 4 times its products.
cudaError_t launch_gemm1(GemmParams p, const CUtensorMap& m_w1, const CUtensorMap& m_w3, long long rows, bool fp8, bool narrow, bool few,
                         cudaStream_t st) {
  p.n_tiles = narrow ? (p.N + 63) / 64 : (p.N + 127) / 128;
  const bool overlap = (double)rows * p.K * p.N <= 137438953472.;   // 2^37
  return fp8 ? launch_width<true, false>(p, m_w1, m_w3, narrow, few, overlap, st)
             : launch_width<false, false>(p, m_w1, m_w3, narrow, few, overlap, st);
}

// GEMM-2 through the single-CTA kernel (128-row tiles): p.a_src = h (or its E4M3 copy), p.a_ld = f,
// p.tile_prefix = the 128-row tile prefix; m_w2 is the weight map.
cudaError_t launch_gemm2_single(GemmParams p, const CUtensorMap& m_w2, bool fp8, bool narrow, bool few, cudaStream_t st) {
  p.n_tiles = narrow ? (p.N + 63) / 64 : (p.N + 255) / 256;
  return fp8 ? launch_width<true, true>(p, m_w2, m_w2, narrow, few, true, st)
             : launch_width<false, true>(p, m_w2, m_w2, narrow, few, true, st);
}

}  // namespace ffn
}  // namespace tcmoe
