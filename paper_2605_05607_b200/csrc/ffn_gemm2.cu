// GEMM-2 of the expert FFN with the gate weight in the epilogue (paper Sec. II-A "GEMM-2";
// Sec. III-C: expert i scales its output by w_i in GEMM-2's epilogue so that Combine can be an
// un-weighted reduction):
//     o[r, n] = w_r * (h_r . W2[e][:, n])
//
// The same kernel, with GLU = true, is the CTA-pair form of GEMM-1 (Sec. II-A "GEMM-1") on rows that Dispatch
// has already placed in expert-sorted order (the per-expert layout tensors of Sec. III-D):
//     h[r, n] = silu(a_r . W1[e][:, n]) * (a_r . W3[e][:, n])
// Each CTA of the pair then holds 64 columns of W1 and the same 64 of W3, so the pair's 256 accumulator columns are
// [a.W1 | a.W3 | a.W1 | a.W3], 64 each, for every row and the epilogue applies SwiGLU to columns c and c + 64.
//
// Both operands come by TMA (h rows are contiguous in expert-sorted order).  CTAs work in pairs
// (cluster of 2, tcgen05 cta_group::2): each CTA holds 128 rows of h and one half of the
// 256-column W2 tile; one UMMA of M = 256 spans the pair, so every weight byte is fetched and read
// from shared memory once per 256 rows.  Rank 0 of the pair (the leader) issues every UMMA.
//
// A row tile of at most 128 rows (most tiles of small experts, half of the last ones of large experts) takes UMMAs of M = 128
// instead, 64 rows in each CTA, which need half the tensor-pipe time; B is the same.  The accumulator of a CTA is then 64 rows
// in 128 TMEM columns: lanes 0-63 hold the tile's first 128 accumulator columns, lanes 64-127 the others.
// Weight-streaming layers (12004 pairs on 128 experts of 2880 x 2880, mostly below 128 rows) were bound by the padded UMMAs:
// dH 395 -> 352 us, GEMM-1 recomputed 797 -> 693, dX 790 -> 681, against 325 / 645 / 645 for reading the weights.
//
// Barrier ownership in a pair:
//   full[s]    leader's copy: the leader announces the bytes of both CTAs, both CTAs' TMA loads
//              credit it
//   empty[s]   each CTA's own copy, signalled by the leader's tcgen05.commit
//   tfull[b]   each CTA's own copy (accumulator buffer b complete), same
//   tempty[b]  leader's copy: the 8 epilogue warps of each CTA arrive when buffer b is drained
//
// Warp roles: 0-7 epilogue, 8 TMA producer, 9 UMMA issuer (leader only) and TMEM owner.  Eight epilogue warps (two per row
// quarter, half of the columns each): with four, a tile's epilogue took 4500-6400 cycles and bound every short K walk
// (weight gradients of experts with a hundred rows; FP8 with K = 1536, whose main loop is 6100 cycles).
// Accumulators are double-buffered in TMEM; every wait is bounded; neither CTA retires before its
// peer has stopped touching its shared memory and TMEM (cluster barrier at the end).
#include "ffn_common.cuh"

#include <atomic>

namespace tcmoe {
namespace ffn {
namespace {

constexpr int NSTAGE = 6;
constexpr int A_BYTES = BM * BK * 2;            // 16 KiB: this CTA's 128 rows
constexpr int B_BYTES = (UMMA_N / 2) * BK * 2;  // 16 KiB: this CTA's half of the B tile (two 64-column slabs)
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int NUM_BARS = 2 * NSTAGE + 4;
constexpr int BOX_BYTES = 64 * BM * 2;          // 64 columns x 128 rows of bf16: what a weight gradient stores by TMA at once
constexpr int EPI_WARPS = 8, TMA_WARP = EPI_WARPS, MMA_WARP = EPI_WARPS + 1;
constexpr int STAGE_OUT_WARP = 32 * 64;           // epilogue transpose buffer of one warp: 32 rows x 32 columns, swizzled
constexpr int TABLE_BYTES = (2 * (MAX_E + 1) * 4 + 15) & ~15;
constexpr int COLSCALE_WARP = UMMA_N / 2 * 4;      // FP8: the scales of the 128 output columns that a warp owns
constexpr int SMEM_BYTES =
    1024 + NSTAGE * STAGE_BYTES + NUM_BARS * 8 + 64 + TABLE_BYTES + EPI_WARPS * (STAGE_OUT_WARP + COLSCALE_WARP);
constexpr int THREADS = (EPI_WARPS + 2) * 32;
constexpr uint32_t IDESC = idesc_bf16(2 * BM);
constexpr uint32_t IDESC_F8 = idesc_e4m3(2 * BM);
constexpr uint32_t IDESC_BK = idesc_bf16(2 * BM) & ~(1u << 16);   // bf16 with a K-major B operand
constexpr uint32_t IDESC_WG = idesc_bf16(2 * BM) | (1u << 15);    // bf16 with both operands MN-major
constexpr uint32_t HINT = 4000;   // try_wait suspend-time hint (ns), see ptx::mbar_try_wait

// RED = false: rows go to o (bf16), Combine is a later pass.  RED = true: Combine happens here
// (Sec. IV: the fused pipeline reduces expert outputs as GEMM-2 produces them): each weighted row is
// added into the fp32 accumulator row of its token with vector reductions; o is never written.
// FP8 = true: h rows and weights are E4M3 codes, a stage holds 128 elements of K (the same 128 bytes
// per row), W2 comes K-major from [E, N, K] as one 128-row box per CTA, and the epilogue applies
// a_scale[row] * b_scale[e, n] together with the gate weight.
// MODE selects the epilogue and the operand walk:
//   PAIR_PLAIN    o = row weight x acc (GEMM-2; also dH = dO . W2^T of the backward pass): map_b0 = map_b1 = the weight,
//                 CTA `rank` takes columns n0 + 128 * rank
//   PAIR_GLU      GEMM-1 with the SwiGLU epilogue (see the head of this file): map_b0 = W1, map_b1 = W3, 128 output
//                 columns per tile
//   PAIR_GLU_BWD  the same GEMM recomputed in the backward pass: from a1 = a.W1, a3 = a.W3 and the incoming dh tile the
//                 epilogue writes h, da1 = dh * a3 * silu'(a1) and da3 = dh * silu(a1), and per 64 columns the row sums of h * dh
//   PAIR_WGRAD    dW[e] = A_e^T . B_e over the rows of expert e in the padded row space (segments start at poff[e], a multiple of 64, pad
//                 rows zero, so no block of 64 rows mixes experts and an expert without rows gets zeros): a task is a
//                 256 x 256 tile of one expert's gradient (p.K = its row count M, p.N its columns), the K walk runs over
//                 the expert's rows in blocks of 64, both operands are MN-major boxes of 64 columns x 64 rows; CTA `rank`
//                 holds rows m0 + 128 * rank of the tile and columns n0 + 128 * rank of B
//                 OUT > 0: the tile goes through shared memory, in the last OUT stages of the ring, and leaves by TMA (map_b1: dW), instead
//                 of warp by warp.
//   PAIR_KSPLIT   acc = A0 . B0 + A1 . B1 (dX = dA1 . W1^T + dA3 . W3^T): the first p.k_split k-blocks come from
//                 (rows.a0, map_b0), the rest from (rows.a1, map_b1); plain epilogue
// BKMAJ: the bf16 weight operand is read K-major (one box of 128 columns x 64 K per CTA and stage), which is how
// W^T looks when W is stored [K, N] with N contiguous: the backward GEMMs read the forward weights in place.
enum { PAIR_PLAIN = 0, PAIR_GLU = 1, PAIR_GLU_BWD = 2, PAIR_KSPLIT = 3, PAIR_WGRAD = 4 };

// Maps of the row operand(s): boxes of 32, 64, 96 and 128 rows ([3] alone for PAIR_WGRAD, whose boxes are 64 columns x 64 rows).
// A CTA loads the rows its tile has, rounded up to 32, in one box; what the stage held before stays behind them and only
// reaches accumulator rows that are not stored.  Training step of the Small layer 2003 -> 1967 us; no change where weights or
// the padded UMMAs themselves are the bound.
struct RowMaps { CUtensorMap a0[4], a1[4]; };

template <bool RED, bool FP8, int MODE, bool BKMAJ, int OUT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
ffn_gemm2_kernel(const __grid_constant__ CUtensorMap map_b0, const __grid_constant__ CUtensorMap map_b1,
                 const __grid_constant__ RowMaps rows, const GemmParams p) {
  constexpr bool GLU = MODE == PAIR_GLU || MODE == PAIR_GLU_BWD;
  constexpr bool KMAJ = FP8 || BKMAJ;   // the weight operand is K-major in shared memory
  constexpr bool TILE_OUT = OUT > 0;
  constexpr int NST = NSTAGE - OUT;
  static_assert(!TILE_OUT || MODE == PAIR_WGRAD, "whole tiles leave by TMA in the weight gradients only");
  static_assert(2 * BOX_BYTES == STAGE_BYTES && OUT <= 2, "four boxes are the CTA's part of a tile");
  static_assert(!(MODE != PAIR_PLAIN && (RED || FP8)), "only the plain form has the reducing / FP8 variants");
  constexpr int BN_OUT = GLU ? 128 : 256;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + NSTAGE * STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + NUM_BARS);
  int* abort_s = reinterpret_cast<int*>(tmem_slot + 1);
  int* tp_s = reinterpret_cast<int*>(tmem_slot + 16);
  int* eoff_s = tp_s + (MAX_E + 1);
  const uint32_t stage_base = ptx::smem_u32(tp_s) + TABLE_BYTES;   // 16-byte aligned
  float* colscale_base = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(tp_s) + TABLE_BYTES + EPI_WARPS * STAGE_OUT_WARP);

  const uint32_t smem_base = ptx::smem_u32(smem);
  const uint32_t bar_base = ptx::smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (NSTAGE + s); };
  auto tfull_bar = [&](int b) { return bar_base + 8u * (2 * NSTAGE + b); };
  auto tempty_bar = [&](int b) { return bar_base + 8u * (2 * NSTAGE + 2 + b); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)ptx::cluster_ctarank();
  const int cluster_id = blockIdx.x >> 1, num_clusters = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      ptx::mbar_init(full_bar(s), 1);       // leader TMA thread (expect_tx for both CTAs)
      ptx::mbar_init(empty_bar(s), 1);      // tcgen05.commit
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(tfull_bar(b), 1);      // tcgen05.commit
      ptx::mbar_init(tempty_bar(b), 2 * EPI_WARPS);   // one lane per epilogue warp, both CTAs
    }
    ptx::fence_mbar_init();
  }
  if (warp == TMA_WARP && lane == 0) {
    ptx::prefetch_tensormap(&map_b0);
    ptx::prefetch_tensormap(&map_b1);
    ptx::prefetch_tensormap(&rows.a0[3]);
    if (MODE == PAIR_KSPLIT) ptx::prefetch_tensormap(&rows.a1[3]);
  }
  if (warp == MMA_WARP) {
    ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), 512);
    ptx::tmem_relinquish_pair();
  }
  grid_dependency_sync();   // nothing above touches global data
  for (int i = threadIdx.x; i <= p.E; i += blockDim.x) {
    tp_s[i] = p.tile_prefix[i];
    eoff_s[i] = p.expert_offsets[i];
  }
  if (threadIdx.x == 0) *abort_s = p.status[ST_ABORT];
  ptx::tc_fence_before();
  __syncthreads();
  ptx::cluster_sync();   // the peer's barriers are initialised before anything signals them
  ptx::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  constexpr bool WGRAD = MODE == PAIR_WGRAD;
  const int wg_mt = (p.K + 2 * BM - 1) / (2 * BM), wg_per_expert = wg_mt * p.n_tiles;   // weight-gradient tiles per expert
  const int total = WGRAD ? p.E * wg_per_expert : tp_s[p.E] * p.n_tiles;
  // 128-row tiles where they are most of the tiles, or where a pair has enough tiles to even out the two lengths.  With a handful
  // of mixed tiles the longest chain is as long as before, and pairs that read the same weights no longer do so at the same time:
  // GEMM-2 of 4096 x 14336 experts with 1024 skewed rows (8 tiles per pair) 705 -> 724 us, its GEMM-1 (54 per pair) 1443 -> 1397.
  // Layer of both GEMMs on pairs, 128-row tiles on / off, us, even routing, by (rows, tiles per pair of GEMM-1 and GEMM-2): 4096 x 14336
  // experts (100, 12 and 2) 505 / 584, (300, 24 and 3) 1122 / 1095, (600, 36 and 5) 1572 / 1694; 2880 x 2880 (300, 20 and 10) 670 / 647,
  // (600, 30 and 16) 984 / 1034; 4096 x 4096 (260, 7 and 3) 281 / 288, (600, 10 and 5) 479 / 509.  So with even routing fewer tiles than
  // twelve gain as well, and up to 3 % are lost where the tiles left are just over 128 rows; the line follows the skewed layer.
  const bool halves = total >= 12 * num_clusters || eoff_s[p.E] < 160 * tp_s[p.E];
  constexpr int BK_ELEMS = FP8 ? 2 * BK : BK;   // K elements per stage: 128 bytes per row either way
  const int KB = MODE == PAIR_KSPLIT ? 2 * p.k_split : (p.K + BK_ELEMS - 1) / BK_ELEMS;
  volatile int* abort_flag = abort_s;
  const volatile int* global_abort = p.status + ST_ABORT;

  auto timeout = [&](int detail) {
    report_error(p.status, DEV_TIMEOUT, GLU ? KID_GEMM1 : KID_GEMM2, detail, blockIdx.x);
    p.status[ST_ABORT] = 1;
    *abort_flag = 1;
  };
  auto tile_of = [&](int w) {   // .half: a tile of at most 128 rows, 64 in each CTA
    if (WGRAD) {   // (expert, m-tile of 256, n-tile of 256), m-tile fastest: neighbours share the B rows in L2
      Tile t;
      t.e = w / wg_per_expert;
      const int rem = w - t.e * wg_per_expert;
      const int m0 = (rem % wg_mt) * 2 * BM + rank * BM;
      t.n0 = (rem / wg_mt) * BN_OUT;
      t.row0 = eoff_s[t.e];                                  // first (padded) row of the expert: start of the K walk
      t.kb = (eoff_s[t.e + 1] - t.row0) / BK;
      t.rows = min(BM, p.K - m0);                            // rows of dW[e] this CTA owns (<= 0: none)
      t.left = 0;
      t.half = false;
      t.out_row0 = t.e * p.K + m0;
      return t;
    }
    Tile t = decode_tile(w, tp_s, eoff_s, p.E, p.n_tiles, BN_OUT, 2 * BM, rank);
    t.half = halves && t.left <= BM;
    if (t.half) {
      t.row0 -= rank * (BM / 2);
      t.rows = min(BM / 2, t.left - rank * (BM / 2));
      t.out_row0 = t.row0;
    }
    return t;
  };

  if (warp < EPI_WARPS) {
    // ================================ epilogue (both CTAs) ================================
    const int quarter = warp & 3, half = warp >> 2;   // TMEM lanes and half of their columns this warp owns
    constexpr int COLS = BN_OUT / 2;                  // output columns of a warp (tiles of at most 128 rows: half of them)
    // A thread owns one accumulator row, but 32 threads storing 16 bytes each to 32 different rows cost 32 memory
    // transactions per instruction.  The warp transposes 32 columns at a time through shared memory (64-byte rows, pieces
    // swizzled by row pair: conflict-free both ways) and stores 64-byte row segments, 8 rows per instruction.
    const uint32_t stage = stage_base + (uint32_t)(warp * STAGE_OUT_WARP);
    const int srow = lane >> 2, piece = lane & 3;
    auto put = [&](int v, uint32_t q0, uint32_t q1, uint32_t q2, uint32_t q3) {   // columns 8 v .. + 7 of this thread's row
      ptx::st_shared_v4(stage + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4), q0, q1, q2, q3);
    };
    int tl = 0;
    // TILE_OUT: all eight warps (OUT = 2) or the four of a column half meet at barriers in every tile.  Whether a warp's wait ends with the tile
    // or with an abort is a race between them, so none leaves early: one that gave up walks the rest of the tiles without waiting (what they
    // hold is undefined then, as after any abort).  Left by a vote of the warps instead, a backward pass of 7 tokens on 128 experts of 2880 x 2880
    // took 1690 us, 1654 so.
    constexpr int MEET = EPI_WARPS * 32 / (OUT == 1 ? 2 : 1);
    const int meet_id = 1 + threadIdx.x / MEET;
    const bool leader = threadIdx.x % MEET == 0;
    auto free_boxes = [&] {   // the stores before have read theirs
      if (leader) ptx::bulk_wait_read();
      ptx::named_barrier(meet_id, MEET);
    };
    bool go = !TILE_OUT || __all_sync(0xFFFFFFFFu, !*abort_flag);   // no wait has given up (the same in all lanes)
    for (int w = cluster_id; w < total && (TILE_OUT || !*abort_flag); w += num_clusters, ++tl) {
      const Tile t = tile_of(w);
      const int buf = tl & 1;
      // 128-row halves: rows 32 quarter + lane, columns `half`.  64-row halves: rows 32 (quarter & 1) + lane, columns quarter >> 1,
      // which the two warps of a quarter share (the backward SwiGLU leaves them to one, for the sums over 64 columns).
      const int row_w = (t.half ? quarter & 1 : quarter) * 32, part = t.half ? quarter >> 1 : half;
      const int sub = t.half && MODE != PAIR_GLU_BWD ? half * (COLS / 2) : 0;
      const int chunks = t.half ? COLS / 64 : COLS / 32;
      const bool idle = MODE == PAIR_GLU_BWD && t.half && half != 0;
      const int col0 = t.n0 + part * COLS + sub;      // first output column of this warp
      uint4 dh[2][4];
      if (MODE == PAIR_GLU_BWD) {   // the incoming gradient of h, 64 columns of the warp's rows, while the main loop runs
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = row_w + i * 8 + srow, col = col0 + c * 32 + piece * 8;
            dh[c][i] = r < t.rows && col < p.N && !idle
                           ? __ldg(reinterpret_cast<const uint4*>(p.dh + (size_t)(t.row0 + r) * (size_t)p.out_ld + col))
                           : make_uint4(0u, 0u, 0u, 0u);
          }
      }
      if (go && !ptx::mbar_wait_warp<false, HINT>(tfull_bar(buf), (tl >> 1) & 1, abort_flag, global_abort)) { timeout(1); go = false; }
      if (!TILE_OUT && !go) break;
      ptx::tc_fence_after();
      const int lrow = row_w + lane;
      const bool valid = lrow < t.rows;
      const size_t grow = (size_t)(valid ? t.row0 + lrow : 0);
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * UMMA_N + (t.half ? 0 : half * 128) + sub);
      auto send = [&](__nv_bfloat16* out, int c) {    // 32 staged columns -> rows of out
        __syncwarp();
        const int col = col0 + c * 32 + piece * 8;
        if (col < p.N) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = i * 8 + srow;               // row of this warp's 32
            if (row_w + r < t.rows) {
              const uint4 q = ptx::ld_shared_v4(stage + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4));
              *reinterpret_cast<uint4*>(out + (size_t)(t.out_row0 + row_w + r) * (size_t)p.out_ld + col) = q;
            }
          }
        }
        __syncwarp();
      };
      float* yrow = nullptr;
      float wr = 1.f;
      if (valid && !GLU && !WGRAD && (RED || p.topk_w != nullptr)) {
        const int pair = __ldg(p.row_pair + grow);
        if (p.topk_w != nullptr) wr = __ldg(p.topk_w + pair);
        if (RED) yrow = p.y_acc + (size_t)(pair / p.y_div) * (size_t)p.N + col0;
      }
      if (FP8 && valid) wr *= __ldg(p.a_scale + grow);   // row scale of h joins the gate weight
      // FP8: the tile's output-column scales, one copy per warp (0 beyond N), staged while the
      // main loop of this tile may still be running
      float* sb_col = colscale_base + warp * (UMMA_N / 2);
      if (FP8) {
        const float* g = p.b_scale + (size_t)t.e * p.N + col0;
#pragma unroll
        for (int i = 0; i < COLS / 32; ++i) {
          const int n = lane + 32 * i;
          sb_col[n] = (col0 + n < p.N) ? __ldg(g + n) : 0.f;
        }
        __syncwarp();
      }
      if (MODE == PAIR_GLU_BWD && idle) {
      } else if (MODE == PAIR_GLU_BWD) {
        // backward of SwiGLU on the recomputed pre-activations, 32 columns at a time: dh comes to the owner of its row through
        // the staging buffer, h / dA1 / dA3 leave through it
        float dot = 0.f;   // h . dh over this warp's columns, of the rounded values (the gate's gradient needs it)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = i * 8 + srow;
            ptx::st_shared_v4(stage + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4), dh[c][i].x, dh[c][i].y, dh[c][i].z, dh[c][i].w);
          }
          uint32_t a1[32], a3[32];
          ptx::tmem_ld32(taddr + c * 32, a1);
          ptx::tmem_ld32(taddr + 64 + c * 32, a3);
          ptx::tmem_ld_wait_on(a1, a3);
          __syncwarp();
          uint32_t q1[16], q3[16];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            const uint4 dq = ptx::ld_shared_v4(stage + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4));
            const __nv_bfloat162* dp = reinterpret_cast<const __nv_bfloat162*>(&dq);
            uint32_t qh[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int j = v * 8 + 2 * i;
              const float2 dhv = __bfloat1622float2(dp[i]);
              float hh[2], d1[2], d3[2];
#pragma unroll
              for (int u = 0; u < 2; ++u) {
                const float x1 = __uint_as_float(a1[j + u]), x3 = __uint_as_float(a3[j + u]);
                const float dv = u ? dhv.y : dhv.x;
                const float sg = __fdividef(1.f, 1.f + __expf(-x1));
                const float sl = x1 * sg;
                hh[u] = sl * x3;
                d3[u] = dv * sl;
                d1[u] = dv * x3 * (sg * (1.f + x1 * (1.f - sg)));
              }
              qh[i] = pack2(hh[0], hh[1]);
              q1[v * 4 + i] = pack2(d1[0], d1[1]);
              q3[v * 4 + i] = pack2(d3[0], d3[1]);
              const float2 hr = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&qh[i]));
              dot = fmaf(hr.x, dhv.x, fmaf(hr.y, dhv.y, dot));
            }
            put(v, qh[0], qh[1], qh[2], qh[3]);   // over the piece just read: the same row and place
          }
          send(p.out, c);
#pragma unroll
          for (int v = 0; v < 4; ++v) put(v, q1[v * 4], q1[v * 4 + 1], q1[v * 4 + 2], q1[v * 4 + 3]);
          send(p.out2, c);
#pragma unroll
          for (int v = 0; v < 4; ++v) put(v, q3[v * 4], q3[v * 4 + 1], q3[v * 4 + 2], q3[v * 4 + 3]);
          send(p.out3, c);
        }
        if (valid) p.row_dots[(size_t)(t.n0 / BN_OUT * 2 + part) * p.dots_ld + grow] = dot;
      } else if (GLU) {
        // SwiGLU of 64 columns of W1 and the 64 of W3 behind them
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          uint32_t a1[32], a3[32];
          ptx::tmem_ld32(taddr + c * 32, a1);
          ptx::tmem_ld32(taddr + 64 + c * 32, a3);
          ptx::tmem_ld_wait_on(a1, a3);
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            uint32_t q[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int j = v * 8 + 2 * i;
              q[i] = pack2(silu_mul(__uint_as_float(a1[j]), __uint_as_float(a3[j])),
                           silu_mul(__uint_as_float(a1[j + 1]), __uint_as_float(a3[j + 1])));
            }
            put(v, q[0], q[1], q[2], q[3]);
          }
          send(p.out, c);
        }
      } else if (RED) {
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          uint32_t acc[32];
          ptx::tmem_ld32(taddr + c * 32, acc);
          ptx::tmem_ld_wait_on(acc);
          if (FP8) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int n = c * 32 + j;
              acc[j] = __float_as_uint(__uint_as_float(acc[j]) * sb_col[n]);
            }
          }
          if (valid) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              if (col0 + c * 32 + v * 8 < p.N) {
                float* dst = yrow + c * 32 + v * 8;
                ptx::red_add_v4(dst, wr * __uint_as_float(acc[v * 8]), wr * __uint_as_float(acc[v * 8 + 1]),
                                wr * __uint_as_float(acc[v * 8 + 2]), wr * __uint_as_float(acc[v * 8 + 3]));
                ptx::red_add_v4(dst + 4, wr * __uint_as_float(acc[v * 8 + 4]), wr * __uint_as_float(acc[v * 8 + 5]),
                                wr * __uint_as_float(acc[v * 8 + 6]), wr * __uint_as_float(acc[v * 8 + 7]));
              }
            }
          }
        }
      } else if (OUT == 1) {
        // As below, in boxes of 64 columns of which a column half has one place: its warps fill a box when the store of the one before has read
        // it.
        const uint32_t box = smem_base + NST * STAGE_BYTES + half * BOX_BYTES, dst = box + (quarter * 32 + lane) * 128;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c == 0) free_boxes();
          uint32_t lo[32], hi[32];
          ptx::tmem_ld32(taddr + c * 64, lo);
          ptx::tmem_ld32(taddr + c * 64 + 32, hi);
          ptx::tmem_ld_wait_on(lo, hi);
          if (t.kb == 0) {   // an expert without rows: the accumulator was never written
#pragma unroll
            for (int j = 0; j < 32; ++j) lo[j] = hi[j] = 0u;
          }
          uint32_t q[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            q[j] = pack2(__uint_as_float(lo[2 * j]), __uint_as_float(lo[2 * j + 1]));
            q[16 + j] = pack2(__uint_as_float(hi[2 * j]), __uint_as_float(hi[2 * j + 1]));
          }
          if (c > 0) free_boxes();
#pragma unroll
          for (int v = 0; v < 8; ++v) ptx::st_shared_v4(dst + ((v ^ (lane & 7)) << 4), q[v * 4], q[v * 4 + 1], q[v * 4 + 2], q[v * 4 + 3]);
          ptx::fence_proxy_async_smem();
          ptx::named_barrier(meet_id, MEET);
          const int col = t.n0 + half * 128 + c * 64;
          if (leader && go && t.rows > 0 && col < p.N) {
            ptx::tma_store_3d(&map_b1, box, col, t.out_row0 - t.e * p.K, t.e);
            ptx::bulk_commit();
          }
        }
      } else if (OUT == 2) {
        // The CTA's 128 x 256 part of the tile through shared memory, four boxes of 64 columns in the layout of a 128-byte swizzle, and
        // out by TMA, which clips at the edges of dW[e].
        const uint32_t dst = smem_base + NST * STAGE_BYTES + (quarter * 32 + lane) * 128;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c == 0) free_boxes();
          uint32_t lo[32], hi[32];
          ptx::tmem_ld32(taddr + c * 64, lo);
          ptx::tmem_ld32(taddr + c * 64 + 32, hi);
          ptx::tmem_ld_wait_on(lo, hi);
          if (t.kb == 0) {   // an expert without rows: the accumulator was never written
#pragma unroll
            for (int j = 0; j < 32; ++j) lo[j] = hi[j] = 0u;
          }
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            const uint32_t* q = v < 4 ? lo + v * 8 : hi + (v - 4) * 8;
            ptx::st_shared_v4(dst + (half * 2 + c) * BOX_BYTES + ((v ^ (lane & 7)) << 4), pack2(__uint_as_float(q[0]), __uint_as_float(q[1])),
                              pack2(__uint_as_float(q[2]), __uint_as_float(q[3])), pack2(__uint_as_float(q[4]), __uint_as_float(q[5])),
                              pack2(__uint_as_float(q[6]), __uint_as_float(q[7])));
          }
        }
        ptx::fence_proxy_async_smem();
        ptx::named_barrier(meet_id, MEET);
        if (leader && go && t.rows > 0) {
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (t.n0 + c * 64 < p.N)
              ptx::tma_store_3d(&map_b1, smem_base + NST * STAGE_BYTES + c * BOX_BYTES, t.n0 + c * 64, t.out_row0 - t.e * p.K, t.e);
          ptx::bulk_commit();
        }
      } else {
#pragma unroll 1
        for (int c = 0; c < chunks; ++c) {
          uint32_t acc[32];
          ptx::tmem_ld32(taddr + c * 32, acc);
          ptx::tmem_ld_wait_on(acc);
          if (WGRAD && t.kb == 0) {   // an expert without rows: the accumulator was never written
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = 0u;
          }
          if (FP8) {   // per-output-column weight scales
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = __float_as_uint(__uint_as_float(acc[j]) * sb_col[c * 32 + j]);
          }
#pragma unroll
          for (int v = 0; v < 4; ++v)
            put(v, pack2(wr * __uint_as_float(acc[v * 8]), wr * __uint_as_float(acc[v * 8 + 1])),
                pack2(wr * __uint_as_float(acc[v * 8 + 2]), wr * __uint_as_float(acc[v * 8 + 3])),
                pack2(wr * __uint_as_float(acc[v * 8 + 4]), wr * __uint_as_float(acc[v * 8 + 5])),
                pack2(wr * __uint_as_float(acc[v * 8 + 6]), wr * __uint_as_float(acc[v * 8 + 7])));
          send(p.out, c);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      // "accumulator buffer drained": the tcgen05.ld results are in registers (wait::ld above), so a
      // relaxed arrival is enough; a releasing one would first wait for this warp's row stores to
      // become visible cluster-wide, which on short-K tiles stalls the next-but-one main loop
      // (K = 512: 860 -> 1049 TFLOP/s with the relaxed form)
      if (lane == 0) ptx::mbar_arrive_cluster_relaxed(ptx::mapa(tempty_bar(buf), 0));
    }
    if (TILE_OUT && leader) ptx::bulk_wait();
  } else if (warp == TMA_WARP) {
    // ================================ TMA producer (both CTAs) ================================
    if (lane == 0) {
      uint32_t it = 0;
      for (int w = cluster_id; w < total && !*abort_flag; w += num_clusters) {
        const Tile t = tile_of(w);
        bool ok = true;
        const int KBt = WGRAD ? t.kb : KB;
        // 32-row blocks of the tile in this CTA and in both (the expert's rows from the pair's first row on: t.left)
        const int cta_rows = t.half ? BM / 2 : BM;
        auto blocks32 = [&](int left) { return min(max(left + 31, 0), cta_rows) >> 5; };
        const int mine = WGRAD ? 4 : blocks32(t.left - rank * cta_rows);
        const uint32_t bytes = 2 * B_BYTES + (WGRAD ? 8 : blocks32(t.left) + blocks32(t.left - cta_rows)) * (A_BYTES / 4);
        for (int kb = 0; kb < KBt; ++kb, ++it) {
          const int s = it % NST;
          if (!ptx::mbar_wait<false, HINT>(empty_bar(s), ((it / NST) & 1) ^ 1, abort_flag, global_abort)) {
            timeout(2); ok = false; break;
          }
          const uint32_t sa = smem_base + s * STAGE_BYTES, sb = sa + A_BYTES;
          const uint32_t lead_full = ptx::mapa(full_bar(s), 0);
          // the leader announces the bytes of both CTAs; the peer's copies only complete them
          if (rank == 0) ptx::mbar_arrive_expect_tx(full_bar(s), bytes);
          if (WGRAD) {   // four MN-major boxes of 64 columns x 64 rows: this CTA's 128 rows of A^T and 128 columns of B
            const int r0 = t.row0 + kb * BK, ma = t.out_row0 - t.e * p.K;
            ptx::tma_load_2d_pair(sa, &rows.a0[3], lead_full, ma, r0);
            ptx::tma_load_2d_pair(sa + 8192, &rows.a0[3], lead_full, ma + 64, r0);
            ptx::tma_load_2d_pair(sb, &map_b0, lead_full, t.n0 + rank * 128, r0);
            ptx::tma_load_2d_pair(sb + 8192, &map_b0, lead_full, t.n0 + rank * 128 + 64, r0);
            continue;
          }
          const bool second = MODE == PAIR_KSPLIT && kb >= p.k_split;     // second (A, B) pair of the K walk
          const int k0 = (second ? kb - p.k_split : kb) * BK_ELEMS;
          if (mine > 0) ptx::tma_load_2d_pair(sa, (second ? rows.a1 : rows.a0) + mine - 1, lead_full, k0, t.row0);
          const CUtensorMap* map_b = second ? &map_b1 : &map_b0;
          const int nb = t.n0 + rank * (BN_OUT / 2);   // this CTA's columns of the B tile
          if (KMAJ) {   // one K-major box: this CTA's 128 output columns x 128 bytes of K
            ptx::tma_load_3d_pair(sb, map_b, lead_full, k0, nb, t.e);
          } else {     // two MN-major slabs of 64 output columns x 64 rows of K, or one of W1 and the same of W3
            ptx::tma_load_3d_pair(sb, map_b, lead_full, nb, k0, t.e);
            ptx::tma_load_3d_pair(sb + 8192, GLU ? &map_b1 : map_b, lead_full, GLU ? nb : nb + 64, k0, t.e);
          }
        }
        if (!ok) break;
      }
    }
  } else if (warp == MMA_WARP) {
    // ================================ UMMA issuer (leader CTA only) ================================
    // the warp walks the loop, one elected lane issues (see ptx::elect_one)
    if (rank == 0) {
      const bool elected = ptx::elect_one();
      const uint32_t base = __shfl_sync(0xFFFFFFFFu, smem_base, 0), tmem = __shfl_sync(0xFFFFFFFFu, tmem_base, 0);
      const uint64_t mn = desc_base(BK * 128, 1024), km = desc_base(16, 1024);   // MN-major, K-major
      const uint64_t a_desc = desc_at(WGRAD ? mn : km, base), b_desc = desc_at(KMAJ ? km : mn, base + A_BYTES);
      constexpr int A_STEP = WGRAD ? 128 : 2, B_STEP = KMAJ ? 2 : 128;            // 32 bytes of K: 16 bf16 / 32 E4M3
      constexpr uint32_t ID = FP8 ? IDESC_F8 : WGRAD ? IDESC_WG : BKMAJ ? IDESC_BK : IDESC;
      constexpr uint32_t ID_HALF = (ID & ~(0x1Fu << 24)) | ((uint32_t)(BM >> 4) << 24);   // M = 128
      int s = 0, tl = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int w = cluster_id; ok && w < total && !*abort_flag; w += num_clusters, ++tl) {
        const int buf = tl & 1;
        const Tile t = tile_of(w);
        const uint32_t id = t.half ? ID_HALF : ID;
        if (!ptx::mbar_wait_cluster<HINT>(tempty_bar(buf), ((tl >> 1) & 1) ^ 1, abort_flag, global_abort)) {
          timeout(3); break;
        }
        ptx::tc_fence_after();
        const uint32_t d_tmem = tmem + (uint32_t)(buf * UMMA_N);
        const int KBt = WGRAD ? t.kb : KB;
        for (int kb = 0; kb < KBt; ++kb) {
          if (!ptx::mbar_wait_cluster<HINT>(full_bar(s), ph, abort_flag, global_abort)) {
            timeout(4); ok = false; break;
          }
          ptx::tc_fence_after();
          if (elected) {
            const uint64_t ad = a_desc + (uint64_t)(s * (STAGE_BYTES >> 4)), bd = b_desc + (uint64_t)(s * (STAGE_BYTES >> 4));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              if (FP8) ptx::umma_f8_pair(d_tmem, ad + (uint64_t)(k * A_STEP), bd + (uint64_t)(k * B_STEP), id, (kb | k) != 0);
              else ptx::umma_bf16_pair(d_tmem, ad + (uint64_t)(k * A_STEP), bd + (uint64_t)(k * B_STEP), id, (kb | k) != 0);
            }
            ptx::umma_commit_both(empty_bar(s));   // free the stage in both CTAs once these UMMAs have read it
          }
          if (++s == NST) { s = 0; ph ^= 1u; }
        }
        if (ok && elected) ptx::umma_commit_both(tfull_bar(buf));   // accumulator complete, both halves
      }
    }
  }

  ptx::tc_fence_before();
  __syncthreads();
  if (*abort_flag || *global_abort) {
    // abort path only: give bulk copies still in flight time to land before the CTAs retire
    for (int i = 0; i < 64; ++i) __nanosleep(1000);
  }
  ptx::cluster_sync();   // neither CTA leaves while its peer may still touch its shared memory / TMEM
  if (warp == MMA_WARP) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc_pair(tmem_base, 512);
  }
}

// Persistent grid: two CTAs per resident cluster, at most one CTA per SM.
int pair_grid() {
  static std::atomic<int> grid_of[MAX_DEVICES];   // 0 = not computed yet; recomputing gives the same value
  std::atomic<int>& cached = grid_of[current_device()];
  int g = cached.load(std::memory_order_relaxed);
  if (g == 0) {
    int clusters = 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sm_count() & ~1);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&clusters, ffn_gemm2_kernel<false, false, PAIR_PLAIN, false, 0>, &cfg) != cudaSuccess || clusters <= 0) {
      (void)cudaGetLastError();
      clusters = sm_count() / 2;
    }
    g = 2 * min(clusters, sm_count() / 2);
    cached.store(g, std::memory_order_relaxed);
  }
  return g;
}

}  // namespace

namespace {
cudaError_t set_pair_attributes() {
  // per device; several host threads may get here at once: setting the attribute twice is harmless
  static std::atomic<bool> attr_set[MAX_DEVICES];
  const int dev = current_device();
  if (!attr_set[dev].load(std::memory_order_acquire)) {
    const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_PLAIN, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<true, false, PAIR_PLAIN, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, true, PAIR_PLAIN, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<true, true, PAIR_PLAIN, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_GLU, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_PLAIN, true, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_GLU_BWD, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_KSPLIT, true, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 0>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 1>, attr, SMEM_BYTES);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 2>, attr, SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set[dev].store(true, std::memory_order_release);
  }
  return cudaSuccess;
}
}  // namespace

// every row operand: p.a_src [p.a_rows, K] (PAIR_KSPLIT: p.a_src2 too)
static bool make_row_maps(RowMaps* m, const GemmParams& p, bool fp8) {
  for (int i = 0; i < 4; ++i) {
    if (!make_act_map(&m->a0[i], p.a_src, p.a_rows, p.K, fp8, 32 * (i + 1))) return false;
    if (p.a_src2 != nullptr && !make_act_map(&m->a1[i], p.a_src2, p.a_rows, p.K, fp8, 32 * (i + 1))) return false;
  }
  return true;
}

cudaError_t launch_gemm2(const GemmParams& p, const CUtensorMap& m_w2, bool fp8, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  RowMaps rows{};
  if (!make_row_maps(&rows, p, fp8)) return cudaErrorInvalidValue;
  ProfileScope prof(KID_GEMM2, st);
  const bool red = p.y_acc != nullptr;
  const int g = pair_grid();
  if (fp8) {
    if (red) return launch_pdl(ffn_gemm2_kernel<true, true, PAIR_PLAIN, false, 0>, g, THREADS, SMEM_BYTES, st, m_w2, m_w2, rows, p);
    return launch_pdl(ffn_gemm2_kernel<false, true, PAIR_PLAIN, false, 0>, g, THREADS, SMEM_BYTES, st, m_w2, m_w2, rows, p);
  }
  if (red) return launch_pdl(ffn_gemm2_kernel<true, false, PAIR_PLAIN, false, 0>, g, THREADS, SMEM_BYTES, st, m_w2, m_w2, rows, p);
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_PLAIN, false, 0>, g, THREADS, SMEM_BYTES, st, m_w2, m_w2, rows, p);
}

// GEMM-1 on CTA pairs from the expert-sorted activation rows (p.a_src = xs); p.tile_prefix = the 256-row pair-tile
// prefix, p.n_tiles = ceil(N / 128), p.out = h.
cudaError_t launch_gemm1_pair(const GemmParams& p, const CUtensorMap& m_w1, const CUtensorMap& m_w3, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  RowMaps rows{};
  if (!make_row_maps(&rows, p, false)) return cudaErrorInvalidValue;
  ProfileScope prof(KID_GEMM1, st);
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_GLU, false, 0>, pair_grid(), THREADS, SMEM_BYTES, st, m_w1, m_w3, rows, p);
}

// Backward pass, all on CTA pairs (see bwd.cu for the sequence):
//   launch_bwd_dh    dh = dO . W2^T          p.a_src = dO, B = W2 read K-major (m_w2t), N = f, K = d
//   launch_bwd_glu   GEMM-1 recomputed with the backward SwiGLU epilogue: p.dh in, p.out = h, p.out2 = dA1, p.out3 = dA3
//   launch_bwd_dx    dXs = dA1 . W1^T + dA3 . W3^T   p.a_src = dA1, p.a_src2 = dA3, B = (m_w1t, m_w3t) K-major, p.k_split k-blocks each
cudaError_t launch_bwd_dh(const GemmParams& p, const CUtensorMap& m_w2t, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  RowMaps rows{};
  if (!make_row_maps(&rows, p, false)) return cudaErrorInvalidValue;
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_PLAIN, true, 0>, pair_grid(), THREADS, SMEM_BYTES, st, m_w2t, m_w2t, rows, p);
}
cudaError_t launch_bwd_glu(const GemmParams& p, const CUtensorMap& m_w1, const CUtensorMap& m_w3, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  RowMaps rows{};
  if (!make_row_maps(&rows, p, false)) return cudaErrorInvalidValue;
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_GLU_BWD, false, 0>, pair_grid(), THREADS, SMEM_BYTES, st, m_w1, m_w3, rows, p);
}
cudaError_t launch_bwd_dx(const GemmParams& p, const CUtensorMap& m_w1t, const CUtensorMap& m_w3t, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  RowMaps rows{};
  if (!make_row_maps(&rows, p, false)) return cudaErrorInvalidValue;
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_KSPLIT, true, 0>, pair_grid(), THREADS, SMEM_BYTES, st, m_w1t, m_w3t, rows, p);
}

// Weight gradient on CTA pairs: dw[e] = A_e^T . B_e, A = [rows, M], B = [rows, N] in the padded row space (maps with
// boxes of 64 columns x 64 rows; rows_total: pairs of the layer, unused slots of a sparse table among them), dw [E, M, N] bf16, fully written.
cudaError_t launch_wgrad_pair(const CUtensorMap& m_a, const CUtensorMap& m_b, const int32_t* poff, long long rows_total, void* dw, int E,
                              int M, int N, int32_t* status, cudaStream_t st) {
  cudaError_t e = set_pair_attributes();
  if (e != cudaSuccess) return e;
  GemmParams p{};
  p.out = static_cast<__nv_bfloat16*>(dw);
  p.out_ld = N;
  p.expert_offsets = poff;
  p.tile_prefix = poff;      // not used by this mode (the table load needs a valid array)
  p.E = E;
  p.K = M;                   // rows of dw[e]
  p.N = N;
  p.n_tiles = (N + 255) / 256;
  p.status = status;
  RowMaps rows{};
  rows.a0[3] = m_a;
  ProfileScope prof(KID_WGRAD, st);
  // Experts of few rows: the gradients are bound by their stores, and by what the stores take of the board's power; whole tiles leave by
  // TMA then.  A tile on its way out takes two of the ring's six stages, or one, whose boxes are filled one after the other: up to 80 rows
  // per expert the stores are all that counts, but four stages do not cover the latency of a long K walk, and with skewed routing the
  // popular experts have one at any average.  Backward pass, us, by the warps / two stages / one stage, rows per expert in brackets, even and
  // skewed routing: 128 x 2048 x 2048 (50) 1656 / 1611 / 1711, 1317 / 1283 / 1318; 128 x 2880 x 2880 (94) 4010 / 3810 / 3750, 4117 / 3977 / 3930; 128 x
  // 1904 x 480 (100) 608 / 596 / 596, 597 / 616 / 589; 128 x 1024 x 512 (190) 430 / 433 / 424, 530 / 558 / 529; 128 x 4096 x 1536 (190) 3830 / 3773 /
  // 3616, 4240 / 4384 / 4223.  From 192 rows on the tensor cores are the bound and the warps store.
  // Ragged rows (they start inside a 32-byte sector) leave by TMA at any size: in pieces of 64 bytes twice as many sectors are written in
  // two halves.  Boxes of neighbouring columns had better leave together there, so two stages are taken for longer where the gradient is large:
  // 128 x 2888 x 2872 (100) two 4510 / one 4910, 4783 / 5330; 64 x 1896 x 480 (190) 419 / 410, 551 / 530.
  const bool ragged = (N & 15) != 0;
  if (rows_total < 192ll * E || ragged) {
    CUtensorMap m_dw;
    if (!make_store_map(&m_dw, dw, E, M, N)) return cudaErrorInvalidValue;
    const bool two = rows_total < 80ll * E || (ragged && rows_total < 192ll * E && (long long)M * N >= 4000000);   // stages for the tile
    const auto kernel = two ? ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 2> : ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 1>;
    return launch_pdl(kernel, pair_grid(), THREADS, SMEM_BYTES, st, m_b, m_dw, rows, p);
  }
  return launch_pdl(ffn_gemm2_kernel<false, false, PAIR_WGRAD, false, 0>, pair_grid(), THREADS, SMEM_BYTES, st, m_b, m_b, rows, p);
}

}  // namespace ffn
}  // namespace tcmoe
