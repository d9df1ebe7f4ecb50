// Grouped bf16 GEMM for groups of 17 to about a thousand rows, of few wide shapes up to some three thousand (decode batches,
// classification heads, single images, prompts of some hundred tokens): C = epi(A W^T + bias) with the operands swapped on the tensor core.
//
// With so few rows the work is streaming W once, or too few output tiles to fill the chip.  The MMA's 128-row
// operand is a tile of W (128 output columns) and the batch is the MMA's N: one tile of up to 256 rows, several of
// them beyond that (nb rows each, a multiple of 16).  D[n, m] = sum_k W[n, k] A[m, k]: the accumulator holds C
// transposed, TMEM lane = output column, TMEM column = batch row.
//
// At small batches what bounds these kernels is how many bytes of W a CTA has in flight: at full rate HBM answers a
// request after about 5 us, so the whole device needs some 30 MB outstanding, about 200 KB per SM (measured: a CTA's
// ingest is its ring size divided by that latency, whatever the tile shape).  Activation tiles come from L2, a
// fraction of that latency away, and must not take ring space from W: the two operands have rings of their own, up to ten
// stages of 16 KB for W and two to eight short-lived stages for the activations (tiles of more than 128 rows: four
// stages of activations, the rest for W, since there the MMA time of a k-block is what has to be covered).
//
// A matrix has only N / 128 such tiles (16 to 24 for the projections of a 1B-scale decoder), too few CTAs to pull
// HBM bandwidth.  So K is cut into S ranges (fixed from rows, N and K when the model is placed) and the S CTAs of a
// thread-block cluster work one tile: each accumulates its k range in its own TMEM.  CTA r owns a share of the
// tile's batch rows: once every CTA of the cluster is past its last MMA (a cluster barrier: the slices land in the
// owners' idle operand rings), every CTA sends the matching slice of its fp32 partial into CTA r's shared memory
// (distributed-shared-memory stores, which nobody waits for), and after a second cluster barrier CTA r adds the S
// slices in rank order out of its own shared memory and runs the epilogue for its rows, a warp per row, 128 output
// columns contiguous.  No partial ever travels through global memory and the reduction order is fixed, so a
// request's bits do not depend on timing or on what else is in the launch.
//
// Pairs (PAIR; from 129 rows on, see gemm_swap2_config()).  With hundreds of rows what counts is what a CTA takes in: a tile of 128 columns and 256
// rows asks for 48 KB a k-block, as much as the MMAs of one SM can use in 512 cycles, and L2 delivers 61 bytes a cycle to an SM.
// Here a tile has 256 columns and two CTAs (cta_group::2): each loads its own 128 rows of W and half of the batch rows, the first
// one issues M = 256 MMAs for both (two per step when the tile has more than 256 rows), and each accumulates, exchanges and writes
// out its own 128 columns as above, with the CTAs of the same half in the other k ranges.  Against tiles of 256 batch rows on
// CTA pairs (the tile-pair kernel) the row tile is free: 536 rows are four of 160 and not two of 256 and a third that is nearly
// empty, and K can be split where the tiles are few.  (One barrier a stage for both operands: with one each, as in the form on one
// CTA, a k-block cost the issuer 650 cycles, now 360; 16 epilogue warps instead of eight gained nothing.)  Whole steps without
// and with it (the builds before and after, in turn): 1B decoder, a prompt of 250 tokens 1408 and 1269 us, of 450 1632 and 1570, of 520 2074
// and 1917, 512-token chunk beside 24 decode requests 2498 and 2367; 8B decoder, 300 tokens 7916 and 6236; one image through ViT-B 599 and 547.
//
// Roles per CTA (converged warps, an elected lane issues): warp 0 TMA producer of W -- it does not wait for the earlier
// kernels of the stream, weights being static, so its ring is full when they finish; the last warp TMA producer of the
// activations; warp 1 tcgen05.mma issuer; warps 2..9 read the accumulator (two warps per TMEM lane
// quarter) and run the epilogue.  Every mbarrier wait is bounded; a CTA that gives up records a code in *status and
// still meets its cluster at the barriers.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace epara {

namespace {

using namespace tc;

constexpr int SW_BM = 128;                       // W rows (output columns) per tile
constexpr int SW_W_BYTES = SW_BM * TC_BK * 2;    // 16 KB
constexpr int SW_RING_BYTES_1 = 192 * 1024;      // one CTA per SM
constexpr int SW_RING_BYTES_2 = 104 * 1024;      // two CTAs per SM: launches with more CTAs than SMs, where a second
                                                 // MMA-issuing thread per SM and no second wave pay (the LM head:
                                                 // 45 -> 31 us at 128 rows), while launches that fit one wave were a
                                                 // little faster with the deeper ring
// (the exchange of a tile's partial sums, a row of 128 columns in fp32 for each of its rows, lies over the idle ring)
static_assert(GEMM_SWAP2_TILE_ROWS * SW_BM * 4 <= SW_RING_BYTES_1 && GEMM_SWAP_TILE_ROWS * SW_BM * 4 <= SW_RING_BYTES_1, "exchange buffer");
constexpr int SW_W_STAGES_MAX = 10;
constexpr int SW_A_STAGES_MAX = 8;
constexpr int SW_EPI_WARPS = 8;
constexpr int SW_A_WARP = 2 + SW_EPI_WARPS;      // the warp after the accumulator warps loads the activations
constexpr int SW_THREADS = 32 * (SW_A_WARP + 1);
constexpr int SW_BAR_BYTES = 512;
inline size_t sw_smem(int ring_bytes) { return 1024 + (size_t)ring_bytes + SW_BAR_BYTES; }

__device__ __forceinline__ int find_group_sw(const GemmGroup* groups, int n, int item) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (groups[mid].tile_start <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Rows of the first MMA of a PAIR tile: all of up to 256, the larger half of more.
__host__ __device__ inline int swap2_first(int nb) { return nb <= 256 ? nb : (nb + 63) / 64 * 32; }

// S: CTAs per cluster = k ranges per tile.  One cluster per (group, tile of 128 output columns, tile of nb rows).
// BESIDE: runs beside the launch before it (see pdl_begin(); the residual then comes past L1.  A run-time switch cost 6 us of 1195 in
// a step of 27 requests through the 1B decoder).
// PAIR: a tile has 256 output columns and up to 384 batch rows and each of its k ranges two CTAs (see above).
template <int S, bool BESIDE, bool PAIR>
__global__ void __launch_bounds__(SW_THREADS, PAIR ? 1 : 2)
gemm_swap_kernel(const GemmGroup* __restrict__ groups, int n_groups, int* __restrict__ status, int ring_bytes) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  const uint32_t bars = base + ring_bytes;
  auto wfull_bar = [&](int s) { return bars + 8u * s; };
  auto wempty_bar = [&](int s) { return bars + 8u * (SW_W_STAGES_MAX + s); };
  auto afull_bar = [&](int s) { return bars + 8u * (2 * SW_W_STAGES_MAX + s); };
  auto aempty_bar = [&](int s) { return bars + 8u * (2 * SW_W_STAGES_MAX + SW_A_STAGES_MAX + s); };
  const uint32_t tfull_bar = bars + 8u * (2 * SW_W_STAGES_MAX + 2 * SW_A_STAGES_MAX);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + ring_bytes + 8 * (2 * SW_W_STAGES_MAX + 2 * SW_A_STAGES_MAX + 1));
  static_assert(8 * (2 * SW_W_STAGES_MAX + 2 * SW_A_STAGES_MAX + 1) + 16 <= SW_BAR_BYTES, "barrier area");
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool acc_ok = true;
  constexpr int CTAS = PAIR ? 2 * S : S;          // of a cluster
  const int crank = CTAS == 1 ? 0 : (int)cluster_ctarank();
  const int rank = PAIR ? crank >> 1 : crank;     // k range
  const int half = PAIR ? crank & 1 : 0;          // which 128 of the tile's 256 output columns, and which half of its batch rows to load
  const int item = blockIdx.x / CTAS;

  const GemmGroup* g = groups + find_group_sw(groups, n_groups, item);
  const int nb = g->bn;                           // batch rows of a tile as the MMA's N: multiple of 16, at most 256 (PAIR: of 32, 384)
  const int tiles_m = g->tiles_m;
  const int local = item - g->tile_start;
  const int n0 = (local / tiles_m) * (PAIR ? 2 * SW_BM : SW_BM) + half * SW_BM;   // first output column (W row); the row tiles of one
  const int m0 = (local % tiles_m) * nb;          // W tile are neighbours in the launch and share it through L2
  const int rows = min(nb, g->M - m0);            // live rows of this tile (at least one)
  const int kblocks = (g->K + TC_BK - 1) / TC_BK;
  const int per = (kblocks + S - 1) / S;
  const int kb0 = rank * per, kb1 = min(kblocks, kb0 + per);
  const bool empty = kb0 >= kb1;                  // K too short for this rank: its partial is zero
  // activation ring first (a_stages tiles of nb x 64), then the W ring (w_stages tiles of 128 x 64)
  const int nb1 = PAIR ? swap2_first(nb) : nb, nb2 = nb - nb1;        // PAIR: the tile's rows in one MMA or two
  const int a_bytes = PAIR ? nb * TC_BK : nb * TC_BK * 2;
  // (a load from L2 takes some 1100 cycles to land and its stage another 300 to come back, a k-block's MMAs a tenth of
  // that: with few rows the whole k range of a split tile fits the ring, so nothing waits for a stage)
  // (two CTAs per SM: the smaller ring stays with W)
  const int a_stages = PAIR ? min(SW_A_STAGES_MAX, ring_bytes / (SW_W_BYTES + a_bytes)) : ring_bytes < SW_RING_BYTES_1 ? (nb > 64 ? 2 : 4) : nb > 128 ? 4 : nb > 64 ? 3 : nb > 32 ? 6 : SW_A_STAGES_MAX;
  const int w_stages = PAIR ? a_stages : min(SW_W_STAGES_MAX, (ring_bytes - a_stages * a_bytes) / SW_W_BYTES);
  const uint32_t w_base = base + a_stages * a_bytes;        // a multiple of 2 KB from a 1 KB-aligned base ...
  static_assert(SW_W_BYTES % 1024 == 0, "swizzle atoms");   // ... since nb is a multiple of 16
  const uint32_t tmem_cols = nb > 256 ? 512u : nb > 128 ? 256u : 128u;
  // what the epilogue needs of the descriptor and the bias (static), read here so that it is at hand when the
  // accumulator is; a lane owns four consecutive output columns
  const int N = g->N, epi = g->epi, ldc = g->ldc;
  void* const Cptr = g->C;
  const int col = lane * 4, n = n0 + col;
  float bias[4] = {0.f, 0.f, 0.f, 0.f};
  if ((epi & EPI_BIAS) && warp >= 2 && warp < SW_A_WARP) {
    const bf16* const bias_ptr = g->bias;
#pragma unroll
    for (int j = 0; j < 4; ++j) if (n + j < N) bias[j] = bf2f(bias_ptr[n + j]);
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < w_stages; ++s) { mbar_init(wfull_bar(s), 1); mbar_init(wempty_bar(s), 1); }
    for (int s = 0; s < a_stages; ++s) { mbar_init(afull_bar(s), 1); mbar_init(aempty_bar(s), 1); }
    mbar_init(tfull_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();          // the pair's leader has its barriers before anything is counted on them
  tc_fence_after();
  const uint32_t leader = (uint32_t)(2 * rank);    // PAIR: issues the MMAs of both
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer of W (tmW: box of 128 rows)
    tensormap_acquire(&g->tmW);
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      // (a stage's first use has nothing to wait for)
      if (kb - kb0 >= w_stages && !mbar_wait(wempty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 41); break; }
      if constexpr (PAIR) {
        if (half == 0) mbar_expect_tx_elect(wfull_bar(stage), 2u * (SW_W_BYTES + (uint32_t)a_bytes));   // (activations too)
        tma_load_2d_pair_elect(w_base + stage * SW_W_BYTES, &g->tmW, kb * TC_BK, n0, mapa_shared(wfull_bar(stage), leader));
      } else {
        mbar_expect_tx_elect(wfull_bar(stage), (uint32_t)SW_W_BYTES);
        tma_load_2d_elect(w_base + stage * SW_W_BYTES, &g->tmW, kb * TC_BK, n0, wfull_bar(stage));
      }
      if (++stage == w_stages) { stage = 0; phase ^= 1u; }
    }
    pdl_begin(BESIDE);                                    // (not beside: every thread of the kernel waits once, see common.cuh)
    if (!ok) { *abort_flag = 1; drain_sleep(200000ull); }
  } else if (warp == SW_A_WARP) {
    // ------------------------------------------------------------ TMA producer of the activations (tmA: box of nb rows)
    tensormap_acquire(&g->tmA);
    // the first copy after the wait finds its map (1B decoder, 27 requests: 1226 -> 1210 us a step; the larger tiles of the
    // tile-pair kernel and attention gained nothing)
    tensormap_prefetch_elect(&g->tmA);
    if (PAIR && nb2) { tensormap_acquire(&g->tmC); tensormap_prefetch_elect(&g->tmC); }
    pdl_begin(BESIDE);
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (kb - kb0 >= a_stages && !mbar_wait(PAIR ? wempty_bar(stage) : aempty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 44); break; }
      if constexpr (PAIR) {
        // (half of each MMA's rows; tmC holds the map for the second MMA's)
        const uint32_t bar = mapa_shared(wfull_bar(stage), leader);
        tma_load_2d_pair_elect(base + stage * a_bytes, &g->tmA, kb * TC_BK, m0 + half * (nb1 >> 1), bar);
        if (nb2) tma_load_2d_pair_elect(base + stage * a_bytes + nb1 * TC_BK, &g->tmC, kb * TC_BK, m0 + nb1 + half * (nb2 >> 1), bar);
      } else {
        mbar_expect_tx_elect(afull_bar(stage), (uint32_t)a_bytes);
        tma_load_2d_elect(base + stage * a_bytes, &g->tmA, kb * TC_BK, m0, afull_bar(stage));
      }
      if (++stage == a_stages) { stage = 0; phase ^= 1u; }
    }
    if (!ok) { *abort_flag = 1; drain_sleep(200000ull); }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (PAIR: of the pair, in its first CTA)
    if (half == 0) {
      bool ok = true;
      if constexpr (PAIR) {
        // (one barrier a stage for both operands and a look ahead under the issue, as in the tile-pair kernel)
        const uint32_t idesc = make_idesc_pair(nb1), idesc2 = make_idesc_pair(nb2);
        int stage = 0;
        uint32_t phase = 0;
        bool ready = false;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!ready && !mbar_wait<false>(wfull_bar(stage), phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 42); break; }
          const uint64_t dw = make_smem_desc(w_base + stage * SW_W_BYTES), da = make_smem_desc(base + stage * a_bytes);
          const uint64_t da2 = make_smem_desc(base + stage * a_bytes + nb1 * TC_BK);
          const uint32_t used = wempty_bar(stage);
          if (++stage == w_stages) { stage = 0; phase ^= 1u; }
          ready = mbar_test(wfull_bar(stage), phase);
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            mma_f16_pair_elect(tmem_base, dw + (uint64_t)(k * 2), da + (uint64_t)(k * 2), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          if (nb2) {
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)
              mma_f16_pair_elect(tmem_base + (uint32_t)nb1, dw + (uint64_t)(k * 2), da2 + (uint64_t)(k * 2), idesc2, (kb > kb0 || k > 0) ? 1u : 0u);
          }
          mma_commit_pair_elect(used, 3u << leader);
        }
      } else {
        const uint32_t idesc = make_idesc(nb);
        int ws = 0, as = 0;
        uint32_t wphase = 0, aphase = 0;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_both(afull_bar(as), aphase, wfull_bar(ws), wphase, abort_flag)) {
            ok = false;
            const int code = mbar_test(afull_bar(as), aphase) ? 42 : 45;
            if (lane == 0) atomicExch(status, code);
            break;
          }
          const uint64_t dw = make_smem_desc(w_base + ws * SW_W_BYTES), da = make_smem_desc(base + as * a_bytes);
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            mma_f16_elect(tmem_base, dw + (uint64_t)(k * 2), da + (uint64_t)(k * 2), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          mma_commit_elect(wempty_bar(ws));
          mma_commit_elect(aempty_bar(as));
          if (++ws == w_stages) { ws = 0; wphase ^= 1u; }
          if (++as == a_stages) { as = 0; aphase ^= 1u; }
        }
      }
      if (!ok) *abort_flag = 1;
      else if (!empty) {
        if constexpr (PAIR) mma_commit_pair_elect(tfull_bar, 3u << leader);
        else mma_commit_elect(tfull_bar);
      }
    }
  } else {
    // ------------------------------------------------------------ wait for this CTA's accumulator (warps 2..9)
    pdl_begin(BESIDE);
    acc_ok = empty || mbar_wait(tfull_bar, 0u, abort_flag);
    if (!acc_ok) {
      if (lane == 0) atomicExch(status, 43);
      *abort_flag = 1;
    }
  }
  // The slices go into the owners' operand rings, which must be idle: every CTA of the cluster has to be past
  // its last MMA before anyone sends.
  __syncthreads();
  if (S > 1) cluster_sync_relaxed();
  const int rp = ((nb + S - 1) / S + 3) & ~3;       // batch rows per owner
  if (warp >= 2 && warp < SW_A_WARP) {
    // ------------------------------------------------------------ accumulator -> the owners' shared memory
    // Batch row m0 + c (TMEM column c) belongs to CTA c / rp of the cluster.  Its buffer, over the idle operand
    // ring, is [S sources][rp batch rows][128 columns] fp32; this CTA fills plane `rank` of every owner.  The two
    // warps of a lane quarter take alternate blocks of 16 rows.
    const int quarter = warp & 3, alt = (warp - 2) >> 2;
    const uint32_t col_off = (uint32_t)(quarter * 32 + lane) * 4u;
    tc_fence_after();
    const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t plane = (uint32_t)(rank * rp) * (SW_BM * 4u) + col_off;
    for (int c = alt * 16; c < rows; c += 32) {
      uint32_t r[16];
      if (empty || !acc_ok) {
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = 0u;      // no k-block for this rank (or a wait that ran out): a zero partial
      } else {
        tmem_ld16(taddr + (uint32_t)c, r);
      }
      // (rp is a multiple of four, so four rows go to one owner; rows past the live ones are sent along with them)
#pragma unroll
      for (int j4 = 0; j4 < 16; j4 += 4) {
        const int owner = S == 1 ? 0 : (c + j4) / rp;
        const uint32_t dst = (S == 1 ? base : mapa_shared(base, (uint32_t)(PAIR ? 2 * owner + half : owner))) + plane + (uint32_t)(c + j4 - owner * rp) * (SW_BM * 4u);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (S == 1)
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + (uint32_t)j * (SW_BM * 4u)), "f"(__uint_as_float(r[j4 + j])) : "memory");
          else
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + (uint32_t)j * (SW_BM * 4u)), "f"(__uint_as_float(r[j4 + j])) : "memory");
        }
      }
    }
    tc_fence_before();
  }
  __syncthreads();
  if (S > 1) cluster_sync_all();                     // every slice has reached its owner (release / acquire)

  if (warp >= 2 && warp < SW_A_WARP) {
    // ------------------------------------------------------------ reduction in rank order + epilogue
    // This CTA owns rows m0 + rank * rp .. of the tile.  A warp takes whole rows, a lane four consecutive columns;
    // the S slices of U rows (and, for a residual output, the old values of C) are requested together, then added
    // in rank order.
    constexpr int U = 4;
    const int r0 = rank * rp;
    const int nrows = min(rp, rows - r0);            // this CTA's live rows (none when <= 0)
    const float* const red = reinterpret_cast<const float*>(base_ptr);
    const bool full = n + 4 <= N, some = n < N;
    const bool resid = (epi & EPI_RESID_F32) != 0;
#pragma unroll 1
    for (int l0 = warp - 2; l0 < nrows; l0 += SW_EPI_WARPS * U) {
      float4 old[U], v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int l = l0 + u * SW_EPI_WARPS;
        old[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (resid && l < nrows && some) {
          const float* cf = reinterpret_cast<const float*>(Cptr) + (size_t)(m0 + r0 + l) * ldc + n;
          if (full) old[u] = BESIDE ? __ldcg(reinterpret_cast<const float4*>(cf)) : *reinterpret_cast<const float4*>(cf);
          else { old[u].x = BESIDE ? __ldcg(cf) : cf[0]; if (n + 1 < N) old[u].y = BESIDE ? __ldcg(cf + 1) : cf[1]; if (n + 2 < N) old[u].z = BESIDE ? __ldcg(cf + 2) : cf[2]; }
        }
      }
      // (rows past the live ones read stale shared memory and are not stored: the U rows stay one straight piece of code)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int l = min(l0 + u * SW_EPI_WARPS, nrows - 1);
        v[u] = *reinterpret_cast<const float4*>(red + l * SW_BM + col);
#pragma unroll
        for (int q = 1; q < S; ++q) {
          const float4 p = *reinterpret_cast<const float4*>(red + (q * rp + l) * SW_BM + col);
          v[u].x += p.x; v[u].y += p.y; v[u].z += p.z; v[u].w += p.w;
        }
        v[u].x += bias[0]; v[u].y += bias[1]; v[u].z += bias[2]; v[u].w += bias[3];
      }
      if (epi & EPI_GELU) {
#pragma unroll
        for (int u = 0; u < U; ++u) { v[u].x = gelu_erf(v[u].x); v[u].y = gelu_erf(v[u].y); v[u].z = gelu_erf(v[u].z); v[u].w = gelu_erf(v[u].w); }
      }
      if (epi & EPI_SWIGLU) {
        // gate and up are adjacent output columns
#pragma unroll
        for (int u = 0; u < U; ++u) { v[u].x = silu_f(v[u].x) * v[u].y; v[u].y = silu_f(v[u].z) * v[u].w; }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int l = l0 + u * SW_EPI_WARPS;
          bf16* cb = reinterpret_cast<bf16*>(Cptr) + (size_t)(m0 + r0 + l) * ldc + (n >> 1);
          if (l < nrows && full) *reinterpret_cast<uint32_t*>(cb) = pack2(v[u].x, v[u].y);
          else if (l < nrows && n + 1 < N) {
            cb[0] = f2bf(v[u].x);
            if (n + 3 < N) cb[1] = f2bf(v[u].y);
          }
        }
      } else if (resid) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int l = l0 + u * SW_EPI_WARPS;
          float* cf = reinterpret_cast<float*>(Cptr) + (size_t)(m0 + r0 + l) * ldc + n;
          if (l < nrows && full) *reinterpret_cast<float4*>(cf) = make_float4(old[u].x + v[u].x, old[u].y + v[u].y, old[u].z + v[u].z, old[u].w + v[u].w);
          else if (l < nrows && some) { cf[0] = old[u].x + v[u].x; if (n + 1 < N) cf[1] = old[u].y + v[u].y; if (n + 2 < N) cf[2] = old[u].z + v[u].z; }
        }
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int l = l0 + u * SW_EPI_WARPS;
          bf16* cb = reinterpret_cast<bf16*>(Cptr) + (size_t)(m0 + r0 + l) * ldc + n;
          if (l < nrows && full) *reinterpret_cast<uint2*>(cb) = make_uint2(pack2(v[u].x, v[u].y), pack2(v[u].z, v[u].w));
          else if (l < nrows && some) {
            cb[0] = f2bf(v[u].x); if (n + 1 < N) cb[1] = f2bf(v[u].y); if (n + 2 < N) cb[2] = f2bf(v[u].z);
          }
        }
      }
    }
  }
  // (after the barrier above nobody touches another CTA's shared memory, so the CTAs may leave one by one)
  // (a pair leaves together: its first CTA's MMAs have read the other's operands and report to its barriers)
  pdl_end(BESIDE);
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
    else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

template <int S, bool PAIR>
cudaError_t launch_swap(const GemmGroup* groups, int n_groups, int total_items, int max_nb, int* status, int sm_count, cudaStream_t st, int beside) {
  const auto kernel = beside ? gemm_swap_kernel<S, true, PAIR> : gemm_swap_kernel<S, false, PAIR>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sw_smem(SW_RING_BYTES_1));
  if (e != cudaSuccess) return e;
  // Tiles of more than 128 rows need the large ring (the reduction lands nb x 512 bytes in it).
  // (clusters of eight one-SM CTAs were slow to place: 25.8 us against 15.4 with two CTAs per SM, 2048 x 8192 at 128 rows)
  const int ring_bytes = (!PAIR && max_nb <= 128 && (total_items * S > sm_count || S == 8)) ? SW_RING_BYTES_2 : SW_RING_BYTES_1;
  constexpr int CTAS = PAIR ? 2 * S : S;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(total_items * CTAS);
  cfg.blockDim = dim3(SW_THREADS);
  cfg.dynamicSmemBytes = sw_smem(ring_bytes);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CTAS;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, groups, n_groups, status, ring_bytes);
}

}  // namespace

// Rows of a tile (the MMA's N), k ranges per tile, and an estimate of the launch's time in microseconds.
// Up to 128 rows: ranges are doubled while the CTAs still fit two per SM and every range keeps at least four
// k-blocks (sixteen for the step from four to eight ranges, which pays only on a long K: 19.6 -> 15.4 us for
// 2048 x 8192 at 128 rows, nothing for 2048 x 2048).
// Above, one CTA takes an SM and the clusters have to be resident together: 74 of two CTAs, 33 of four and 15 of eight
// fit on 148 SMs (sizes between them fit no more CTAs; one cluster too many costs a second wave: 2048 x 2048 at 256
// rows 27 us with 16 clusters of eight, 15 on tile pairs).  A k-block costs 0.13 us + 0.7 ns per row, a seventh more once
// most SMs are at it (they share what L2 delivers), exchange and epilogue 20 ns per row; clusters
// of eight start later.  (Calls on their own, W cold, against tile pairs: 2048 x 8192 at 160 / 224 / 400 rows 26.7 / 28.7 / 30.0 and
// 41 / 41 / 42 us; 4096 x 4096 at 144 rows 25.0 and 29.7; 6144 x 4096 at 144 / 208 rows 27.8 / 29.9 and 31.8; 3072 x 2048 at 272 rows
// 21.5 and 21.7; 768 x 3072 at 394 rows 21.7 and 23.7; 32000 x 2048 at 272 rows 66.6 and 68.6.)
double gemm_swap_config(long long rows_cap, int N, int K, int sm_count, int* nb, int* ksplit) {
  const int tiles_n = (N + SW_BM - 1) / SW_BM, kblocks = (K + TC_BK - 1) / TC_BK;
  const int tiles_m = (int)((rows_cap + GEMM_SWAP_TILE_ROWS - 1) / GEMM_SWAP_TILE_ROWS);
  const int per = (int)((rows_cap + tiles_m - 1) / tiles_m);
  *nb = (per + 15) / 16 * 16;
  int s = 1;
  if (*nb <= 128) {
    while (s < 8 && tiles_n * s * 2 <= 2 * sm_count && kblocks / (s * 2) >= (s == 4 ? 16 : 4)) s *= 2;
    *ksplit = s;
    return 0.0;
  }
  const int tiles = tiles_n * tiles_m;
  const int fit[4] = {sm_count, sm_count / 2, sm_count * 33 / 148, sm_count * 15 / 148};
  for (int i = 1; i < 4; ++i)
    if (tiles <= fit[i] && kblocks >= 3 << i) s = 1 << i;
  *ksplit = s;
  const double rounds = (double)((tiles + fit[0] - 1) / fit[0]);
  const bool full = tiles * s > 2 * sm_count / 3;
  return 8.0 + 0.02 * *nb + (full ? 1.5 : 0.0) + (s == 8 ? 1.5 : 0.0) + rounds * ((kblocks + s - 1) / s) * (0.13 + 0.0007 * *nb) * (full ? 1.15 : 1.0);
}

int gemm_swap_tiles_n(int N) { return (N + SW_BM - 1) / SW_BM; }

cudaError_t launch_gemm_swap(const GemmGroup* groups, int n_groups, int total_items, int ksplit, int max_nb, int* status,
                             int sm_count, cudaStream_t st, int beside) {
  if (n_groups == 0 || total_items == 0) return cudaSuccess;
  switch (ksplit) {
    case 1: return launch_swap<1, false>(groups, n_groups, total_items, max_nb, status, sm_count, st, beside);
    case 2: return launch_swap<2, false>(groups, n_groups, total_items, max_nb, status, sm_count, st, beside);
    case 4: return launch_swap<4, false>(groups, n_groups, total_items, max_nb, status, sm_count, st, beside);
    case 8: return launch_swap<8, false>(groups, n_groups, total_items, max_nb, status, sm_count, st, beside);
  }
  return cudaErrorInvalidValue;
}

// ---- pairs of CTAs on 256 output columns
int gemm_swap2_first(int nb) { return swap2_first(nb); }
int gemm_swap2_tiles_n(int N) { return (N + 2 * SW_BM - 1) / (2 * SW_BM); }

// The estimate, in microseconds: a k-block costs what its operands take to arrive (0.14 us + 0.3 ns a row; two ranges of a K of 4096
// and more on all resident pairs 8 ns on top: W is then asked for twice as fast) or its MMAs, a tile
// 26 ns a row for exchange and epilogue; pairs of one launch: 74 clusters of two CTAs or 33 of four are resident.  Chosen from 129 rows
// (N and K decide) to some three thousand.  Calls on their own, W cold, the call's own 6 to 9 us included, against tile pairs:
//   2048 x 8192    513 / 1100 / 1280 / 1536 / 1792 / 2500 / 3000 rows  33.7 / 46 / 44 / 50 / 54 / 73 / 83  and  44 / 54 / 54 / 56 / 56 / 93 / 95
//   4096 x 14336   400 / 536 / 1100 / 1536 / 1792 rows                 59 / 66 / 101 / 130 / 155           and  71 / 87 / 153 / 155 / 159
//   4096 x 4096    256 / 536 / 1100 / 1536 rows                        25.6 / 31.8 / 43 / 53               and  29.7 / 35.9 / 55 / 57
//   3072 x 2048    192 / 1600 / 1900 rows                              20.5 / 32.8 / 33.8                  and  21.6 / 36.9 / 35.9
//   16384 x 2048   288 rows                                            42                                  and  46
// and against the form on one CTA, where the term for long K decides: 2048 x 8192 at 336 rows 30.6 and 29.1, at 512 31.8 and 34.8;
// 4096 x 14336 at 192 rows 49.7 and 44.3, at 256 50.4 and 52.2; 4096 x 4096 at 129 rows 25.7 and 25.0, at 208 25.6 and 27.1.
// Whole steps: 1B decoder, a prompt of 340 tokens 1484 us without that term and 1463 with it, 8B decoder, 144 tokens 4433 and 4392.
// Products it still gets wrong by more than a twentieth: 768 x 768 at 577 to 768 rows (17.4 us, tile pairs 15.4; a step of three images
// through ViT-B takes the same time with either).
// With a short K most of a tile's W is requested before the dependency wait, which a launch on its own does not show: one image through
// ViT-B (K 768) 578 us a step with its projections on tile pairs, 549 here.
double gemm_swap2_config(long long rows_cap, int N, int K, int sm_count, int* nb, int* ksplit) {
  const int tiles_n = gemm_swap2_tiles_n(N), kblocks = (K + TC_BK - 1) / TC_BK;
  const double start = kblocks <= 16 ? 7.0 : 8.5;
  double best = 0;
  *nb = 0;
  *ksplit = 1;
  for (int tiles_m = (int)((rows_cap + GEMM_SWAP2_TILE_ROWS - 1) / GEMM_SWAP2_TILE_ROWS); tiles_m <= 8; ++tiles_m) {
    const int rows = (int)(((rows_cap + tiles_m - 1) / tiles_m + 31) / 32 * 32);
    if (rows < 64) break;
    const double tile = 0.026 * rows;
    for (int s = 1; s <= 2; ++s) {
      const int tiles = tiles_n * tiles_m, fit = s == 1 ? sm_count / 2 : sm_count * 33 / 148;
      if (s == 2 && (tiles > fit || kblocks < 8)) continue;
      const int rounds = (tiles + fit - 1) / fit;
      const double arrival = 0.14 + 0.00031 * rows + (s == 2 && kblocks >= 64 && tiles >= 0.95 * fit ? 0.008 : 0.0);
      const double t = start + rounds * (tile + (kblocks + s - 1) / s * std::max(arrival, 0.00112 * rows)) + (rounds - 1) * 3.0;
      if (*nb == 0 || t < best) { best = t; *nb = rows; *ksplit = s; }
    }
  }
  return best;
}

// Up to 128 rows a tile of A would be mostly padding for the tile-pair kernel.  Above, the estimates decide.
int gemm_tc_choice(long long rows_cap, int N, int K, int epi, int sm_count, int* bn, int* ksplit) {
  int nb = 0, s = 1, nb2 = 0, s2 = 1, w = 0;
  const double t_swap = gemm_swap_config(rows_cap, N, K, sm_count, &nb, &s);
  if (rows_cap <= TC_BM) { *bn = nb; *ksplit = s; return GEMM_SWAP; }
  const double t_pair = gemm_pair_config(rows_cap, N, K, epi, sm_count, &w), t_swap2 = gemm_swap2_config(rows_cap, N, K, sm_count, &nb2, &s2);
  if (nb2 > 0 && t_swap2 < t_pair && t_swap2 < t_swap) { *bn = nb2; *ksplit = s2; return GEMM_SWAP2; }
  if (t_swap < t_pair) { *bn = nb; *ksplit = s; return GEMM_SWAP; }
  *bn = w; *ksplit = 1;
  return GEMM_PAIR;
}

cudaError_t launch_gemm_swap2(const GemmGroup* groups, int n_groups, int total_items, int ksplit, int* status, int sm_count, cudaStream_t st, int beside) {
  if (n_groups == 0 || total_items == 0) return cudaSuccess;
  if (ksplit == 1) return launch_swap<1, true>(groups, n_groups, total_items, 0, status, sm_count, st, beside);
  if (ksplit == 2) return launch_swap<2, true>(groups, n_groups, total_items, 0, status, sm_count, st, beside);
  return cudaErrorInvalidValue;
}

}  // namespace epara
