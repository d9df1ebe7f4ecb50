// Grouped bf16 GEMM on the sm_100a tensor cores: C_g = epi(A_g W_g^T + bias_g) for groups of more than 128 rows.
//
// One persistent launch covers every group (one group = one model's GEMM in this wave, with its own M, N, K and tile
// width bn in {128, 192, 256}; 64 in a finer last round, see fine_tail in epara_api.cu).  Work items -- tiles of 256 rows x bn columns, each worked by two CTAs of a cluster --
// are numbered group after group; pair i takes items i, i + pairs, ...  Inside a CTA the roles run concurrently:
//   warp 0            TMA producer of A: its own 128 rows x 64 columns of every k-block;
//   warp 18           TMA producer of W: half of the tile's W rows (plain, non-multicast cp.async.bulk.tensor;
//                     out-of-range rows / columns arrive as zeros);
//   warp 1 of rank 0  MMA issuer: tcgen05.mma cta_group::2 (M 256, N bn, K 16) into one of two TMEM accumulators (256
//                     columns each), releasing stages with tcgen05.commit (warp 1 of rank 1 prefetches residual rows);
//   warps 2..17       epilogue: tcgen05.ld of the finished accumulator (four warps per TMEM lane quarter, a quarter of
//                     the tile's columns each; two of them half each of a tile 64 wide), bias / GELU / SwiGLU / fp32 residual update, bf16 store -- while the
//                     MMA warp already fills the other accumulator.
// The K reduction of an output element is the same sequence whatever else is in the launch.
// Every mbarrier wait is bounded: when a wait runs out the kernel records a code in *status, all roles leave their
// loops, TMEM is freed and the kernel returns.
#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace epara {

namespace {

using namespace tc;

constexpr int A_BYTES = TC_BM * TC_BK * 2;          // 16 KB
constexpr int PAIR_STAGES = 6;
constexpr int PAIR_STAGE_BYTES = 2 * A_BYTES;       // 32 KB: A 16 KB + at most 128 rows of W
constexpr int RING_BYTES = PAIR_STAGES * PAIR_STAGE_BYTES;
constexpr int ACC_COLS = TC_BN_MAX;                 // TMEM columns per accumulator
constexpr int TMEM_COLS = 2 * ACC_COLS;             // 512: the whole TMEM of the SM
constexpr int EPI_WARPS = 16;
constexpr int N_THREADS = 64 + EPI_WARPS * 32;
constexpr int STAGE_OUT_BYTES = EPI_WARPS * 2048;    // epilogue staging: 2 KB (32 rows x 64 bytes) per warp
constexpr size_t SMEM_BYTES = 1024 + (size_t)RING_BYTES + STAGE_OUT_BYTES + 256;

__device__ __forceinline__ int find_group_tc(const GemmGroup* groups, int n, int item) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (groups[mid].tile_start <= item) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Register copy of a group's scalar fields for the epilogue threads.  The descriptors live in
// global memory and the epilogue is full of asm statements that clobber memory, so reading
// fields through the descriptor pointer would reload them (at L2 latency) again and again.
struct GView {
  const bf16* bias;
  const CUtensorMap* tmC;
  int N, epi, tile_start, tiles_m, tiles_n, bn, c_rows, m_base, n_base;
};
__device__ __forceinline__ GView load_view(const GemmGroup* g) {
  GView v;
  v.bias = g->bias; v.N = g->N; v.epi = g->epi; v.tile_start = g->tile_start;
  v.tiles_m = g->tiles_m; v.tiles_n = g->tiles_n; v.bn = g->bn;
  v.tmC = &g->tmC; v.c_rows = g->c_rows; v.m_base = g->m_base; v.n_base = g->n_base;
  return v;
}

// Per-thread copy of the fields the producer and issuer roles need, refreshed only when the item leaves
// the current group (descriptor reads from global memory are latency the MMA issuer cannot hide).
struct GroupCache {
  const GemmGroup* g;
  int start, end, tiles_n, bn, kblocks, m_base, n_base;
};
__device__ __forceinline__ void group_cache(GroupCache& c, const GemmGroup* groups, int n_groups, int item) {
  if (c.g != nullptr && item >= c.start && item < c.end) return;
  const GemmGroup* g = groups + find_group_tc(groups, n_groups, item);
  c.g = g;
  c.start = g->tile_start;
  c.tiles_n = g->tiles_n;
  c.bn = g->bn;
  c.m_base = g->m_base;
  c.n_base = g->n_base;
  c.end = c.start + g->tiles_m * g->tiles_n;
  c.kblocks = (g->K + TC_BK - 1) / TC_BK;
}

// Columns of a tile that an epilogue warp works: a quarter, of 64-wide tiles half (two of the four then have none).
__device__ __forceinline__ int part_cols(int bn) { return max(bn >> 2, 32); }

// A work item of a group as the CTA of the given rank sees it: its first row and the tile's first column.
struct Item {
  int m0, n0;
};
template <class G>
__device__ __forceinline__ Item decode_item(const G& g, int local, int rank) {
  Item it;
  it.m0 = g.m_base + (local / g.tiles_n) * (2 * TC_BM) + rank * TC_BM;
  it.n0 = g.n_base + (local % g.tiles_n) * g.bn;
  return it;
}

// Direct epilogue of one warp for one tile, with no block-level barrier.  Warp (quarter, part) owns
// rows quarter*32..+31 and the part-th part_cols() of the tile's columns (a quarter; none is left for parts 2 and 3 of a tile 64 wide).  Per chunk (32 accumulator
// columns; 16 for an fp32 residual) each lane turns its row's values into outputs and parks them in
// the warp's 2 KB staging area (64-byte rows, SwiGLU 32-byte rows, 16-byte pieces in the TMA swizzle
// pattern, which also keeps the stores free of bank conflicts); one lane then hands the 32-row box to
// the TMA unit: a plain store for bf16 outputs, a reduce-add for the fp32 residual (the addition
// happens at L2; the SM never reads C).  The hardware clips rows and columns outside the tensor.
// The accumulator is handed back to the MMA warp as soon as this warp's last chunk has left TMEM.
// MODE: 0 bf16 output, 1 SwiGLU, 2 fp32 residual.
// tempty is a shared::cluster address (the accumulator barrier of the pair's leader).
template <int MODE>
__device__ __forceinline__ void epi_direct(const GView& g, const Item& it, uint32_t taddr, unsigned char* wst, int quarter,
                                           int part, int lane, uint2 bias_reg, uint32_t tempty) {
  constexpr int CW = (MODE == 2) ? 16 : 32;                  // accumulator columns per chunk
  const uint32_t wst_u = smem_u32(wst);
  const int y0 = it.m0 + quarter * 32;
  const bool box_ok = y0 < g.c_rows;                         // some row of this warp's box is inside the tensor
  const int c_begin = part * part_cols(g.bn);
  const int c_end = min(c_begin + part_cols(g.bn), min(g.bn, g.N - it.n0));
  if (c_begin >= c_end) {                                    // nothing to do for this warp: release at once
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(tempty);
    return;
  }
#pragma unroll 1
  for (int c = c_begin; c < c_end; c += CW) {
    const int n = it.n0 + c;
    float v[CW];
    {
      uint32_t r[CW];
      if (MODE == 2) tmem_ld16(taddr + (uint32_t)c, r); else tmem_ld32(taddr + (uint32_t)c, r);
#pragma unroll
      for (int j = 0; j < CW; ++j) v[j] = __uint_as_float(r[j]);
    }
    if (c + CW >= c_end) {                                   // that was this warp's last read of the accumulator
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(tempty);
    }
    if (g.epi & EPI_BIAS) {
      // the bias values of this chunk sit in consecutive lanes of bias_reg (zero past N)
      const int lane0 = (c - c_begin) >> 2;
#pragma unroll
      for (int jj = 0; jj < CW / 2; ++jj) {
        const uint32_t w = __shfl_sync(0xffffffffu, (jj & 1) ? bias_reg.y : bias_reg.x, lane0 + (jj >> 1));
        v[2 * jj] += __uint_as_float(w << 16);
        v[2 * jj + 1] += __uint_as_float(w & 0xffff0000u);
      }
    }
    if (g.epi & EPI_GELU) {
#pragma unroll
      for (int j = 0; j < CW; j += 2) gelu_erf2(v[j], v[j + 1]);
    }
    // the previous box of this warp must have been read out of the staging area
    if (lane == 0) bulk_wait_read0();
    __syncwarp();
    if (MODE == 2) {
      unsigned char* srow = wst + lane * 64;
      const int sw = (lane >> 1) & 3;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        *reinterpret_cast<float4*>(srow + ((k ^ sw) << 4)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    } else if (MODE == 1) {
      unsigned char* srow = wst + lane * 32;                 // 32 columns -> 16 outputs -> 2 pieces
      const int sw = (lane >> 2) & 1;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint4 o;
        o.x = pack2(silu_f(v[16 * k]) * v[16 * k + 1], silu_f(v[16 * k + 2]) * v[16 * k + 3]);
        o.y = pack2(silu_f(v[16 * k + 4]) * v[16 * k + 5], silu_f(v[16 * k + 6]) * v[16 * k + 7]);
        o.z = pack2(silu_f(v[16 * k + 8]) * v[16 * k + 9], silu_f(v[16 * k + 10]) * v[16 * k + 11]);
        o.w = pack2(silu_f(v[16 * k + 12]) * v[16 * k + 13], silu_f(v[16 * k + 14]) * v[16 * k + 15]);
        *reinterpret_cast<uint4*>(srow + ((k ^ sw) << 4)) = o;
      }
    } else {
      unsigned char* srow = wst + lane * 64;                 // 32 columns -> 4 pieces
      const int sw = (lane >> 1) & 3;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint4 o;
        o.x = pack2(v[8 * k], v[8 * k + 1]); o.y = pack2(v[8 * k + 2], v[8 * k + 3]);
        o.z = pack2(v[8 * k + 4], v[8 * k + 5]); o.w = pack2(v[8 * k + 6], v[8 * k + 7]);
        *reinterpret_cast<uint4*>(srow + ((k ^ sw) << 4)) = o;
      }
    }
    fence_async_smem();                      // the staged values must be visible to the TMA unit
    __syncwarp();
    if (lane == 0 && box_ok) {
      if (MODE == 2) tma_reduce_add_2d(g.tmC, wst_u, n, y0);
      else tma_store_2d(g.tmC, wst_u, MODE == 1 ? (n >> 1) : n, y0);
      bulk_commit();
    }
  }
}

// ---------------------------------------------------------------------------------- tile pairs
// 256 x bn tiles worked by two CTAs of a cluster (the two SMs of a TPC): each CTA loads its own 128 rows of A and
// bn / 2 rows of W per k-block (32 KB at bn 256, against 48 for a CTA on its own: six ring stages, and a third less
// traffic from L2 per flop -- an SM takes in some 64 bytes a cycle, which is what bounds the main loop: 540 cycles per
// k-block at bn 256, 430 at bn 128, where the MMAs take 512 and 256).  Rank 0 issues one M = 256 MMA for both, the
// accumulator rows of a CTA's half live in its own TMEM and its own epilogue warps write them out.  Barriers: every
// CTA's loads are counted on rank 0's full barrier; the MMA completion is reported to the empty / accumulator-full
// barriers of both CTAs; the epilogue warps of both report a drained accumulator to rank 0.

// A producer that gives up cannot await its copies in flight (their bytes are counted on the leader's
// barrier, which may never complete once the peer has given up too): it sleeps this long instead, far
// more than a copy takes, before the CTAs meet at the closing cluster barrier.
constexpr unsigned long long PAIR_DRAIN_NS = 200000ull;
constexpr int PAIR_W_WARP = 2 + EPI_WARPS;                     // the warp after the epilogue warps loads W
constexpr int PAIR_THREADS = N_THREADS + 32;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PAIR_THREADS, 1)
gemm_tc_pair_kernel(const GemmGroup* __restrict__ groups, int n_groups, int total_items, int* __restrict__ status, int beside) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  unsigned char* stage_out = base_ptr + RING_BYTES;
  const uint32_t bars = base + RING_BYTES + STAGE_OUT_BYTES;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (PAIR_STAGES + s); };
  auto tfull_bar = [&](int a) { return bars + 8u * (2 * PAIR_STAGES + a); };
  auto tempty_bar = [&](int a) { return bars + 8u * (2 * PAIR_STAGES + 2 + a); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + RING_BYTES + STAGE_OUT_BYTES + 8 * (2 * PAIR_STAGES + 4));
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < PAIR_STAGES; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), 2 * EPI_WARPS); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                        // the peer's barriers exist before anything is reported to them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer of A (one per CTA)
    // (A and W have a warp each: a k-block costs its issuer a wait and a TMA issue, and with both operands on one
    // warp that is more than the MMAs of a k-block take once tiles are short.)
    int stage = 0, used = 0;                   // (a stage's first use has nothing to wait for)
    uint32_t phase = 0;
    bool ok = true;
    const GemmGroup* g_prev = nullptr;
    GroupCache gc;
    gc.g = nullptr;
    if (pair < total_items) {
      group_cache(gc, groups, n_groups, pair);
      tensormap_acquire(&gc.g->tmA);
      g_prev = gc.g;
    }
    pdl_begin(beside);
    for (int item = pair; item < total_items && ok; item += n_pairs) {
      group_cache(gc, groups, n_groups, item);
      const GemmGroup* g = gc.g;
      const Item it = decode_item(gc, item - gc.start, rank);
      if (g != g_prev) { tensormap_acquire(&g->tmA); g_prev = g; }
      const uint32_t bytes = 2u * (A_BYTES + (uint32_t)(gc.bn >> 1) * TC_BK * 2);   // both CTAs' boxes of a k-block
      for (int kb = 0; kb < gc.kblocks; ++kb) {
        if (++used > PAIR_STAGES && !mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 31); break; }
        if (rank == 0) mbar_expect_tx_elect(full_bar(stage), bytes);
        tma_load_2d_pair_elect(base + stage * PAIR_STAGE_BYTES, &g->tmA, kb * TC_BK, it.m0, mapa_shared(full_bar(stage), 0));
        if (++stage == PAIR_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) { *abort_flag = 1; drain_sleep(PAIR_DRAIN_NS); }
  } else if (warp == PAIR_W_WARP) {
    // ------------------------------------------------------------ TMA producer of W (one per CTA)
    // Weights are never written by a kernel, so this warp does not wait for the earlier kernels of the
    // stream: the first stages' W boxes are on their way while those still run.  (Bytes that land before
    // rank 0 has announced them leave the barrier's count negative for a while, which is allowed; the
    // phase cannot complete before that thread's own arrival.)
    int stage = 0, used = 0;                   // (a stage's first use has nothing to wait for)
    uint32_t phase = 0;
    bool ok = true;
    const GemmGroup* g_prev = nullptr;
    GroupCache gc;
    gc.g = nullptr;
    for (int item = pair; item < total_items && ok; item += n_pairs) {
      group_cache(gc, groups, n_groups, item);
      const GemmGroup* g = gc.g;
      const Item it = decode_item(gc, item - gc.start, rank);
      if (g != g_prev) { tensormap_acquire(&g->tmW); g_prev = g; }
      const int n_half = it.n0 + rank * (gc.bn >> 1);
      for (int kb = 0; kb < gc.kblocks; ++kb) {
        if (++used > PAIR_STAGES && !mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 35); break; }
        tma_load_2d_pair_elect(base + stage * PAIR_STAGE_BYTES + A_BYTES, &g->tmW, kb * TC_BK, n_half, mapa_shared(full_bar(stage), 0));
        if (++stage == PAIR_STAGES) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok) { *abort_flag = 1; drain_sleep(PAIR_DRAIN_NS); }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------------------------------------------------- MMA issuer
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true, ready = false;
      GroupCache gc;
      gc.g = nullptr;
      for (int item = pair; item < total_items && ok; item += n_pairs) {
        group_cache(gc, groups, n_groups, item);
        const uint32_t idesc = make_idesc_pair(gc.bn);
        if (!mbar_wait(tempty_bar(acc), acc_phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 32); break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * ACC_COLS);
        for (int kb = 0; kb < gc.kblocks; ++kb) {
          if (!ready && !mbar_wait<false>(full_bar(stage), phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 33); break; }
          const uint32_t sa = base + stage * PAIR_STAGE_BYTES;
          const uint64_t da = make_smem_desc(sa), db = make_smem_desc(sa + A_BYTES);
          const uint32_t used = empty_bar(stage);
          if (++stage == PAIR_STAGES) { stage = 0; phase ^= 1u; }
          ready = mbar_test(full_bar(stage), phase);      // a look ahead, under the issue of this k-block
#pragma unroll
          for (int k = 0; k < TC_BK / 16; ++k)
            mma_f16_pair_elect(d_tmem, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc, (kb > 0 || k > 0) ? 1u : 0u);
          mma_commit_pair_elect(used);
        }
        if (!ok) break;
        mma_commit_pair_elect(tfull_bar(acc));
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
      if (!ok) *abort_flag = 1;
    } else {
      // ---------------------------------------------------------- L2 prefetch of residual tiles
      // The fp32 residual of both CTAs' rows is added to at L2 by the epilogue's reduce stores: this otherwise idle
      // warp asks for those lines ahead of time so that the additions do not wait on HBM.
      pdl_begin(beside);
      for (int item = pair; item < total_items; item += n_pairs) {
        const GemmGroup& g = groups[find_group_tc(groups, n_groups, item)];
        if (!(g.epi & EPI_RESID_F32)) continue;
        const Item it = decode_item(g, item - g.tile_start, 0);
        const int ncols = min(g.bn, g.N - it.n0);
        for (int r = lane; r < 2 * TC_BM && it.m0 + r < g.M; r += 32) {
          const float* rowp = reinterpret_cast<const float*>(g.C) + (size_t)(it.m0 + r) * g.ldc + it.n0;
          for (int c = 0; c < ncols; c += 32)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rowp + c));
        }
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..17 of both CTAs)
    pdl_begin(beside);
    const int ew = warp - 2;
    const int quarter = warp & 3;
    const int part = ew >> 2;
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    GView g;
    int g_end = -1;
    g.tile_start = 0;
    for (int item = pair; item < total_items && ok; item += n_pairs) {
      if (item >= g_end || item < g.tile_start) {
        g = load_view(groups + find_group_tc(groups, n_groups, item));
        g_end = g.tile_start + g.tiles_m * g.tiles_n;
        if (lane == 0) tensormap_acquire(g.tmC);
      }
      const Item it = decode_item(g, item - g.tile_start, rank);
      uint2 bias_reg = make_uint2(0u, 0u);
      if (g.epi & EPI_BIAS) {
        const int nb = it.n0 + part * part_cols(g.bn) + lane * 4;
        if (lane * 4 >= part_cols(g.bn)) {
          // beyond this warp's columns
        } else if (nb + 4 <= g.N) {
          bias_reg = __ldg(reinterpret_cast<const uint2*>(g.bias + nb));
        } else {
          unsigned short e[4] = {0, 0, 0, 0};
#pragma unroll
          for (int j = 0; j < 4; ++j) if (nb + j < g.N) e[j] = __bfloat16_as_ushort(g.bias[nb + j]);
          bias_reg = make_uint2((uint32_t)e[0] | ((uint32_t)e[1] << 16), (uint32_t)e[2] | ((uint32_t)e[3] << 16));
        }
      }
      if (!mbar_wait(tfull_bar(acc), acc_phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 34); break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(acc * ACC_COLS);
      unsigned char* wst = stage_out + ew * 2048;
      const uint32_t te = mapa_shared(tempty_bar(acc), 0);
      if (g.epi & EPI_RESID_F32) epi_direct<2>(g, it, taddr, wst, quarter, part, lane, bias_reg, te);
      else if (g.epi & EPI_SWIGLU) epi_direct<1>(g, it, taddr, wst, quarter, part, lane, bias_reg, te);
      else epi_direct<0>(g, it, taddr, wst, quarter, part, lane, bias_reg, te);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (lane == 0) bulk_wait_done0();
    if (!ok) *abort_flag = 1;
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                        // neither CTA leaves while the other may still read its operands or signal it
  pdl_end(beside);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------------------------- fused MLP block
// z += GELU(h W1^T + b1) W2^T + b2 for encoder blocks with d <= 384: the 4d-wide hidden tensor never leaves
// the SM.  A cluster of two CTAs works one 256-row tile (cta_group::2, as in the tile-pair kernel).  Per tile
// the CTA's 128 rows of h stay in shared memory (d / 64 k-blocks of 16 KB); the hidden layer is taken in chunks
// of 128 columns:
//   S = h W1_c^T         (M 256, N 128, K d)  into tensor-memory columns 384..511,
//   P = bf16(GELU(S + b1_c)) by the 16 epilogue warps, written to shared memory in the K-major 128-byte-swizzled
//                        layout an A operand has (two units of 128 rows x 64 columns),
//   O += P W2_c^T        (M 256, N d, K 128)  into columns 0..d-1 (two MMAs of N = d / 2 per k step when d > 256),
// and after the last chunk O + b2 is added to z by TMA reduce-adds, as in any fp32-residual GEMM.  The rounding points are those of the unfused pair of GEMMs (the hidden tensor is rounded to bf16 once,
// the k order of both contractions is ascending), so a request's bits do not change with the kernel.
// The two contractions have an issuing thread each (warp 1 for S, the last warp for O): the chains only meet
// through the epilogue warps (S -> P), so the tensor core works on the next chunk's S while this chunk's GELU is
// computed and on this chunk's O while the next S is read out, and neither thread's issue time delays the other chain.
// P is a ring of three units of 64 hidden columns, so that a chunk's P is written while the O of the chunk before still runs
// (with one buffer of a whole chunk that was one chain: 5.5 thousand cycles a chunk, 2.8 of them an epilogue warp's wait for the
// buffer; with the ring 4.3, with GELU two values an instruction and biases by load instead of shuffle 3.5).
// What bounds it: per chunk 3.07 thousand cycles of tensor work and about as many of shared memory (h is read again for every
// S, P for every O: 290 KB of operands, 100 KB of arriving weights, 32 KB of P at 128 bytes a cycle); an epilogue warp spends 1.0
// thousand waiting for S, 0.2 reading it, 1.5 on bias and GELU, 0.6 on P.  A tile's output takes 11 thousand, 2 to 3 of them until O is
// complete: 196 KB a CTA at the rate of the reductions at L2, all CTAs at once (boxes of 16-column rows: 15 thousand).
// 203 images of ViT-S: 94 us a launch before, 80 now, at 1.69 GHz under the power cap (1.77 before).
// Weights stream through two rings (W1: four slots of one k-block of a chunk half, 8 KB; W2: two of 24 KB), each with its own
// producer thread.  P's ring doubles as the staging area of the final epilogue (P is idle by then).
constexpr int MLP_W1_BYTES = 64 * 128, MLP_W2_BYTES = 24 * 1024;   // a k-block of a chunk half
constexpr int MLP_W1_SLOTS = 4, MLP_W2_SLOTS = 2, MLP_SLOTS = MLP_W1_SLOTS + MLP_W2_SLOTS;
constexpr int MLP_O_WARP = PAIR_W_WARP + 1;                    // issues the second contraction
constexpr int MLP_THREADS = PAIR_THREADS + 32;
constexpr int MLP_X_BYTES = 6 * A_BYTES;                       // d <= 384: at most six k-blocks of 128 x 64
constexpr int MLP_P_UNITS = 3;                                 // 128 rows x 64 hidden columns each, bf16
constexpr int MLP_P_BYTES = MLP_P_UNITS * A_BYTES;
constexpr int MLP_OFF_P = MLP_X_BYTES;
constexpr int MLP_OFF_RING = MLP_OFF_P + MLP_P_BYTES;
constexpr int MLP_OFF_W2 = MLP_OFF_RING + MLP_W1_SLOTS * MLP_W1_BYTES;
constexpr int MLP_OFF_BAR = MLP_OFF_W2 + MLP_W2_SLOTS * MLP_W2_BYTES;
constexpr size_t MLP_SMEM_BYTES = 1024 + (size_t)MLP_OFF_BAR + 256;
static_assert(MLP_SMEM_BYTES <= 227 * 1024, "shared memory of one SM");
static_assert(EPI_WARPS * 2048 <= MLP_P_BYTES, "the final epilogue stages its boxes in P");
constexpr int MLP_S_COL = 384;                                 // S behind the output accumulator
constexpr int MLP_CHUNK = 128;
enum { MB_W_FULL = 0, MB_W_EMPTY = MLP_SLOTS, MB_X_FULL = 2 * MLP_SLOTS, MB_X_EMPTY, MB_S_FULL, MB_S_EMPTY, MB_O_FULL, MB_O_EMPTY,
       MB_STAGE_FREE, MB_P_FULL, MB_P_EMPTY = MB_P_FULL + MLP_P_UNITS, MB_COUNT = MB_P_EMPTY + MLP_P_UNITS };
static_assert(8 * MB_COUNT + 16 <= 256, "barrier area");

__device__ __forceinline__ int find_group_mlp(const MlpGroup* groups, int n, int item) {
  int gi = 0;
  for (int i = 1; i < n; ++i) if (groups[i].tile_start <= item) gi = i;
  return gi;
}
// Geometry of a group in registers (the single-thread roles cannot hide descriptor loads).
struct MlpGeo {
  const MlpGroup* g;
  int start, end, kb1, nc, n2, n2i;
};
__device__ __forceinline__ void mlp_geo(MlpGeo& c, const MlpGroup* groups, int n_groups, int item) {
  if (c.g != nullptr && item >= c.start && item < c.end) return;
  const MlpGroup* g = groups + find_group_mlp(groups, n_groups, item);
  c.g = g;
  c.start = g->tile_start;
  c.end = c.start + g->tiles_m;
  const int d = g->d;
  c.kb1 = d >> 6;                       // k-blocks of the first contraction
  c.nc = g->F / MLP_CHUNK;              // chunks of the hidden layer
  c.n2i = d > 256 ? 2 : 1;              // MMAs per k step of the second contraction
  c.n2 = d / c.n2i;                     // and their N
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(MLP_THREADS, 1)
gemm_mlp_pair_kernel(const MlpGroup* __restrict__ groups, int n_groups, int total_items, int* __restrict__ status, int beside) {
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  const uint32_t bars = base + MLP_OFF_BAR;
  auto bar = [&](int i) { return bars + 8u * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + MLP_OFF_BAR + 8 * MB_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MLP_SLOTS; ++s) { mbar_init(bar(MB_W_FULL + s), 1); mbar_init(bar(MB_W_EMPTY + s), 1); }
    mbar_init(bar(MB_X_FULL), 1); mbar_init(bar(MB_X_EMPTY), 1);
    mbar_init(bar(MB_S_FULL), 1); mbar_init(bar(MB_S_EMPTY), 2 * EPI_WARPS);
    for (int u = 0; u < MLP_P_UNITS; ++u) { mbar_init(bar(MB_P_FULL + u), EPI_WARPS); mbar_init(bar(MB_P_EMPTY + u), 1); }
    mbar_init(bar(MB_O_FULL), 1); mbar_init(bar(MB_O_EMPTY), 2 * EPI_WARPS);
    mbar_init(bar(MB_STAGE_FREE), EPI_WARPS);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"((uint32_t)TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                        // the peer's barriers exist before anything is reported to them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer of h and W1 (one per CTA)
    // Per tile: the CTA's rows of h (once the tile before has been used by its last S), then W1 chunk by chunk.
    bool ok = true;
    bool waited = false;
    const MlpGroup* g_prev = nullptr;
    MlpGeo gc;
    gc.g = nullptr;
    int slot = 0;
    uint32_t phase = 0, t = 0;
    for (int item = pair; item < total_items && ok; item += n_pairs, ++t) {
      mlp_geo(gc, groups, n_groups, item);
      const MlpGroup* g = gc.g;
      if (g != g_prev) { tensormap_acquire(&g->tmX); tensormap_acquire(&g->tmW1); g_prev = g; }
      const int m0 = (item - gc.start) * (2 * TC_BM) + rank * TC_BM;
      if (!mbar_wait(bar(MB_X_EMPTY), (t & 1u) ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 41); break; }
      if (!waited) { pdl_begin(beside); waited = true; }   // h is written by the kernel before this one
      if (rank == 0) mbar_expect_tx_elect(bar(MB_X_FULL), 2u * (uint32_t)gc.kb1 * A_BYTES);
      for (int kb = 0; kb < gc.kb1; ++kb)
        tma_load_2d_pair_elect(base + kb * A_BYTES, &g->tmX, kb * TC_BK, m0, mapa_shared(bar(MB_X_FULL), 0));
      for (int c = 0; c < gc.nc && ok; ++c) {
        for (int kb = 0; kb < gc.kb1; ++kb) {
          if (!mbar_wait(bar(MB_W_EMPTY + slot), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 42); break; }
          if (rank == 0) mbar_expect_tx_elect(bar(MB_W_FULL + slot), 2u * MLP_W1_BYTES);
          tma_load_2d_pair_elect(base + MLP_OFF_RING + slot * MLP_W1_BYTES, &g->tmW1, kb * TC_BK, c * MLP_CHUNK + rank * 64, mapa_shared(bar(MB_W_FULL + slot), 0));
          if (++slot == MLP_W1_SLOTS) { slot = 0; phase ^= 1u; }
        }
      }
    }
    if (!ok) { *abort_flag = 1; drain_sleep(PAIR_DRAIN_NS); }
  } else if (warp == PAIR_W_WARP) {
    // ------------------------------------------------------------ TMA producer of W2 (one per CTA)
    // (Weights are never written by a kernel: no wait for earlier kernels.)
    int slot = 0;
    uint32_t phase = 0;
    bool ok = true;
    const MlpGroup* g_prev = nullptr;
    MlpGeo gc;
    gc.g = nullptr;
    for (int item = pair; item < total_items && ok; item += n_pairs) {
      mlp_geo(gc, groups, n_groups, item);
      const MlpGroup* g = gc.g;
      if (g != g_prev) { tensormap_acquire(&g->tmW2); g_prev = g; }
      const int half = gc.n2 >> 1;                         // rows of one MMA's B operand held by this CTA
      for (int c = 0; c < gc.nc && ok; ++c) {
        for (int j = 0; j < 2; ++j) {                      // the chunk's two k-blocks
          if (!mbar_wait(bar(MB_W_EMPTY + MLP_W1_SLOTS + slot), phase ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 43); break; }
          if (rank == 0) mbar_expect_tx_elect(bar(MB_W_FULL + MLP_W1_SLOTS + slot), 2u * (uint32_t)gc.n2i * (uint32_t)half * 128u);
          for (int i = 0; i < gc.n2i; ++i)
            tma_load_2d_pair_elect(base + MLP_OFF_W2 + slot * MLP_W2_BYTES + i * half * 128, &g->tmW2, (2 * c + j) * TC_BK,
                                   i * gc.n2 + rank * half, mapa_shared(bar(MB_W_FULL + MLP_W1_SLOTS + slot), 0));
          if (++slot == MLP_W2_SLOTS) { slot = 0; phase ^= 1u; }
        }
      }
    }
    if (!ok) { *abort_flag = 1; drain_sleep(PAIR_DRAIN_NS); }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer of S = h W1_c^T (rank 0 only)
    if (rank == 0) {
      int slot = 0;
      uint32_t phase = 0;
      uint32_t n_s = 0, t = 0;                // chunks issued, tiles started
      bool ok = true;
      MlpGeo gc;
      gc.g = nullptr;
      const uint32_t idesc_s = make_idesc_pair(MLP_CHUNK);
      for (int item = pair; item < total_items && ok; item += n_pairs, ++t) {
        mlp_geo(gc, groups, n_groups, item);
        if (!mbar_wait<false>(bar(MB_X_FULL), t & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 49); break; }
        for (int c = 0; c < gc.nc && ok; ++c, ++n_s) {
          // S is free once the epilogue warps have read the chunk before out of it
          if (n_s > 0 && !mbar_wait<false>(bar(MB_S_EMPTY), (n_s - 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 44); break; }
          tc_fence_after();
          for (int kb = 0; kb < gc.kb1; ++kb) {
            if (!mbar_wait<false>(bar(MB_W_FULL + slot), phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 45); break; }
            const uint64_t da = make_smem_desc(base + kb * A_BYTES), db = make_smem_desc(base + MLP_OFF_RING + slot * MLP_W1_BYTES);
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)
              mma_f16_pair_elect(tmem_base + MLP_S_COL, da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc_s, (kb > 0 || k > 0) ? 1u : 0u);
            mma_commit_pair_elect(bar(MB_W_EMPTY + slot));
            if (++slot == MLP_W1_SLOTS) { slot = 0; phase ^= 1u; }
          }
          if (!ok) break;
          mma_commit_pair_elect(bar(MB_S_FULL));
          if (c == gc.nc - 1) mma_commit_pair_elect(bar(MB_X_EMPTY));     // the tile's rows of h are no longer needed
        }
      }
      if (!ok) *abort_flag = 1;
    }
  } else if (warp == MLP_O_WARP) {
    // ------------------------------------------------------------ MMA issuer of O += P W2_c^T (rank 0 only)
    if (rank == 0) {
      int slot = 0;
      uint32_t phase = 0;
      uint32_t unit = 0, unit_phase = 0, t = 0;
      bool ok = true;
      MlpGeo gc;
      gc.g = nullptr;
      for (int item = pair; item < total_items && ok; item += n_pairs, ++t) {
        mlp_geo(gc, groups, n_groups, item);
        const uint32_t idesc_o = make_idesc_pair(gc.n2);
        const int half = gc.n2 >> 1;
        for (int c = 0; c < gc.nc && ok; ++c) {
          // the first chunk overwrites O: the tile before must have been read out of it
          if (c == 0 && t > 0 && !mbar_wait<false>(bar(MB_O_EMPTY), (t - 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 47); break; }
          for (int j = 0; j < 2; ++j) {
            if (!mbar_wait<false>(bar(MB_P_FULL + unit), unit_phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 46); break; }
            tc_fence_after();
            if (!mbar_wait<false>(bar(MB_W_FULL + MLP_W1_SLOTS + slot), phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 48); break; }
            const uint64_t da = make_smem_desc(base + MLP_OFF_P + unit * A_BYTES);
#pragma unroll
            for (int k = 0; k < TC_BK / 16; ++k)
              for (int i = 0; i < gc.n2i; ++i) {
                const uint64_t db = make_smem_desc(base + MLP_OFF_W2 + slot * MLP_W2_BYTES + i * half * 128);
                mma_f16_pair_elect(tmem_base + (uint32_t)(i * gc.n2), da + (uint64_t)(k * 2), db + (uint64_t)(k * 2), idesc_o,
                                   (c > 0 || j > 0 || k > 0) ? 1u : 0u);
              }
            mma_commit_pair_elect(bar(MB_W_EMPTY + MLP_W1_SLOTS + slot));
            mma_commit_pair_elect(bar(MB_P_EMPTY + unit));
            if (++slot == MLP_W2_SLOTS) { slot = 0; phase ^= 1u; }
            if (++unit == MLP_P_UNITS) { unit = 0; unit_phase ^= 1u; }
          }
          if (!ok) break;
          if (c == gc.nc - 1) mma_commit_pair_elect(bar(MB_O_FULL));
        }
      }
      if (!ok) *abort_flag = 1;
    }
  } else {
    // ------------------------------------------------------------ epilogue warps (2..17 of both CTAs)
    pdl_begin(beside);
    const int ew = warp - 2;
    const int quarter = warp & 3;
    const int part = ew >> 2;
    const int row = quarter * 32 + lane;
    bool ok = true;
    uint32_t n_c = 0, t = 0;                  // chunks and tiles done by this warp
    const MlpGroup* g = nullptr;
    int g_start = 0, g_end = -1, nc = 0, d = 0, c_rows = 0;
    const bf16 *b1 = nullptr, *b2 = nullptr;
    const uint32_t s_taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(MLP_S_COL + part * 32);
    unsigned char* const prow0 = base_ptr + MLP_OFF_P + row * 128;
    uint32_t unit = part >> 1, unit_phase = 1;                // this warp's next unit of P: every other one, from its half of the chunk on
    const int piece0 = (part & 1) * 4, sw = row & 7;
    const uint32_t s_empty_r = mapa_shared(bar(MB_S_EMPTY), 0), p_full_r = mapa_shared(bar(MB_P_FULL), 0);   // (of unit 0)
    const uint32_t o_empty_r = mapa_shared(bar(MB_O_EMPTY), 0);
    for (int item = pair; item < total_items && ok; item += n_pairs, ++t) {
      if (item >= g_end || item < g_start) {
        g = groups + find_group_mlp(groups, n_groups, item);
        g_start = g->tile_start; g_end = g_start + g->tiles_m;
        nc = g->F / MLP_CHUNK; d = g->d; c_rows = g->c_rows; b1 = g->b1; b2 = g->b2;
        if (lane == 0) tensormap_acquire(&g->tmC);
      }
      for (int c = 0; c < nc && ok; ++c, ++n_c) {
        // this warp's 32 hidden columns of the chunk: every lane has all their bias values (requested before the wait; handed
        // around with shuffles they took a quarter of the loop's issue slots)
        uint4 bias[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) bias[j] = b1 != nullptr ? __ldg(reinterpret_cast<const uint4*>(b1 + c * MLP_CHUNK + part * 32) + j) : make_uint4(0u, 0u, 0u, 0u);
        if (!mbar_wait(bar(MB_S_FULL), n_c & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 50); break; }
        tc_fence_after();
        float v[32];
        {
          uint32_t r[32];
          tmem_ld32(s_taddr, r);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(s_empty_r);       // the next chunk's S may be issued
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          add_bias2(v[8 * j], v[8 * j + 1], bias[j].x);
          add_bias2(v[8 * j + 2], v[8 * j + 3], bias[j].y);
          add_bias2(v[8 * j + 4], v[8 * j + 5], bias[j].z);
          add_bias2(v[8 * j + 6], v[8 * j + 7], bias[j].w);
        }
#pragma unroll
        for (int j = 0; j < 32; j += 2) gelu_erf2(v[j], v[j + 1]);
        // the unit may still feed the second contraction of an earlier chunk; at a tile's first chunk P also was the
        // staging area of the final epilogue of the tile before, which every warp of this CTA must have left
        if (!mbar_wait(bar(MB_P_EMPTY + unit), unit_phase, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 51); break; }
        if (c == 0 && t > 0 && !mbar_wait(bar(MB_STAGE_FREE), (t - 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 52); break; }
        unsigned char* const prow = prow0 + unit * A_BYTES;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint4 o;
          o.x = pack2(v[8 * k], v[8 * k + 1]); o.y = pack2(v[8 * k + 2], v[8 * k + 3]);
          o.z = pack2(v[8 * k + 4], v[8 * k + 5]); o.w = pack2(v[8 * k + 6], v[8 * k + 7]);
          *reinterpret_cast<uint4*>(prow + (((piece0 + k) ^ sw) << 4)) = o;
        }
        fence_async_smem();                     // P must be visible to the tensor core's reads
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(p_full_r + 8u * unit);
        unit += 2;
        if (unit >= MLP_P_UNITS) { unit -= MLP_P_UNITS; unit_phase ^= 1u; }
      }
      if (!ok) break;
      // ---- the tile's output: O + b2 added to z, in boxes of 16 rows x 32 columns staged in P: the rows of a box are whole
      // 128-byte lines, which is what the reduction at L2 is fast with
      uint2 bias_reg = make_uint2(0u, 0u);
      const int n_out = (d >> 5) - part;                       // this warp's blocks of 32 columns: part, part + 4, ...
      if (b2 != nullptr && (lane >> 3) * 4 < n_out) bias_reg = __ldg(reinterpret_cast<const uint2*>(b2 + part * 32 + (lane >> 3) * 128 + (lane & 7) * 4));
      if (!mbar_wait(bar(MB_O_FULL), t & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 53); break; }
      tc_fence_after();
      const uint32_t o_taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * 32);
      unsigned char* const wst = base_ptr + MLP_OFF_P + ew * 2048;
      const int y0 = (item - g_start) * (2 * TC_BM) + rank * TC_BM + quarter * 32;
#pragma unroll 1
      for (int i = 0; i * 4 < n_out; ++i) {
        float v[32];
        {
          uint32_t r[32];
          tmem_ld32(o_taddr + (uint32_t)(i * 128), r);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
        }
        if ((i + 1) * 4 >= n_out) {                            // that was this warp's last read of O
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(o_empty_r);
        }
        if (b2 != nullptr) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) {
            const uint32_t w = __shfl_sync(0xffffffffu, (jj & 1) ? bias_reg.y : bias_reg.x, i * 8 + (jj >> 1));
            v[2 * jj] += __uint_as_float(w << 16);
            v[2 * jj + 1] += __uint_as_float(w & 0xffff0000u);
          }
        }
#pragma unroll
        for (int hr = 0; hr < 2; ++hr) {                       // rows 0 .. 15, then 16 .. 31
          if (lane == 0) bulk_wait_read0();                    // the box before has left the staging area
          __syncwarp();
          if (lane >> 4 == hr) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              *reinterpret_cast<float4*>(wst + (lane & 15) * 128 + ((k ^ (lane & 7)) << 4)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0 && y0 + hr * 16 < c_rows) {
            tma_reduce_add_2d(&g->tmC, smem_u32(wst), part * 32 + i * 128, y0 + hr * 16);
            bulk_commit();
          }
        }
      }
      if (n_out <= 0) { if (lane == 0) mbar_arrive_cluster(o_empty_r); }
      if (lane == 0) { bulk_wait_read0(); mbar_arrive(bar(MB_STAGE_FREE)); }   // this warp's boxes have left P
    }
    if (lane == 0) bulk_wait_done0();
    if (!ok) *abort_flag = 1;
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                        // neither CTA leaves while the other may still read its operands or signal it
  pdl_end(beside);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)TMEM_COLS) : "memory");
  }
}

}  // namespace

// Tile width of a GEMM whose row capacity is rows_cap and an estimate of the launch's time in microseconds (fixed when
// the model is placed, so a request's bits never depend on the batch it happens to share).
// The estimate: rounds of tiles over the SM pairs, a k-block per 0.285 us (bn 256; 0.26 at 192, 0.23 at 128) in each,
// and what a launch spends outside the main loop (10.4 / 9 / 7.9 us, half of it launch and set-up that a step hides).
// It follows the measured times of 256 to 1024 rows within 10 %: 3072 x 2048 at 512 rows 17.8 us with 256-wide tiles,
// 15.2 with 128-wide ones; 16384 x 2048 at 512 rows 35.0 and 43.1; 768 x 3072 at 768 rows 23.8 and 18.4.
// fp32-residual outputs leave in 16-column boxes, so their tiles may be 192 wide (48 columns per epilogue warp):
// N = 384 then fills two tiles exactly instead of wasting a quarter of two 256-wide ones.
double gemm_pair_config(long long rows_cap, int N, int K, int epi, int sm_count, int* bn) {
  const long long kblocks = (K + TC_BK - 1) / TC_BK, tiles_m = (rows_cap + 2 * TC_BM - 1) / (2 * TC_BM), pairs = sm_count / 2;
  const int widths[3] = {256, 192, 128};
  const double per_kb[3] = {0.285, 0.26, 0.23}, fixed[3] = {10.4, 9.0, 7.9};
  double best = 0;
  *bn = 0;
  for (int i = 0; i < 3; ++i) {
    if (widths[i] == 192 && (!(epi & EPI_RESID_F32) || N % 192)) continue;
    const long long tiles = tiles_m * ((N + widths[i] - 1) / widths[i]);
    const double t = fixed[i] + (double)((tiles + pairs - 1) / pairs) * kblocks * per_kb[i];
    if (*bn == 0 || t < best) { best = t; *bn = widths[i]; }
  }
  return best;
}

cudaError_t launch_gemm_tc_pair(const GemmGroup* groups, int n_groups, int total_items, int* status, int sm_count,
                                cudaStream_t st, int beside) {
  if (n_groups == 0 || total_items == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int pairs = total_items < sm_count / 2 ? total_items : sm_count / 2;
  return launch_pdl(gemm_tc_pair_kernel, dim3(2 * pairs), dim3(PAIR_THREADS), SMEM_BYTES, st, groups, n_groups, total_items, status, beside);
}

// The fused MLP kernel takes an encoder block when its accumulators fit the tensor memory (d <= 384 beside one
// 128-column chunk of S), the shapes tile evenly, and the model has more than one 128-row tile at capacity.
bool gemm_mlp_eligible(long long rows_cap, int d, int F) {
  return rows_cap > TC_BM && d >= 64 && d <= 384 && d % 64 == 0 && F >= 128 && F % 128 == 0;
}

cudaError_t launch_gemm_mlp_pair(const MlpGroup* groups, int n_groups, int total_items, int* status, int sm_count,
                                 cudaStream_t st, int beside) {
  if (n_groups == 0 || total_items == 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(gemm_mlp_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MLP_SMEM_BYTES);
  if (e != cudaSuccess) return e;
  const int pairs = total_items < sm_count / 2 ? total_items : sm_count / 2;
  return launch_pdl(gemm_mlp_pair_kernel, dim3(2 * pairs), dim3(MLP_THREADS), MLP_SMEM_BYTES, st, groups, n_groups, total_items, status, beside);
}

}  // namespace epara
