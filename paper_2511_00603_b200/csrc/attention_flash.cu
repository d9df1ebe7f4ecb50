// Attention of many query rows on the sm_100a tensor cores: encoder attention (bidirectional, head size 64, keys and
// values straight from the qkv matrix) and the causal attention of prompt chunks over the paged KV cache (head size 64
// or 128).
//
// One persistent CTA per SM walks over work items.  An item is one or two tiles of 128 query rows that see the same
// keys: two row tiles of an (image, head), or the same 128 tokens for two query heads of one kv head.  Keys are loaded in
// blocks of 128 and worked on in steps of 64.  Roles:
//   warp 8     TMA producer: the Q tiles, then K and V blocks through one ring (128-byte swizzle).  Paged: a box of 16
//              rows per page, page ids read from the block table a block ahead and checked against the pool (an id
//              outside it is reported and its box read from past the tensor, which fills it with zeros);
//   warp 9     issues S_g = Q_g K^T (M 128, N 64) into one of two buffers per tile, up to two steps ahead of P V and
//              across items, so that the softmax warps find their next scores waiting;
//   warps 10, 11  issue O_g += P_g V, g = 0 and 1, with P as the A operand from tensor memory and V consumed as the TMA
//              wrote it (MN-major B operand).  (An MMA costs its issuer some 60 cycles here and a step as much again in
//              waits and bookkeeping: one warp for all of them was the bound, 3350 cycles per step of two tiles.)
//   warps 0-3  softmax of tile 0, warps 4-7 of tile 1: one thread per query row (but see `HALF` below).  The thread reads its row of S once,
//              keeps it in registers for the maximum and the exponentials and writes P over S: 16 columns of S become 8
//              of P as bf16 and, for prompt chunks, 8 of the bf16 remainder (p = hi + lo up to 2^-17 relative; O then
//              takes two MMAs per step).  The running maximum is only raised, and O and the sum rescaled, when it has
//              grown by more than 2^8: until then the larger p only shift the exponent of O and of the sum.  Masked
//              column blocks of a warp cost nothing; rows past the live ones have no part in the decision to rescale,
//              so a row's bits depend on its own tile only.
// A tile's O and its sum are read out after its last step, normalised and turned through shared memory into whole lines.
// V rows past the last key may hold anything; they meet P columns that are zero, but 0 x NaN is NaN: the P V warps zero
// them before the P V of the last step.
//
// What bounds it: ex2.approx issues 16 per clock and SM, 1024 cycles for a step of two tiles (2 x 128 x 64 scores); the MMAs
// of those take some 450 cycles at head size 64 (550 with the remainder) and 930 at 128.  A softmax warp is one chain of
// latencies around its 512 cycles of exponentials: 100 to see its scores, 140 to read them, 250 for the maximum, 150 to hand
// P over and come around.  So a step is one straight piece of code (cut at every 16 columns it took 1250 cycles for the
// exponentials alone, now 700), and the two warps of a scheduler take turns at them: in step both waited for the
// special-function unit and then left it idle together (2450 cycles a step, now 1880; encoder 2000 and 1600).
//
// Launches with at most one query tile per SM (`HALF`): one tile per item, whose rows both groups of softmax warps share, 32
// columns of a step each; the two tell each other the row's maximum.  A tile's chain of steps, which is all the time such a
// launch takes, is that much shorter (512-token chunk after 1500 cached tokens, 1B decoder: 41 -> 34 us a layer; 509-token
// prompt 21 -> 17).  Two sums per row, one of either half's columns, keep the order of the additions, so that a row has the
// same bits in both forms.
//
// (Four prompts of 2048 tokens, 1B decoder: 467 us per layer on mma.sync, 223 with P in tensor memory, now 192.  Encoder,
// ViT-S, 203 images: 72 us, 58, now 53.  Event-bracketed.  Splitting a tile's keys between the two groups, with a merge at the
// end, shortened the small launches as much but doubled the copies of K and V, whose issue was then the bound: 240 us.)
// Every mbarrier wait is bounded: when one runs out the kernel records a code in *status, all roles leave their loops,
// tensor memory is freed and the kernel returns.
#include <climits>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace epara {

namespace {

using namespace tc;

constexpr int FL_TILE = FLASH_TILE;                   // query rows per tile, keys per block
constexpr int FL_SOFT_WARPS = 8;
constexpr int FL_LOAD_WARP = 8, FL_S_WARP = 9, FL_PV_WARP = 10;   // ... and 11
constexpr int FL_THREADS = 32 * 12;
constexpr int FL_HALF = FL_TILE * 128;                // 16 KB: 128 rows of 64 columns
constexpr float FL_RAISE = 8.0f;                      // log2 units the maximum may lag behind
constexpr int FL_BAR_BYTES = 512;
constexpr int FL_STEP = 64;                           // keys per step

template <int HD>
struct FlashGeo {
  static constexpr int NH = HD / 64;                  // 64-column halves of a row
  static constexpr int TILE_BYTES = FL_HALF * NH;
  static constexpr int STAGES = HD == 64 ? 8 : 4;
  static constexpr int OFF_KV = 2 * TILE_BYTES;
  static constexpr int OFF_OUT = OFF_KV + STAGES * TILE_BYTES;      // staging: 4 KB (32 rows of 128 bytes) per softmax warp
  static constexpr int OFF_BAR = OFF_OUT + FL_SOFT_WARPS * 4096;
  // (HALF: the second Q tile's place holds what the two warps of a row tell each other: [3][2][128] floats)
  static constexpr size_t SMEM = 1024 + OFF_BAR + FL_BAR_BYTES;
  static_assert(SMEM <= 227 * 1024, "shared memory of one SM");
};
// TMEM columns: S / P buffers 0, 1 of tile 0, of tile 1, then O_0, O_1
constexpr int FL_S_COL = 0, FL_O_COL = 256;

// S_FULL, P_READY, PV_DONE: one per tile and buffer (index 2 g + buffer), so that no barrier can complete two phases
// between two looks of its waiter (TURN: see the softmax warps).  K blocks sit in the even slots of the ring, V blocks in the odd ones, whose EMPTY
// barriers count both P V warps (one that has no tile in the item arrives without an MMA).
enum { FB_Q_FULL = 0, FB_Q_EMPTY, FB_S_FULL, FB_P_READY = FB_S_FULL + 4, FB_PV_DONE = FB_P_READY + 4, FB_KV_FULL = FB_PV_DONE + 4,
       FB_KV_EMPTY = FB_KV_FULL + 8, FB_TURN = FB_KV_EMPTY + 8, FB_PAIR = FB_TURN + 8, FB_COUNT = FB_PAIR + 4 };
static_assert(8 * FB_COUNT + 16 <= FL_BAR_BYTES, "barrier area");

__device__ __forceinline__ float fl_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// two fp32 operations per instruction
__device__ __forceinline__ uint64_t pack_f2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack_f2(uint64_t v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_f2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add_f2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// O (+)= P V with P (A operand) in tensor memory: one step of K = 16 (8 columns of packed bf16 pairs)
__device__ __forceinline__ void mma_ts_elect(uint32_t tmem_d, uint32_t tmem_a, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|q, 0xffffffff;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(tmem_d), "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) { tmem_st8(taddr, r); tmem_st8(taddr + 8, r + 8); }
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// V block as the B operand of P V: keys are the K dimension, the head's dims (N) are contiguous (MN-major).  Rows of 128
// bytes, 128-byte swizzle: groups of 8 keys 1024 bytes apart (stride offset), 64-dim halves 16 KB apart (leading offset).
__device__ __forceinline__ uint64_t make_smem_desc_v(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(FL_HALF >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// A work item.  Tile g has its rows at (qy + g * dy, qx + g * dx) of the qkv matrix, `live` of them real, and its output
// at the same row and column.
struct Work {
  int qx, qy, dx, dy;
  int n_mt, live0, live1;
  int n_keys;            // keys 0 .. n_keys - 1 are walked
  int lim0;              // last key row 0 of a tile may see (row r: lim0 + r); not causal: INT_MAX / 2
  int head;              // paged: first query head; else head
  const int32_t* table;  // paged
};

// What a role keeps of the group its items come from (descriptor reads are latency that a softmax warp cannot hide).
struct EncView {
  const AttnEncGroup* g;
  int start, end, H, T, q_blocks, G, mt;
};
struct PreView {
  const AttnPrefillGroup* g;
  int start, end, G, hd;
  int mt, head_shift, Hkv;
  unsigned by_hkv;
  const PrefillTile* tiles;
};
__device__ __forceinline__ void load_view(EncView& v, const AttnEncGroup* groups, int n_groups, int item, int mt) {
  if (v.g != nullptr && item >= v.start && item < v.end) return;
  int gi = 0;
  for (int i = 1; i < n_groups; ++i) if (item >= groups[i].blk_start) gi = i;
  const AttnEncGroup* g = groups + gi;
  v.g = g; v.mt = mt; v.start = g->blk_start; v.H = g->H; v.T = g->T; v.q_blocks = g->q_blocks; v.G = 1;
  v.end = v.start + g->B * g->H * g->q_blocks;
}
__device__ __forceinline__ void load_view(PreView& v, const AttnPrefillGroup* groups, int n_groups, int item, int mt) {
  if (v.g != nullptr && item >= v.start && item < v.end) return;
  int gi = 0;
  for (int i = 1; i < n_groups; ++i) if (item >= groups[i].item_start) gi = i;
  const AttnPrefillGroup* g = groups + gi;
  v.g = g; v.mt = mt; v.start = g->item_start; v.end = v.start + g->n_items; v.G = g->Hq / g->Hkv; v.hd = g->hd; v.tiles = g->tiles;
  v.head_shift = g->head_shift; v.Hkv = g->Hkv; v.by_hkv = g->by_hkv;
}
__device__ __forceinline__ Work get_work(const EncView& v, int item) {
  const int local = item - v.start, bh = v.q_blocks == 1 ? local : local / v.q_blocks, qb = local - bh * v.q_blocks;
  const int b = bh / v.H, h = bh - b * v.H, q0 = qb * v.mt * FL_TILE, left = v.T - q0;
  Work w;
  w.qx = h * 64; w.qy = b * v.T + q0; w.dx = 0; w.dy = FL_TILE;
  w.n_mt = min(v.mt, (left + FL_TILE - 1) / FL_TILE);
  w.live0 = min(FL_TILE, left); w.live1 = min(FL_TILE, left - FL_TILE);
  w.n_keys = v.T; w.lim0 = INT_MAX / 2;
  w.head = h; w.table = nullptr;
  return w;
}
__device__ __forceinline__ Work get_work(const PreView& v, int item) {
  const int local = item - v.start, kv_item = local >> v.head_shift;
  const int tile = v.by_hkv ? (int)__umulhi((unsigned)kv_item, v.by_hkv) : kv_item, kvh = kv_item - tile * v.Hkv;
  const int h = (local - (kv_item << v.head_shift)) * v.mt;                         // the first of n_mt heads of kv head kvh
  const PrefillTile pi = v.tiles[tile];
  Work w;
  w.head = kvh * v.G + h;
  w.qx = w.head * v.hd; w.qy = pi.row; w.dx = v.hd; w.dy = 0;
  w.n_mt = min(v.mt, v.G - h);
  w.live0 = w.live1 = pi.live;
  w.n_keys = pi.pos + pi.live;
  w.lim0 = pi.pos;
  w.table = pi.table;
  return w;
}
__device__ __forceinline__ const CUtensorMap* map_q(const AttnEncGroup* g) { return &g->tmQ; }
__device__ __forceinline__ const CUtensorMap* map_q(const AttnPrefillGroup* g) { return &g->maps->tmQ; }
__device__ __forceinline__ const CUtensorMap* map_kv(const AttnEncGroup* g) { return &g->tmQ; }
__device__ __forceinline__ const CUtensorMap* map_kv(const AttnPrefillGroup* g) { return &g->maps->tmKV; }
__device__ __forceinline__ int out_stride(const AttnEncGroup* g) { return g->H * 64; }
__device__ __forceinline__ int out_stride(const AttnPrefillGroup* g) { return g->Hq * g->hd; }

// Items of a CTA: one per round of the grid, every other round in reverse, so that a list sorted by length spreads evenly.
__device__ __forceinline__ int item_of_round(int round) {
  const int G = gridDim.x, i = blockIdx.x;
  return round * G + ((round & 1) ? G - 1 - i : i);
}

// The sequence of (item, step) that an MMA-issuing warp walks.
template <class View, class Group>
struct Cursor {
  const Group* groups;
  int n_groups, total_items, mt;
  View view;
  int round, n_mt, n_keys, step, steps;
  uint32_t first;                              // ring index of the item's K(0)
  bool valid;
  __device__ __forceinline__ void next_item() {
    first += (uint32_t)((steps + 1) >> 1) * 2;
    for (;; ++round) {
      valid = round * (int)gridDim.x < total_items;
      if (!valid) return;
      const int item = item_of_round(round);
      if (item >= total_items) continue;
      ++round;
      load_view(view, groups, n_groups, item, mt);
      const Work w = get_work(view, item);
      n_mt = w.n_mt; n_keys = w.n_keys; step = 0; steps = (n_keys + FL_STEP - 1) / FL_STEP;
      return;
    }
  }
  __device__ __forceinline__ void init(const Group* g, int ng, int total, int m) {
    groups = g; n_groups = ng; total_items = total; mt = m;
    view.g = nullptr; round = 0; steps = 0; first = 0;
    next_item();
  }
  __device__ __forceinline__ void advance() { if (++step == steps) next_item(); }
  __device__ __forceinline__ int keys() const { return min(FL_STEP, n_keys - step * FL_STEP); }
};

template <int HD, bool PAGED, bool HALF, class Group, class View>
__global__ void __launch_bounds__(FL_THREADS, 1)
attn_flash_kernel(const Group* __restrict__ groups, int n_groups, int total_items, int mt, int* __restrict__ status, int beside) {
  using Geo = FlashGeo<HD>;
  constexpr int ST = Geo::STAGES;
  constexpr bool SPLIT = PAGED;                  // P as head + remainder
  extern __shared__ unsigned char smem_dyn[];
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_dyn + (base - smem_u32(smem_dyn));
  const uint32_t bars = base + Geo::OFF_BAR;
  auto bar = [&](int i) { return bars + 8u * i; };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base_ptr + Geo::OFF_BAR + 8 * FB_COUNT);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(bar(FB_Q_FULL), 1); mbar_init(bar(FB_Q_EMPTY), 1);
    for (int i = 0; i < 4; ++i) { mbar_init(bar(FB_S_FULL + i), 1); mbar_init(bar(FB_P_READY + i), HALF ? 8 : 4); mbar_init(bar(FB_PV_DONE + i), 1); }
    for (int i = 0; i < 8; ++i) mbar_init(bar(FB_TURN + i), 1);
    for (int i = 0; i < 4; ++i) mbar_init(bar(FB_PAIR + i), 2);
    for (int s = 0; s < ST; ++s) { mbar_init(bar(FB_KV_FULL + s), 1); mbar_init(bar(FB_KV_EMPTY + s), 1 + (s & 1)); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == FL_S_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == FL_LOAD_WARP) {
    // ------------------------------------------------------------------ TMA producer
    bool ok = true;
    View view;
    view.g = nullptr;
    const Group* g_prev = nullptr;
    uint32_t kv = 0, it = 0;                     // ring tiles issued, items started
    bool waited = false;
    int Hkv = 0, kv_row0 = 0, oob = 0;           // (oob: a row past the tensor: filled with zeros)
    long long kv_pages = 0;
    const CUtensorMap *tmQ = nullptr, *tmKV = nullptr;
    for (int round = 0; ok; ++round) {
      const int item = item_of_round(round);
      if (round * (int)gridDim.x >= total_items) break;
      if (item >= total_items) continue;
      load_view(view, groups, n_groups, item, mt);
      const Work w = get_work(view, item);
      const Group* g = view.g;
      if (g != g_prev) {
        tmQ = map_q(g); tmKV = map_kv(g);
        tensormap_acquire(tmQ); tensormap_acquire(tmKV);
        g_prev = g;
        if constexpr (PAGED) { Hkv = g->Hkv; kv_pages = g->kv_pages; kv_row0 = g->kv_row0; oob = g->kv_rows; }
      }
      const int nblk = (w.n_keys + FL_TILE - 1) / FL_TILE;
      int page = 0, kvh = 0, kx = 0, vx = 0, ky = 0;
      if constexpr (PAGED) {
        page = (lane < 8 && lane * 16 < w.n_keys) ? w.table[lane] : 0;        // lanes 0 .. 7: page ids of the next block
        kvh = w.head / view.G;
      } else {
        kx = (view.H + w.head) * 64; vx = kx + view.H * 64;
        ky = (w.qy / view.T) * view.T;
      }
      if (!waited) { pdl_begin(beside); waited = true; }                 // q, k, v come from the kernels before this one
      for (int j = 0; j < nblk && ok; ++j) {
        const int n = min(FL_TILE, w.n_keys - j * FL_TILE), pages = (n + 15) >> 4;
        int yk = oob;
        if (PAGED) {
          if (lane < pages) {
            if (page >= 0 && page < kv_pages) yk = kv_row0 + (page * 2 * Hkv + kvh) * 16;
            else atomicExch(status, ERR_PAGE_ATTEND);
          }
          page = (lane < 8 && (j + 1) * FL_TILE + lane * 16 < w.n_keys) ? w.table[(j + 1) * 8 + lane] : 0;
          __syncwarp();
        }
        for (int kvi = 0; kvi < 2 && ok; ++kvi) {                 // K, then V
          const int slot = kv % ST;
          if (!mbar_wait<false>(bar(FB_KV_EMPTY + slot), ((kv / ST) & 1u) ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 12); break; }
          const uint32_t dst = base + Geo::OFF_KV + slot * Geo::TILE_BYTES;
          if (PAGED) {
            mbar_expect_tx_elect(bar(FB_KV_FULL + slot), (uint32_t)(pages * 2048 * Geo::NH));
            for (int p = 0; p < pages; ++p) {
              int y = __shfl_sync(0xffffffffu, yk, p);
              if (kvi && y != oob) y += Hkv * 16;
#pragma unroll
              for (int hh = 0; hh < Geo::NH; ++hh)
                tma_load_2d_elect(dst + hh * FL_HALF + p * 2048, tmKV, hh * 64, y, bar(FB_KV_FULL + slot));
            }
          } else {
            mbar_expect_tx_elect(bar(FB_KV_FULL + slot), (uint32_t)Geo::TILE_BYTES);
            tma_load_2d_elect(dst, tmKV, kvi ? vx : kx, ky + j * FL_TILE, bar(FB_KV_FULL + slot));
          }
          ++kv;
          if (j == 0 && kvi == 0) {
            // Q: free once the last S of the item before is complete
            if (!mbar_wait<false>(bar(FB_Q_EMPTY), (it & 1u) ^ 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 11); break; }
            mbar_expect_tx_elect(bar(FB_Q_FULL), (uint32_t)(w.n_mt * Geo::TILE_BYTES));
            for (int gg = 0; gg < w.n_mt; ++gg)
#pragma unroll
              for (int hh = 0; hh < Geo::NH; ++hh)
                tma_load_2d_elect(base + gg * Geo::TILE_BYTES + hh * FL_HALF, tmQ, w.qx + gg * w.dx + hh * 64, w.qy + gg * w.dy, bar(FB_Q_FULL));
          }
        }
      }
      ++it;
    }
    if (!waited) pdl_begin(beside);
    if (!ok) { *abort_flag = 1; drain_sleep(200000ull); }
  } else if (warp == FL_S_WARP) {
    // ------------------------------------------------------------------ issuer of S
    bool ok = true;
    uint32_t cnt0 = 0, cnt1 = 0;                 // S issued so far, per tile
    uint32_t it = 0;                             // items started
    Cursor<View, Group> c;
    c.init(groups, n_groups, total_items, mt);
    for (; c.valid && ok; c.advance()) {
      const bool last = c.step + 1 == c.steps;
      const uint32_t ik = c.first + (c.step & ~1), slot = ik % ST;
      if (c.step == 0) {
        if (!mbar_wait<false>(bar(FB_Q_FULL), it & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 14); break; }
        ++it;
      }
      if (!(c.step & 1) && !mbar_wait<false>(bar(FB_KV_FULL + slot), (ik / ST) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 13); break; }
      const uint32_t idesc = make_idesc((c.keys() + 15) & ~15);
      const uint64_t dk = make_smem_desc(base + Geo::OFF_KV + slot * Geo::TILE_BYTES + (c.step & 1) * (FL_STEP * 128));
#pragma unroll
      for (int g = 0; g < 2; ++g) {
        if (g >= c.n_mt) break;
        uint32_t& cnt = g ? cnt1 : cnt0;
        const uint32_t b = cnt & 1u;
        // the buffer holds P until the P V of two steps ago is complete
        if (cnt >= 2 && !mbar_wait<false>(bar(FB_PV_DONE + 2 * g + b), ((cnt >> 1) - 1u) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 20); break; }
        ++cnt;
        tc_fence_after();
        const uint64_t dq = make_smem_desc(base + g * Geo::TILE_BYTES);
        const uint32_t d = tmem_base + FL_S_COL + g * 128 + b * 64;
#pragma unroll
        for (int k = 0; k < HD / 16; ++k) {
          const uint64_t o = (uint64_t)((k >> 2) * (FL_HALF >> 4) + (k & 3) * 2);
          mma_f16_elect(d, dq + o, dk + o, idesc, k > 0 ? 1u : 0u);
        }
        mma_commit_elect(bar(FB_S_FULL + 2 * g + b));
      }
      if (!ok) break;
      if (last || (c.step & 1)) mma_commit_elect(bar(FB_KV_EMPTY + slot));      // K back at a block's last step ...
      if (last) mma_commit_elect(bar(FB_Q_EMPTY));                              // ... Q at the item's
    }
    if (!ok) *abort_flag = 1;
    pdl_begin(beside);
  } else if (warp >= FL_PV_WARP) {
    // ------------------------------------------------------------------ issuers of O_g += P_g V
    const int g = warp - FL_PV_WARP;
    bool ok = true;
    uint32_t cnt = 0;                            // P V issued so far
    const uint32_t idesc_o = make_idesc(HD) | (1u << 16);                  // B operand MN-major
    const uint32_t d = tmem_base + FL_O_COL + g * HD;
    Cursor<View, Group> c;
    c.init(groups, n_groups, total_items, mt);
    for (; c.valid && ok; c.advance()) {
      const bool last = c.step + 1 == c.steps, done = last || (c.step & 1);   // `done`: the V block's last step
      const uint32_t iv = c.first + (c.step & ~1) + 1, slot = iv % ST;
      const bool mine = g < c.n_mt;
      if ((mine ? !(c.step & 1) : done) && !mbar_wait<false>(bar(FB_KV_FULL + slot), (iv / ST) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 21); break; }
      if (!mine) {
        if (done && lane == 0) mbar_arrive(bar(FB_KV_EMPTY + slot));
        continue;
      }
      const int n = c.keys(), ksteps = (n + 15) >> 4;
      const uint32_t v_off = Geo::OFF_KV + slot * Geo::TILE_BYTES + (c.step & 1) * (FL_STEP * 128);
      if (n & 15) {
        // V rows n .. up to the next multiple of 16 (with two tiles both warps write the same zeros)
        unsigned char* const v0 = base_ptr + v_off + n * 128;
        for (int i = lane; i < (16 - (n & 15)) * 8; i += 32)
#pragma unroll
          for (int hh = 0; hh < Geo::NH; ++hh) *reinterpret_cast<uint4*>(v0 + hh * FL_HALF + i * 16) = make_uint4(0u, 0u, 0u, 0u);
        fence_async_smem();
        __syncwarp();
      }
      const uint32_t b = cnt & 1u;
      if (!mbar_wait<false>(bar(FB_P_READY + 2 * g + b), (cnt >> 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 15); break; }
      ++cnt;
      tc_fence_after();
      const uint32_t p = tmem_base + FL_S_COL + g * 128 + b * 64;
      const uint64_t dv = make_smem_desc_v(base + v_off);
#pragma unroll
      for (int k = 0; k < FL_STEP / 16; ++k) {
        if (k >= ksteps) break;
        mma_ts_elect(d, p + k * 16, dv + (uint64_t)(k * 128), idesc_o, (c.step > 0 || k > 0) ? 1u : 0u);   // 16 keys = 2 KB
        if (SPLIT) mma_ts_elect(d, p + k * 16 + 8, dv + (uint64_t)(k * 128), idesc_o, 1u);
      }
      mma_commit_elect(bar(FB_PV_DONE + 2 * g + b));
      if (done) mma_commit_elect(bar(FB_KV_EMPTY + slot));
    }
    if (!ok) *abort_flag = 1;
    pdl_begin(beside);
  } else {
    // ------------------------------------------------------------------ softmax (warps 0 .. 7)
    pdl_begin(beside);
    // (HALF: warps w and w + 4 share the rows of the one tile, 32 of a step's 64 columns each)
    const int half = HALF ? warp >> 2 : 0, g = HALF ? 0 : warp >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    constexpr int NC = HALF ? FL_STEP / 2 : FL_STEP;                // columns of a step that this warp works on
    float* const told = reinterpret_cast<float*>(base_ptr + Geo::TILE_BYTES) + row;   // [slot][half][128 rows]
    const float scale = 1.4426950408889634f * (HD == 64 ? 0.125f : 0.08838834764831845f);   // log2(e) / sqrt(HD)
    const uint64_t scale2 = pack_f2(scale, scale);
    const uint32_t lane_base = tmem_base + ((uint32_t)(quarter * 32) << 16);
    const uint32_t s_addr = lane_base + FL_S_COL + g * 128, o_addr = lane_base + FL_O_COL + g * HD;
    unsigned char* const stage = base_ptr + Geo::OFF_OUT + warp * 4096;
    bool ok = true;
    uint32_t cnt = 0;                            // steps of this tile done
    uint32_t turns = 0, pairs = 0;               // turns and pair barriers waited for
    bool turns_seen = false;                     // the first turn of this CTA's paired items is past
    View view;
    view.g = nullptr;
    // this tile's next item; decoded while the last P V of the item before is under way
    int round = 0;
    Work next;
    const Group* next_g = nullptr;
    auto find_next = [&]() {
      for (; round * (int)gridDim.x < total_items; ++round) {
        const int item = item_of_round(round);
        if (item >= total_items) continue;
        load_view(view, groups, n_groups, item, mt);
        next = get_work(view, item);
        if (g < next.n_mt) { ++round; next_g = view.g; return true; }
      }
      return false;
    };
    // What the other half's warp knows of the row: the larger maximum, or the sum of the halves in column order.
    auto tell = [&](int slot, float mine, float& other) {
      told[(slot * 2 + half) * FL_TILE] = mine;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(FB_PAIR + quarter));
      if (!mbar_wait<false>(bar(FB_PAIR + quarter), pairs & 1u, abort_flag)) { if (lane == 0) atomicExch(status, 22); return false; }
      ++pairs;
      other = told[(slot * 2 + (half ^ 1)) * FL_TILE];
      return true;
    };
    bool more = find_next();
    while (ok && more) {
      const Work w = next;
      const Group* const wg = next_g;
      const int steps = (w.n_keys + FL_STEP - 1) / FL_STEP;
      const int live = g ? w.live1 : w.live0;
      const bool warp_live = quarter * 32 < live;
      const bool row_live = row < live;
      const int lim = min(w.lim0 + min(row, live - 1), w.n_keys - 1);                        // last key of this row
      const int warp_first = min(w.lim0 + quarter * 32, w.n_keys - 1);                       // ... of the warp's first row
      const int warp_last = min(w.lim0 + min(quarter * 32 + 31, live - 1), w.n_keys - 1);    // ... and of its last
      // the warp of the other tile on this scheduler has as many steps: the two take turns
      const bool paired = !HALF && w.n_mt == 2 && quarter * 32 < min(w.live0, w.live1);
      float m_ref = 0.f, l[2] = {0.f, 0.f};      // sums of a step's first and second half of the columns
      for (int j = 0; j < steps; ++j) {
        const uint32_t b = cnt & 1u, sb = s_addr + b * 64;
        if (!mbar_wait<false>(bar(FB_S_FULL + 2 * g + b), (cnt >> 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 16); break; }
        tc_fence_after();
        const int k0 = j * FL_STEP;
        // Columns that no row of the warp sees (the upper triangle of a prompt chunk): P is zero and nothing else changes.
        const bool seen = warp_live && k0 <= warp_last;
        if (warp_live && !seen) {
          const uint32_t z[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll
          for (int c = 0; c < NC; c += 8) tmem_st8(sb + half * NC + c, z);
          tmem_st_wait();
        }
        // The two warps of a scheduler take turns at the exponentials, so that one's scores are read and reduced while the
        // other keeps the special-function unit busy (in step they left it idle half of the time).
        // (Strictly in turn, over the ends of items too: only the very first turn of tile 0 is not given to it.  Neither warp
        // can be more than one turn ahead, so a TURN barrier never completes two phases between two looks of its waiter.)
        const bool take_turns = paired && (g == 1 || turns_seen);
        turns_seen |= paired;
        if (seen) {
          uint32_t v[NC];
          tmem_ld32_nowait(sb + half * NC, v);
          if (!HALF) tmem_ld32_nowait(sb + 32, v + NC - 32);
          tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < NC / 16; ++c) tmem_regs_ready16(v + 16 * c);
          if (k0 + FL_STEP - 1 > warp_first) {                      // some row's limit lies in this step or before it
#pragma unroll
            for (int i = 0; i < NC; ++i) if (k0 + half * NC + i > lim) v[i] = 0xff800000u;
          }
          float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
          for (int i = 0; i < NC; i += 8) {
            mx0 = max3(mx0, __uint_as_float(v[i]), __uint_as_float(v[i + 1]));
            mx1 = max3(mx1, __uint_as_float(v[i + 2]), __uint_as_float(v[i + 3]));
            mx2 = max3(mx2, __uint_as_float(v[i + 4]), __uint_as_float(v[i + 5]));
            mx3 = max3(mx3, __uint_as_float(v[i + 6]), __uint_as_float(v[i + 7]));
          }
          float mx = fmaxf(max3(mx0, mx1, mx2), mx3);
          if (HALF) {
            float other;
            if (!tell(j & 1, mx, other)) { ok = false; break; }
            mx = fmaxf(mx, other);
          }
          if (j == 0) {
            m_ref = mx;                                             // (key 0 is in every row's reach)
          } else {
            const float m_new = fmaxf(m_ref, mx);
            if (__any_sync(0xffffffffu, row_live && (m_new - m_ref) * scale > FL_RAISE)) {
              const float f = fl_ex2((m_ref - m_new) * scale);
              m_ref = m_new;
              l[0] *= f;
              l[1] *= f;
              // every P V up to the step before must be complete
              if (!mbar_wait<false>(bar(FB_PV_DONE + 2 * g + (b ^ 1u)), ((cnt - 1u) >> 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 17); break; }
              tc_fence_after();
#pragma unroll 1
              for (int c = half * (HD / 2); c < (HALF ? (half + 1) * (HD / 2) : HD); c += 16) {
                uint32_t o[16];
                tmem_ld16(o_addr + c, o);
#pragma unroll
                for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
                tmem_st16(o_addr + c, o);
              }
            }
          }
          const float nms = -m_ref * scale;
          const uint64_t nms2 = pack_f2(nms, nms), minus1 = pack_f2(-1.f, -1.f);
          if (take_turns) {
            if (!mbar_wait<false>(bar(FB_TURN + 4 * g + quarter), turns & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 19); break; }
            ++turns;
          }
          // p = 2^(s * scale - m * scale), its sum and its bf16 parts; one straight piece of code, so that the exponentials of
          // a block of 16 columns run under the conversions of the block before
#pragma unroll
          for (int h = 0; h < NC / 32; ++h) {
            uint64_t l2a = 0, l2b = 0;
#pragma unroll
            for (int c = 2 * h; c < 2 * h + 2; ++c) {
              const uint32_t* const vc = v + 16 * c;
              uint32_t hi[8], lo[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                float x, y;
                unpack_f2(fma_f2(pack_f2(__uint_as_float(vc[2 * i]), __uint_as_float(vc[2 * i + 1])), scale2, nms2), x, y);
                x = fl_ex2(x);
                y = fl_ex2(y);
                const uint64_t p2 = pack_f2(x, y);
                if (i & 1) l2b = add_f2(l2b, p2); else l2a = add_f2(l2a, p2);
                hi[i] = pack2(x, y);
                if (SPLIT) {
                  float rx, ry;
                  unpack_f2(fma_f2(pack_f2(__uint_as_float(hi[i] << 16), __uint_as_float(hi[i] & 0xffff0000u)), minus1, p2), rx, ry);
                  lo[i] = pack2(rx, ry);
                }
              }
              tmem_st8(sb + half * NC + 16 * c, hi);
              if (SPLIT) tmem_st8(sb + half * NC + 16 * c + 8, lo);
            }
            float a0, a1, a2, a3;
            unpack_f2(l2a, a0, a1);
            unpack_f2(l2b, a2, a3);
            l[h] += (a0 + a1) + (a2 + a3);
          }
          if (paired && lane == 0) mbar_arrive(bar(FB_TURN + 4 * (g ^ 1) + quarter));
          tmem_st_wait();
        } else if (paired) {
          if (take_turns) {
            if (!mbar_wait<false>(bar(FB_TURN + 4 * g + quarter), turns & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 19); break; }
            ++turns;
          }
          if (lane == 0) mbar_arrive(bar(FB_TURN + 4 * (g ^ 1) + quarter));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(FB_P_READY + 2 * g + b));
        ++cnt;
      }
      if (!ok) break;
      // ---- the tile's output: rows through this warp's staging area, then whole 128-byte lines
      const int oy = w.qy + g * w.dy + quarter * 32, ox = w.qx + g * w.dx;
      bf16* const out = wg->out;
      const int ostride = out_stride(wg);
      more = find_next();
      if (!warp_live) continue;
      float sum = l[0] + l[1];
      if (HALF) {
        float other;
        if (!tell(2, l[0], other)) { ok = false; break; }
        sum = l[0] + other;
      }
      const float inv = 1.0f / sum;
      if (!mbar_wait<false>(bar(FB_PV_DONE + 2 * g + ((cnt - 1u) & 1u)), ((cnt - 1u) >> 1) & 1u, abort_flag)) { ok = false; if (lane == 0) atomicExch(status, 18); break; }
      tc_fence_after();
      constexpr int EC = HALF && HD == 64 ? 32 : 64, PIECES = EC / 8;        // columns at a time, their 16-byte pieces
      const int c_end = HALF ? (half + 1) * (HD / 2) : HD;
#pragma unroll 1
      for (int c = half * (HD / 2); c < c_end; c += EC) {
        uint32_t o[EC];
        tmem_ld32_nowait(o_addr + c, o);
        if (EC == 64) tmem_ld32_nowait(o_addr + c + 32, o + EC - 32);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < EC / 16; ++i) tmem_regs_ready16(o + 16 * i);
        auto place = [&](int r, int k) { return stage + r * (EC * 2) + ((k ^ (EC == 64 ? r & 7 : (r >> 1) & 3)) << 4); };
#pragma unroll
        for (int k = 0; k < PIECES; ++k) {
          uint4 u;
          u.x = pack2(__uint_as_float(o[8 * k]) * inv, __uint_as_float(o[8 * k + 1]) * inv);
          u.y = pack2(__uint_as_float(o[8 * k + 2]) * inv, __uint_as_float(o[8 * k + 3]) * inv);
          u.z = pack2(__uint_as_float(o[8 * k + 4]) * inv, __uint_as_float(o[8 * k + 5]) * inv);
          u.w = pack2(__uint_as_float(o[8 * k + 6]) * inv, __uint_as_float(o[8 * k + 7]) * inv);
          *reinterpret_cast<uint4*>(place(lane, k)) = u;
        }
        __syncwarp();
        const int piece = lane % PIECES;
#pragma unroll
        for (int i = 0; i < PIECES; ++i) {
          const int r = i * (32 / PIECES) + lane / PIECES;
          if (quarter * 32 + r < live)
            *reinterpret_cast<uint4*>(out + (size_t)(oy + r) * ostride + ox + c + piece * 8) = *reinterpret_cast<const uint4*>(place(r, piece));
        }
        __syncwarp();
      }
      tc_fence_before();                         // (O has been read: the next item's P V may overwrite it once P is reported)
    }
    if (!ok) *abort_flag = 1;
  }
  tc_fence_before();
  __syncthreads();
  pdl_end(beside);
  if (warp == FL_S_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

template <int HD, bool PAGED, bool HALF, class Group, class View>
cudaError_t launch_flash_as(const Group* groups, int n_groups, int total_items, int mt, int* status, int sm_count, cudaStream_t st, int beside) {
  const auto kernel = attn_flash_kernel<HD, PAGED, HALF, Group, View>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FlashGeo<HD>::SMEM);
  if (e != cudaSuccess) return e;
  const int grid = total_items < sm_count ? total_items : sm_count;
  return launch_pdl(kernel, dim3(grid), dim3(FL_THREADS), FlashGeo<HD>::SMEM, st, groups, n_groups, total_items, mt, status, beside);
}

template <int HD, bool PAGED, class Group, class View>
cudaError_t launch_flash(const Group* groups, int n_groups, int total_items, int mt, int* status, int sm_count, cudaStream_t st, int beside) {
  if (n_groups == 0 || total_items == 0) return cudaSuccess;
  return mt == 1 ? launch_flash_as<HD, PAGED, true, Group, View>(groups, n_groups, total_items, mt, status, sm_count, st, beside)
                 : launch_flash_as<HD, PAGED, false, Group, View>(groups, n_groups, total_items, mt, status, sm_count, st, beside);
}

}  // namespace

cudaError_t launch_attn_encoder_tc(const AttnEncGroup* groups, int n_groups, int total_items, int mt, int* status, int sm_count,
                                   cudaStream_t st, int beside) {
  return launch_flash<64, false, AttnEncGroup, EncView>(groups, n_groups, total_items, mt, status, sm_count, st, beside);
}

cudaError_t launch_attn_prefill(const AttnPrefillGroup* groups, int n_groups, int total_items, int mt, int hd, int* status,
                                int sm_count, cudaStream_t st, int beside) {
  if (hd == 64) return launch_flash<64, true, AttnPrefillGroup, PreView>(groups, n_groups, total_items, mt, status, sm_count, st, beside);
  if (hd == 128) return launch_flash<128, true, AttnPrefillGroup, PreView>(groups, n_groups, total_items, mt, status, sm_count, st, beside);
  return cudaErrorInvalidValue;
}

}  // namespace epara
