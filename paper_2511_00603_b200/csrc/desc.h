// Device-visible descriptors written by the host step planner and read by the kernels.
// One step uploads one blob holding the request table and, per launch, an array of groups
// (one group = one model's problem in that launch).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace epara {

typedef __nv_bfloat16 bf16;

enum : int { EPI_BIAS = 1, EPI_GELU = 2, EPI_SWIGLU = 4, EPI_RESID_F32 = 8 };

// Codes a kernel leaves in the step's device status word (0 = none).  1..59 are bounded waits that ran
// out (the role that gave up); the others are indices found out of range, whose access was skipped.
enum : int { ERR_PAGE_APPEND = 101, ERR_PAGE_ATTEND = 102, ERR_SELFTEST_WAIT = 90, ERR_SELFTEST_SPLIT = 91 };

// Per admitted request (model order, then batch order).
struct ReqDesc {
  const void* input;     // MLP row / ViT image
  const int32_t* table;  // decoder block table
  void* out_logits;
  int32_t* out_argmax;
  int token;             // decoder, single-token request: the token being decoded
  int kv_len;            // cached tokens before this step
  int n_blocks;
  int row_start;         // decoder: first activation row of the request (a prompt chunk takes n_tok rows)
  int n_tok;             // decoder: tokens of the request in this step (1 = decode, > 1 = prompt chunk)
  int pad[3];
};

// Decoder activations have one row per token.  Row r belongs to request `req`, sits at position `pos` of
// its sequence and holds token id `token`.
struct RowDesc {
  int req2;              // 2 * req, + 1 for the only row of a decode request (a prompt chunk's rows: + 0)
  int pos, token;
#ifdef __CUDACC__
  __host__ __device__
#endif
  int req() const { return req2 >> 1; }
#ifdef __CUDACC__
  __host__ __device__
#endif
  bool single() const { return req2 & 1; }
};

// Descriptors that hold TMA maps start on 128 bytes, a map's size.  (64 is all a map needs, but one that lies across two lines is
// slower to fetch: the 65 GEMM launches of a step of 128 requests through the 1B decoder 1310 us between events, 1306 like
// this.)
constexpr int TMAP_ALIGN = 128;

// C = epi(A W^T + bias).  tmA/tmW are the TMA maps of A [rows, K] and W [N, K] (K innermost,
// 128-byte swizzle, 64 columns x the rows a CTA loads of each).
struct alignas(TMAP_ALIGN) GemmGroup {
  CUtensorMap tmA;
  CUtensorMap tmW;
  CUtensorMap tmC;   // swapped operands on pairs: A again, in boxes for a tile's second MMA (their output leaves by plain stores).
                     // Tile pairs: the output, written by TMA from the epilogue's staging rows: bf16 [rows, N] with a
                     // 32 x 32 box (SwiGLU: [rows, N/2], 16 x 32), or fp32 [rows, N] with a 16 x 32 box
                     // for the residual update (TMA reduce-add)
  const bf16* A;
  const bf16* W;
  void* C;
  const bf16* bias;
  int M, N, K;
  int lda, ldw, ldc;
  int epi;
  int tile_start;  // first work item of this group in the launch
  int tiles_m, tiles_n;
  int bn, ksplit;  // tile pairs: bn = tile width; swapped operands: bn = batch rows of a tile, ksplit = k ranges
  int c_rows;      // row extent of tmC (rows at and beyond it are never written)
  int stream;      // 1: weight-streaming kernel (at most 16 rows ever, or a small matrix; 16 W rows per
                   // block, tiles_n = ceil(N / 16), no TMA maps); 2: 256-row tiles on CTA pairs (tiles_m counts 256-row
                   // tiles and tmW's box holds bn / 2 rows); 3: swapped operands (tmA's box holds bn rows, tmW's
                   // 128); 5: swapped operands on CTA pairs (see kernels.h); 0: plain CUDA-core comparator
  const ReqDesc* reqs;   // weight-streaming kernel: when set, row m of A is request m's input (an MLP's first layer)
  int m_base, n_base;    // tile pairs: first row and column of the group's first tile
  int pad[2];
};

enum : int { NORM_LN = 0, NORM_RMS = 1 };
struct NormGroup {
  const float* x;        // fp32 [M rows, row stride x_stride]
  bf16* y;               // bf16 [M, d]
  const bf16* gamma;
  const bf16* beta;      // LN only
  const int* row_index;  // when set, output row m reads input row row_index[m] (a decoder's last-token rows)
  long long x_stride;
  int M, d, kind;
  float eps;
};

struct AttnReq {
  const int32_t* table;
  int len;               // tokens to attend (cached + appended)
  int row;               // activation row of the request's token (q is read and the output written there)
};

// A cache page that a decode request of the step appends to, at position `pos`, from token row `row`.
struct WrittenPage {
  const int32_t* id;     // where the caller's block table holds the page's id
  int pos, row;
};

// LINK: finds the decode requests that attend to tokens which other requests of the step append (see AttnDecGroup::linked).
enum : int { GATHER_ROWS = 0, GATHER_EMB = 1, GATHER_PATCH = 2, GATHER_LINK = 3 };
struct GatherGroup {
  const ReqDesc* reqs;
  const RowDesc* rows;   // EMB: one entry per output row
  const AttnReq* areqs;  // LINK: the decode requests, one block each
  const WrittenPage* written;   // LINK: the decode requests' pages, in their order; B counts them
  void* out;             // ROWS: bf16 [B, ld]; EMB: fp32 [rows, d]; PATCH: bf16 [B*np, 3*p*p]; LINK: int [decode requests]
  const bf16* emb;       // EMB
  int kind, B, width, ld;
  int img, patch;
  int blocks;            // blocks this group needs
  int pad;
};

struct RopeGroup {
  bf16* qkv;             // [rows, (Hq+2Hkv)*hd], q rotated in place
  bf16* kv_layer;        // [pages][2][Hkv][16][hd]
  const ReqDesc* reqs;
  const RowDesc* rows;   // one entry per token row; B counts rows
  const float2* cs;      // [max position + 1][hd/2]: (cos, sin) of position * 10000^(-2j/hd)
  int* status;           // device word: set to ERR_PAGE_APPEND when a block table names a page outside the pool
  long long kv_pages;    // pages of the pool; a page id outside [0, kv_pages) is reported, its write skipped
  int B, Hq, Hkv, hd;
  int only_chunks;       // 1: decode rows are left alone (the attention kernel rotates and appends them itself)
  int pad;
};

// Causal attention of prompt chunks (one layer): a request has n_tok query tokens in consecutive rows, token t at position
// kv_len + t attends to positions 0 .. kv_len + t of its paged cache (the chunk's own k, v were appended by the kernel
// before).  A work item is 128 of its tokens (a tile) and one or two query heads of one kv head; the list holds one entry per
// tile, sorted by the keys it walks, longest first, and a tile's heads are items one after another.  (With an entry per item
// 3900 chunks of two tokens on a model of 32 heads overflowed the step's blob.)
struct PrefillTile {
  const int32_t* table;
  int row, live;         // first activation row, tokens of the tile
  int pos;               // position of the tile's first token
  int pad;
};
// One per model and step; the layers' groups point to it.
struct alignas(TMAP_ALIGN) PrefillMaps {
  CUtensorMap tmQ;       // qkv [rows, (Hq+2Hkv)*hd] bf16, box 64 columns x 128 rows, 128-byte swizzle
  CUtensorMap tmKV;      // the cache as [n_layers * kv_pages * 2 * Hkv * 16, hd], box 64 columns x 16 rows
};
struct AttnPrefillGroup {
  const PrefillMaps* maps;
  const PrefillTile* tiles;
  bf16* out;             // [rows, Hq*hd]
  long long kv_pages;
  int kv_row0, kv_rows;  // this layer's first row of tmKV, rows of tmKV (a box from there on arrives as zeros)
  int n_items, Hq, Hkv, hd;
  int item_start;        // first item of this group in the launch
  int head_shift;        // items of one kv head of a tile, as a power of two: its query heads by the query tiles of an item
  unsigned by_hkv;       // 2^32 / Hkv rounded up (0 for Hkv = 1): items to tiles without a division, which every role of the
                         // kernel would wait for at the start of an item (exact while items x Hkv < 2^32)
  int pad;
};

struct AttnDecGroup {
  const bf16* q;         // [B, q_stride], head h at column h*hd
  bf16* kv_layer;
  const AttnReq* reqs;
  const float2* cs;      // set: row b of q is followed by k and v (qkv), neither rotated nor appended yet; the kernel does
                         // both for position len - 1 (RopeGroup::cs).  Null: q is rotated and the cache complete.
  bf16* out;             // [B, Hq*hd]
  float* partial;        // [B][Hq][max_chunks][hd + 2]  (m, l, o[hd]); requests of more than one chunk
  int* counters;         // [B][Hkv] chunks that have arrived; zero between launches
  int q_stride;
  int B, Hq, Hkv, hd;
  int max_chunks;
  int req_start;         // first grid.z index of this group
  int reqs_stable;       // 1: `reqs` was uploaded before the step's first kernel (a block past a request's
                         // length may leave without the dependency wait); 0: an earlier kernel writes it
  int* status;           // device word: set to ERR_PAGE_ATTEND when a block table names a page outside the pool
  long long kv_pages;    // pages of the pool; a page id outside [0, kv_pages) is reported and read as absent
  // With cs, in a step of several requests: linked[b] != 0 when request b may attend to tokens that other rows of the
  // step append (requests of one sequence in one step).  The block takes those from qkv then, wherever the append stands.
  const int* linked;     // null: a single request
  const WrittenPage* written;
  int n_written;
  int pad;
};

struct alignas(TMAP_ALIGN) AttnEncGroup {
  CUtensorMap tmQ;       // tensor-core kernel: qkv [rows, 3d] bf16, box 64 columns x 128 rows, 128-byte swizzle (K and V blocks too)
  const bf16* qkv;       // [B*T, 3d]: q | k | v, head h at column h*hd within each
  bf16* out;             // [B*T, d]
  int B, T, H, hd;
  int blk_start;         // first block (item) of this group
  int q_blocks;          // query blocks per (image, head)
  int tc;                // 1: runs in the tensor-core kernel, fixed when the model is placed
};

// One transformer MLP block of an encoder as a single work unit of the fused kernel:
// z += GELU(h W1^T + b1) W2^T + b2 with h bf16 [rows, d], W1 [F, d], W2 [d, F], z fp32 [rows, d].
// d is a multiple of 64 and at most 384 (the output accumulator of a 128-row tile must fit the tensor memory
// beside one 128-column chunk of the hidden layer), F a multiple of 128.
struct alignas(TMAP_ALIGN) MlpGroup {
  CUtensorMap tmX;       // h [rows, d] bf16, box 64 columns x 128 rows, 128-byte swizzle
  CUtensorMap tmW1;      // W1 [F, d] bf16, box 64 x 64 rows (one CTA of a pair loads half of a chunk's 128 rows)
  CUtensorMap tmW2;      // W2 [d, F] bf16, box 64 x n2/2 rows (n2 = d, or d / 2 when d > 256: two MMAs per k step)
  CUtensorMap tmC;       // z [rows, d] fp32, box 32 columns x 16 rows, 128-byte swizzle (TMA reduce-add of the epilogue)
  const bf16* b1;        // [F] or null
  const bf16* b2;        // [d] or null
  int M, d, F;
  int tile_start;        // first work item (256-row tile) of this group in the launch
  int tiles_m;
  int c_rows;            // row extent of tmC
  int pad[8];
};

struct AssembleGroup {   // z[b, 0] = cls + pos[0]; z[b, 1+p] = E[b*np + p] + pos[1+p]
  const bf16* E;
  const bf16* cls;
  const bf16* pos;
  float* z;
  int B, T, d, pad;
};

struct OutputGroup {     // copy logits rows to the requests' buffers and take the argmax
  const bf16* logits;    // [B, ld]
  const ReqDesc* reqs;
  int B, N, ld, pad;
};

}  // namespace epara

// Group arrays are packed back to back in the step blob: sizes must keep 8-byte alignment.
namespace epara {
static_assert(sizeof(GemmGroup) % TMAP_ALIGN == 0 && sizeof(PrefillMaps) % TMAP_ALIGN == 0 && sizeof(AttnEncGroup) % TMAP_ALIGN == 0 &&
              sizeof(MlpGroup) % TMAP_ALIGN == 0, "TMA maps on lines of their own");
static_assert(sizeof(AttnPrefillGroup) % 8 == 0 && sizeof(PrefillTile) == 24 && sizeof(RowDesc) == 12 && sizeof(WrittenPage) == 16, "descriptor sizes");
static_assert(sizeof(NormGroup) % 8 == 0 && sizeof(GatherGroup) % 8 == 0 && sizeof(RopeGroup) % 8 == 0 &&
              sizeof(AttnDecGroup) % 8 == 0 && sizeof(AssembleGroup) % 8 == 0 &&
              sizeof(OutputGroup) % 8 == 0 && sizeof(ReqDesc) % 16 == 0 && sizeof(AttnReq) % 16 == 0,
              "descriptor sizes");
}  // namespace epara
