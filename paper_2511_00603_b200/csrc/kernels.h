// Host-side launchers of the step's kernels.  `groups` pointers are device memory.
#pragma once
#include <cuda_runtime.h>
#include "desc.h"

namespace epara {

// (beside: see pdl_begin() in common.cuh)

constexpr int GATHER_PATCH_ROWS = 8;   // patch rows per block of the patch gather
void launch_gather(const GatherGroup* groups, int n_groups, int max_blocks, cudaStream_t st);
int norm_blocks(int M, int d);
void launch_norm(const NormGroup* groups, int n_groups, int max_blocks, cudaStream_t st);
void launch_rope_append(const RopeGroup* groups, int n_groups, int max_B, cudaStream_t st);
void launch_assemble(const AssembleGroup* groups, int n_groups, int max_rows, cudaStream_t st);
void launch_output(const OutputGroup* groups, int n_groups, int max_B, cudaStream_t st);

// Plain CUDA-core grouped GEMM, 64 x 64 tiles (comparator for the tensor-core kernel).
constexpr int SIMT_TILE = 64;
void launch_gemm_simt(const GemmGroup* groups, int n_groups, int total_tiles, cudaStream_t st);

// tcgen05 grouped GEMM of groups with more than 128 rows (GemmGroup::stream == 2): 256 x bn tiles on CTA pairs,
// persistent.  `status` is a device int the kernel sets non-zero if a bounded wait ran out.  total_items = sum over
// groups of tiles_m * tiles_n (tiles_m counts 256-row tiles).  gemm_pair_config() picks bn (128, 192 or 256).
constexpr int TC_BM = 128;
constexpr int TC_BN_MAX = 256;
constexpr int TC_BK = 64;
double gemm_pair_config(long long rows_cap, int N, int K, int epi, int sm_count, int* bn);
cudaError_t launch_gemm_tc_pair(const GemmGroup* groups, int n_groups, int total_items, int* status, int sm_count,
                                cudaStream_t st, int beside = 0);
bool gemm_mlp_eligible(long long rows_cap, int d, int F);
cudaError_t launch_gemm_mlp_pair(const MlpGroup* groups, int n_groups, int total_items, int* status, int sm_count,
                                 cudaStream_t st, int beside = 0);

// Swapped-operand tensor-core GEMM (GemmGroup::stream == 3): a cluster of `ksplit` CTAs per tile of 128 output
// columns and bn batch rows; all groups of a launch share ksplit.  gemm_swap_config() picks bn (a multiple of 16, at
// most GEMM_SWAP_TILE_ROWS) and ksplit from the row capacity; tmW is the weight map (box 128 rows), tmA the activation
// map (box bn rows); tiles_m = ceil(M / bn), tiles_n = gemm_swap_tiles_n(N), tile_start counts tiles_m * tiles_n.
// max_nb: widest bn of the launch.
constexpr int GEMM_SWAP_TILE_ROWS = 256;
double gemm_swap_config(long long rows_cap, int N, int K, int sm_count, int* nb, int* ksplit);
int gemm_swap_tiles_n(int N);
cudaError_t launch_gemm_swap(const GemmGroup* groups, int n_groups, int total_items, int ksplit, int max_nb, int* status,
                             int sm_count, cudaStream_t st, int beside = 0);

// The same on pairs of CTAs (GemmGroup::stream == 5): tiles of 256 output columns and bn batch rows (a multiple of 32, at
// most GEMM_SWAP2_TILE_ROWS), `ksplit` (1 or 2) pairs per tile; from 129 rows to some thousand, wide shapes three thousand, where its estimate is the smallest.  Maps: tmW box 128 rows,
// tmA box half of gemm_swap2_first(bn) rows, tmC the activations again with a box of half the rest (when there is a rest).
constexpr int GEMM_SWAP2_TILE_ROWS = 384;
double gemm_swap2_config(long long rows_cap, int N, int K, int sm_count, int* nb, int* ksplit);
int gemm_swap2_first(int nb);
int gemm_swap2_tiles_n(int N);
cudaError_t launch_gemm_swap2(const GemmGroup* groups, int n_groups, int total_items, int ksplit, int* status, int sm_count, cudaStream_t st,
                              int beside = 0);
enum : int { GEMM_SIMT = 0, GEMM_STREAM = 1, GEMM_PAIR = 2, GEMM_SWAP = 3, GEMM_MLP = 4, GEMM_SWAP2 = 5 };   // GemmGroup::stream
// The kernel for a GEMM that the weight-streaming kernel does not take, with its tile (GemmGroup::bn, ksplit).
int gemm_tc_choice(long long rows_cap, int N, int K, int epi, int sm_count, int* bn, int* ksplit);

// Weight-streaming GEMM (GemmGroup::stream == 1) for groups that never exceed 16 rows, and for small matrices: one block
// per 16 rows of W over the whole K and 32 batch rows, mma.sync, no tensor maps.  total_items = sum of
// tiles_m * tiles_n; max_rows = the most rows of a group in the launch.
constexpr int GEMM_STREAM_MAX_ROWS = 16;
bool gemm_stream_eligible(long long rows_cap, int N, int K);
int gemm_stream_tiles_n(int N);
int gemm_stream_tiles_m(int M);
cudaError_t launch_gemm_stream(const GemmGroup* groups, int n_groups, int total_items, int max_rows, cudaStream_t st);

// Decode attention, split-KV over 256-token chunks.  fused = 1: the block of a (request, kv head) that
// finishes last merges the chunk partials (AttnDecGroup::counters must be zero at launch and is left
// zero); fused = 0: a second kernel merges them.  attn_decode_fused() is the rule that picks the mode
// from the launch's block count, the chunks of a request and the head size; both modes give the same bits.
constexpr int ATTN_CHUNK = 256;
bool attn_decode_fused(int total_B, int max_Hkv, int max_chunks, int hd, int sm_count);
cudaError_t launch_attn_decode(const AttnDecGroup* groups, int n_groups, int total_B, int max_Hkv, int max_Hq,
                               int max_chunks, int hd, int gqa, int fused, cudaStream_t st, int beside = 0);
// Set-up of a single-kernel decode-attention call on the stream: writes `g` to `dst`, clears *g.status and
// g.counters[0 .. n_counters), fills reqs[b] = {tables + b*stride, kv_lens[b] clamped to [0, max_len]}.
void launch_attn_prepare(const AttnDecGroup& g, AttnDecGroup* dst, AttnReq* reqs, const int32_t* kv_lens,
                         const int32_t* tables, int stride, int max_len, int n_counters, cudaStream_t st);
constexpr int DEC_STATUS_OFFSET = 192;   // byte offset of the status word in a single-kernel call's scratch

// Attention of many query rows on tcgen05, persistent over work items of `mt` (1 or 2) tiles of FLASH_TILE query rows;
// `status` as for the GEMM.  Two tiles keep the tensor core and the softmax busy at once; attn_flash_tiles() picks one
// when the launch's tiles do not outnumber the SMs.
constexpr int FLASH_TILE = 128;
// With decode attention beside it the launch also leaves SMs to that one's blocks: one tile keeps the launch short while they
// are few, two tiles leave more SMs (1B decoder, a 512-token chunk, 128 tiles: with 4 / 12 / 24 / 60 decode requests, 14 / 42 /
// 84 / 210 blocks per SM left over, 2306 / 2409 / 2560 / 2818 us a step with one tile and 2467 / 2485 / 2525 / 2779 with two; a
// 256-token chunk with 24 / 60 requests, 20 / 50 blocks: 1822 / 2271 and 1955 / 2236; 128 and 1024 tokens with 4 to 60 requests: the choice
// within 1 % of the better one.  Head size 128, 8B decoder, 32 layers: 256 tokens with 4 / 12 / 24 / 60 requests 6689 / 7025 / 7541 / 9615
// with one tile and 6932 / 7224 / 7723 / 9592 with two, 512 tokens with 24 / 60 12249 / 14171 and 12344 / 14102, where runs differ by 2 %).
// All decode blocks of the step count, whichever model's: they share the SMs left over.
constexpr int FLASH_DEC_BLOCKS = 48;
inline int attn_flash_tiles(long long total_tiles, int sm_count, long long dec_blocks = 0) {
  return total_tiles <= sm_count && dec_blocks <= FLASH_DEC_BLOCKS * (sm_count - total_tiles) ? 1 : 2;
}
// ... causal attention of prompt chunks (head size 64 or 128)
cudaError_t launch_attn_prefill(const AttnPrefillGroup* groups, int n_groups, int total_items, int mt, int hd, int* status,
                                int sm_count, cudaStream_t st, int beside = 0);
// ... encoder attention for groups with AttnEncGroup::tc (hd 64); total_items = sum of B * H * q_blocks.
cudaError_t launch_attn_encoder_tc(const AttnEncGroup* groups, int n_groups, int total_items, int mt, int* status, int sm_count,
                                   cudaStream_t st, int beside = 0);

// Encoder (bidirectional) attention on mma.sync, one block per (image, head, query block).
cudaError_t launch_attn_encoder(const AttnEncGroup* groups, int n_groups, int total_blocks, int max_T,
                                cudaStream_t st);
int attn_encoder_q_blocks(int T);

}  // namespace epara
