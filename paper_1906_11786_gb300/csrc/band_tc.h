// Tensor-core (tcgen05 / TMEM / TMA) band contractions for sm_103a.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"

namespace bg {

// True when the fused tensor-core kernels handle (dtype, H, S, P) for this plan.
bool band_tc_supported(const bg_plan* p, int dtype, int H);
// Whether band_tc_fwd (bwd = false) or band_tc_bwd with `lists` runs the gathered kernel.
bool band_tc_uses_lists(const bg_plan* p, int dtype, int H, bool bwd);
size_t band_tc_fwd_ws_bytes(const bg_plan* p, int dtype, int H);
size_t band_tc_bwd_ws_bytes(const bg_plan* p, int dtype, int H);
// Y = sum_p A_p (E W_p + b_p), bf16 operands, fp32 accumulation and output.  `lists` allows the
// gathered kernel where the plan has edge lists (single propagations; GGNN steps pass false).
cudaError_t band_tc_fwd(const bg_plan* p, int H, const void* E, const void* W, const float* b,
                        float* Y, char* ws, size_t ws_bytes, int* status, cudaStream_t st,
                        bool lists);
// dE (+)= sum_p (A_p^T dY) W_p^T, dW_p (+)= E^T A_p^T dY, db_p (+)= colsum(A_p^T dY).
cudaError_t band_tc_bwd(const bg_plan* p, int H, const void* E, const void* W, const float* dY,
                        float* dE, float* dW, float* db, int accum, char* ws, size_t ws_bytes,
                        int* status, cudaStream_t st, bool lists);
// The band kernel's second-product weights (band_tc_w_bytes): from W [P][H][H] bf16, the forward
// operand W_p^T (bwd = 0) or the backward operand W_p (bwd = 1), fp32 (kind::tf32 product).
size_t band_tc_w_bytes(const bg_plan* p, int H);
// With b (forward): also the bias split b2T [H][64] 16-bit, columns p / 32+p the high part /
// remainder of b[p][h], as bf16, or as fp16 for a plan whose in-degrees exceed 256 (the in-degree
// table is fp16 then; a finite |b| above 65504 is recorded in `status`).
cudaError_t band_tc_prep_w(const bg_plan* p, int H, const void* W, int bwd, void* Wk,
                           const float* b, __nv_bfloat16* b2T, int* status, cudaStream_t st);
// Kernel-level entry points used by the fused GGNN steps (operands already in kernel layout):
//   X: [n_pad][H] bf16 states; Wk: band_tc_prep_w(bwd = 0);
//   b2T: [H][64] bf16 bias split or NULL.  Outputs (each optional): out fp32 [n][H],
//   outb bf16 [n][H], outT bf16 [H][ld_outT].
//   split: fp32 scratch of band_tc_split_floats(p, H) floats (may be NULL: no tile splitting) for
//   the partial outputs of tiles that the launch splits over several CTAs.
//   addend (may be NULL): fp32 [rows_in][H], added to the Y rows of the plan's supernode in-edge
//   targets (row r gets addend[p->d_sin_slot[r]]) before the outputs are written.
size_t band_tc_split_floats(const bg_plan* p, int H);
//   b32: the fp32 bias [P][H] (or NULL) beside its split b2T; the S = 512 kernels at 64-column
//   slices add the bias in their epilogue from it.
cudaError_t band_tc_fwd_core(const bg_plan* p, int H, const __nv_bfloat16* X, const void* Wk,
                             const __nv_bfloat16* b2T, const float* b32, float* out,
                             __nv_bfloat16* outb, __nv_bfloat16* outT, int64_t ld_outT,
                             float* split, const float* addend, int* status, cudaStream_t st,
                             bool lists = false);  // (lists: with `out` alone)
//   dY: [n_pad][H] bf16; Wk: band_tc_prep_w(bwd = 1); dE fp32 (+)=; dM: [n_pad][P*H] bf16, 16-byte
//   aligned.
cudaError_t band_tc_bwd_core(const bg_plan* p, int H, const __nv_bfloat16* dY, const void* Wk,
                             float* dE, int accumulate, __nv_bfloat16* dM, float* split,
                             int* status, cudaStream_t st, bool lists = false);
// out[c * ld_out + r] = bf16(in[r][c]) for `batch` consecutive R x Cc matrices (in fp32 or bf16;
// ld_out <= 0 means R; batches are R*Cc apart on both sides).
cudaError_t prep_transpose_bf16(const void* in, int in_is_f32, __nv_bfloat16* out, int R, int Cc,
                                int batch, cudaStream_t st, int64_t ld_out = 0);
// Builds and uploads the tensor-core path's plan data (no-op where unsupported); 0 on success.
int band_tc_upload(bg_plan* p, cudaStream_t st);
// After it: edge lists for the orientations and state sizes that are faster on them and fit.  They are
// an option: where host or device memory does not suffice, the plan stays without (not an error).
cudaError_t band_tc_upload_lists(bg_plan* p, cudaStream_t st);
// Host side of band_tc_upload (band_tiles.cpp): the bit-interleaved window chunks of every
// 128-row tile, [n_pad / 128][P][C1][128][4] words for C1 128-column chunks per tile, in both
// orientations, and the per-row in-degrees [n_pad][64] as bf16; returns the largest in-degree.
int band_tc_host_tiles(const bg_plan* p, int C1, std::vector<uint32_t>& mi,
                       std::vector<uint32_t>& mti, std::vector<uint16_t>& deg);
// (`edges`, if not NULL: the number of edges in the tiles)
int band_tc_host_degrees(const bg_plan* p, std::vector<uint16_t>& deg, int64_t* edges = nullptr);
void band_tc_host_chunks(const bg_plan* p, int C1, bool transposed, uint32_t* out);
// Edge lists of the gathered band kernel, one orientation.  Per 128-row tile, 16-row group and edge
// type: steps of 16 edges (at least one) in blocks of kGatherBlock, each step 32 words, one per lane of
// the warp that multiplies it (band_tc.cu): bits 0-17 the byte offset, within the tile's window of
// 128-byte state rows, of the 16 bytes this lane names to ldmatrix (edge lane % 16, column chunk
// lane / 16, 128-byte swizzle applied); bit 18 set in the type's last block; bits 19-20 the block's
// steps less one; bits 24-31 this lane's entries of the 16 x 16 0/1 matrix (row of the group, edge)
// in mma fragment order.  The window holds rows row0 - lo .. row0 - lo + rows of the state and 8 zero
// rows after them, which padding entries name.
constexpr uint32_t kGatherLast = 1u << 18, kGatherMore = 1u << 19;
constexpr int kGatherBlock = 4;
struct GatherLists {
  std::vector<uint32_t> words;  // [blocks][32][kGatherBlock]
  std::vector<uint32_t> off;    // [n_tiles][8][P + 1] first block, even types first, then odd
  int lo = 0, rows = 0;
  int64_t steps = 0, blocks = 0;
};
// On the device (band_lists.cu): the edges of each (tile, group, type) in the place of its offset, types in
// the lists' order, with the window's reach before and behind the tile (two ints, cleared before); then,
// with the offsets in place, the words (32 kGatherBlock per block, every one written).
cudaError_t list_count(const bg_plan* p, bool transposed, uint32_t* d_off, int* d_reach, cudaStream_t st);
cudaError_t list_emit(const bg_plan* p, bool transposed, const uint32_t* d_off, int lo, int rows,
                      uint32_t* d_words, cudaStream_t st);
// Their sizes: counts in `off` become offsets, `reach` becomes lo and rows.
void list_layout(const bg_plan* p, const int* reach, GatherLists& out);
// The same lists built on the host, and the number of their steps alone: what tests compare with.
int64_t band_tc_list_steps(const bg_plan* p, bool transposed);
void band_tc_host_lists(const bg_plan* p, bool transposed, GatherLists& out);
// Loads (CUDA lazy loading) every kernel band_tc_fwd can launch for this plan's block size, at
// any H, on the current device.
cudaError_t band_tc_preload_fwd(const bg_plan* p);
// Frees device data the tensor-core path keeps with the plan.
void band_tc_release(bg_plan* p);

}  // namespace bg
