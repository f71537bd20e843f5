// Edge lists of the gathered band kernel, built on the device from the plan's bit tiles at upload
// (format: band_tc.h; the kernel that reads them: band_tc.cu).  On host threads the same lists took longer
// than all the rest of a small plan's upload (1,000 nodes, S = 256, 20 types: 2.0 ms of 3.6; 131k nodes,
// S = 512: 33 of 82), most of it for starting the threads; the masks are on the device anyway.
//
// Both kernels: one block per 16-row group of a 128-row tile, one warp per type.  Bound: a few hundred
// mask words per warp, nearly all zero, then a short serial deal of its edges.
#include <algorithm>

#include "band_tc.h"
#include "kernels.h"

namespace bg {
namespace {

constexpr int kWarps = 8, kMaxWords = 16 * 3 * (512 / 32);  // mask words of one type of a group at S = 512

// One type's mask words of 16 rows from row R, in the order row, diagonal, word: f(t, row, column of bit 0
// less `row0`, word) by the lane that holds word t; every lane of the warp takes part in every round.
template <typename F>
__device__ __forceinline__ void for_words(const uint32_t* __restrict__ masks, int K, int S, int P, int64_t R,
                                          int64_t row0, int q, F f) {
  const int lane = threadIdx.x & 31, W32 = S / 32, per_row = 3 * W32, words = 16 * per_row;
  const int64_t kr = R / S, r0 = R % S;  // (16 rows never cross a block-row)
  for (int t0 = 0; t0 < words; t0 += 32) {
    const int t = t0 + lane, i = t / per_row, dj = t - i * per_row, d = dj / W32, j = dj - d * W32;
    const int64_t kc = kr + d - 1;
    uint32_t w = 0;
    if (t < words && kc >= 0 && kc < K)
      w = masks[((((size_t)kr * 3 + d) * P + q) * S + r0 + i) * W32 + j];
    f(i, (int)(kc * S + 32 * j - row0), w);
  }
}

__global__ void __launch_bounds__(32 * kWarps) k_list_count(const uint32_t* __restrict__ masks, int K, int S,
                                                            int P, uint32_t* __restrict__ off,
                                                            int* __restrict__ reach) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t R = (int64_t)blockIdx.x * 16, row0 = R / 128 * 128;
  int lo = 0, hi = 0;
  for (int q = warp; q < P; q += kWarps) {
    int m = 0;
    for_words(masks, K, S, P, R, row0, q, [&](int, int rel, uint32_t w) {
      if (!w) return;
      m += __popc(w);
      lo = max(lo, -(rel + __ffs(w) - 1));
      hi = max(hi, rel + 31 - __clz(w) - 127);
    });
    m = __reduce_add_sync(0xffffffffu, m);
    if (lane == 0)
      off[(size_t)blockIdx.x * (P + 1) + (q & 1 ? (P + 1) / 2 : 0) + q / 2] = (uint32_t)m;
  }
  lo = __reduce_max_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    atomicMax(reach, lo);
    atomicMax(reach + 1, hi);
  }
}

// Lane r < 8 holds the edges of window-row residue r: where it stands in the type's nonzero words, and how
// many it has left.  A step takes two sets of 8 edges: one of every residue left, the fullest first, then,
// as far as the steps to come could not take the rest, further ones of the fullest; padding entries take a
// zero row of an unused residue (fewer than there are such, since every residue left was used).
__global__ void __launch_bounds__(32 * kWarps) k_list_emit(const uint32_t* __restrict__ masks, int K, int S,
                                                           int P, const uint32_t* __restrict__ off, int lo,
                                                           int rows, uint4* __restrict__ words) {
  __shared__ uint32_t s_word[kWarps][kMaxWords];
  __shared__ uint16_t s_at[kWarps][kMaxWords];  // row << 12 | column of bit 0 less the tile's first row + 2048
  __shared__ uint32_t s_ent[kWarps][16];        // an edge: 1 << 31 | row << 16 | window row; padding: row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t R = (int64_t)blockIdx.x * 16, row0 = R / 128 * 128;
  uint32_t* word = s_word[warp];
  uint16_t* at = s_at[warp];
  uint32_t* ent = s_ent[warp];
  const uint32_t residue = 0x01010101u << (lane & 7);  // (32 j and 128 t are multiples of 8, as lo is)
  for (int q = warp; q < P; q += kWarps) {
    int nz = 0;
    for_words(masks, K, S, P, R, row0, q, [&](int i, int rel, uint32_t w) {
      const uint32_t some = __ballot_sync(0xffffffffu, w != 0);
      if (w) {
        const int k = nz + __popc(some & ((1u << lane) - 1));
        word[k] = w;
        at[k] = (uint16_t)(i << 12 | (rel + 2048));
      }
      nz += __popc(some);
    });
    __syncwarp();
    int cnt = 0;
    for (int k = lane >> 3; k < nz; k += 4) cnt += __popc(word[k] & residue);
    cnt += __shfl_xor_sync(0xffffffffu, cnt, 8);
    cnt += __shfl_xor_sync(0xffffffffu, cnt, 16);
    if (lane >= 8) cnt = 0;
    int rem = __reduce_add_sync(0xffffffffu, cnt);
    const int steps = max(1, (rem + 15) / 16);
    int k_at = 0;
    uint32_t left = nz ? word[0] & residue : 0;
    auto pop = [&]() -> uint32_t {
      while (!left && k_at + 1 < nz) left = word[++k_at] & residue;
      const uint32_t a = at[k_at], bit = __ffs(left) - 1;
      left &= left - 1;
      --cnt;
      return 0x80000000u | (a >> 12) << 16 | ((a & 0xFFFu) + bit - 2048 + lo);
    };
    uint4* o = words + (size_t)off[(size_t)blockIdx.x * (P + 1) + (q & 1 ? (P + 1) / 2 : 0) + q / 2] * 32 + lane;
    uint4 out = make_uint4(0u, 0u, 0u, 0u);
    for (int s = 0; s < steps; ++s) {
      for (int half = 0; half < 2; ++half) {
        const int need = max(0, rem - 8 * (2 * (steps - s) - half - 1));
        const int key = lane < 8 ? cnt << 3 | (7 - lane) : 0;
        int rank = 0;
#pragma unroll
        for (int x = 0; x < 8; ++x) rank += __shfl_sync(0xffffffffu, key, x) > key;
        const bool has = lane < 8 && cnt > 0;
        const uint32_t used = __ballot_sync(0xffffffffu, has);
        if (has) ent[8 * half + rank] = pop();
        int k = __popc(used);
        for (; k < need; ++k) {
          const int top = 7 - (__reduce_max_sync(0xffffffffu, lane < 8 ? cnt << 3 | (7 - lane) : 0) & 7);
          if (lane == top) ent[8 * half + k] = pop();
        }
        rem -= k;
        const uint32_t free = ~used & 0xFFu;
        const int pad = k + __popc(free & ((1u << lane) - 1));
        if (lane < 8 && (free >> lane & 1) && pad < 8) ent[8 * half + pad] = (uint32_t)(rows + lane);
      }
      __syncwarp();
      const uint32_t row = ent[lane & 15] & 0xFFFFu;
      uint32_t w = row * 128 + ((((uint32_t)lane >> 4) ^ (row & 7)) << 4);
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int k = 2 * (lane & 3) + (x & 1) + 8 * (x >> 1);
        const uint32_t e = ent[k], r = e >> 16 & 15u;
        if (e >> 31 && (r & 7) == (uint32_t)lane >> 2) w |= 1u << (24 + (r >> 3) + 2 * (k >> 3) + 4 * (k & 1));
      }
      const int in_blk = s % kGatherBlock, in = min(kGatherBlock, steps - s + in_blk);
      w |= (uint32_t)(in - 1) * kGatherMore + (s - in_blk + in == steps ? kGatherLast : 0u);
      (in_blk == 0 ? out.x : in_blk == 1 ? out.y : in_blk == 2 ? out.z : out.w) = w;
      if (in_blk == in - 1) {
        o[(size_t)(s / kGatherBlock) * 32] = out;
        out = make_uint4(0u, 0u, 0u, 0u);
      }
      __syncwarp();  // the entries are free for the next step
    }
  }
}

}  // namespace

cudaError_t list_count(const bg_plan* p, bool transposed, uint32_t* d_off, int* d_reach, cudaStream_t st) {
  k_list_count<<<p->n_pad() / 16, 32 * kWarps, 0, st>>>(transposed ? p->d_masksT : p->d_masks, p->K, p->S, p->P,
                                                        d_off, d_reach);
  note_launch();
  return cudaGetLastError();
}

cudaError_t list_emit(const bg_plan* p, bool transposed, const uint32_t* d_off, int lo, int rows,
                      uint32_t* d_words, cudaStream_t st) {
  k_list_emit<<<p->n_pad() / 16, 32 * kWarps, 0, st>>>(transposed ? p->d_masksT : p->d_masks, p->K, p->S, p->P,
                                                       d_off, lo, rows, reinterpret_cast<uint4*>(d_words));
  note_launch();
  return cudaGetLastError();
}

}  // namespace bg
