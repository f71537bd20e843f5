// Fused band contraction on the 5th-generation tensor cores (tcgen05, TMEM, TMA) for sm_103a.
//
// Forward (Algorithm 1's aggregate-first order, Eq. 3): for a 128-row tile of block-row k and
// every edge type p,
//     pre_p = sum_{d in -1,0,+1} A_{k,d,p} E_{k+d}        (128 x 3S  times  3S x H, fp32 in TMEM)
//     Y_k  += pre_p W_p                                     (chained MMA, A operand read from TMEM)
// and the per-type bias enters as one more product deg_k [128 x 2P] x [b_hi; b_lo] with exact
// integer in-degrees and b split into two bf16 halves (fp16 for a plan with an in-degree above
// 256, where bf16 integers stop being exact).  pre_p never leaves the SM.
// Backward (transposed band): the same kernel with the transposed tiles, dY instead of E and W_p
// instead of W_p^T gives dE_j += sum_p (A^T dY)_p W_p^T; dM_p = A_p^T dY is also written (bf16,
// [n][P H]) for the weight gradient.
//
// The second product runs as kind::tf32 straight from the fp32 pre_p (W_p staged as fp32), so no
// thread touches pre_p between the two products and no MMA issuer waits on a conversion.  The
// band product is N = 64: at H = 128 the tile makes two passes over 64-column halves of the state,
// pass hh contracting the band with columns 64 hh .. of E and multiplying by rows 64 hh .. of W_p
// (Y = sum_p sum_hh pre_p[:, hh] W_p[hh, :]); the (half, type) jobs alternate between two
// 64-column pre_p units, so a job's band products overlap the previous job's W product.
//
// The 0/1 adjacency is the MMA's A operand.  It is stored as bits (the whole band costs
// 3 P S^2 / 8 bytes per block-row) and expanded on chip straight into tensor memory: the bits of
// each 32-column word are interleaved at upload (column 2j at bit j, column 2j+1 at bit 16+j) so
// that one AND and one multiply give the packed bf16 pair {1.0 or 0, 1.0 or 0}.
//
// Roles (128 x (2 + expander groups) threads, one CTA per SM, persistent over tiles):
//   warp 0      TMA producer: state blocks (B operand of the band product), W tiles, deg, bias
//   warp 1      TMEM allocator and band-product issuer (an elected lane of the converged warp
//               issues), one wait per job (per chunk group at S = 256)
//   warp 2      mask producer: one bulk copy per (tile, type) of the bit tiles into an SMEM ring
//   warp 3      second MMA issuer: the pre_p W_p products and the bias product, so that their
//               waits never stall the band-product stream
//   expanders   thread r of a warpgroup turns row r's mask bits into bf16 A tiles in TMEM; two
//               warpgroups taking the edge types in turn (warps 4-11)
//   converters  the last warpgroup: dM_p to global (backward), final epilogue TMEM -> global
// A tcgen05.mma of N = 64 is about as long as its issue, so any wait on the band-product
// issuer leaves the tensor pipe idle: that issuer waits once per job, on a barrier that the
// expanders (all the job's A tiles are in TMEM), the second issuer (the pre_p unit is free) and
// in the backward pass the converters complete together.
// Consumer warps signal a barrier with one arrive per warp after __syncwarp.  Waiting roles other
// than the expanders sleep between polls so that the MMA issuers keep their issue slots.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <cstdlib>
#include <cstring>
#include <memory>
#include <mutex>
#include <vector>

#include "band_tc.h"
#include "gemm_tc.h"
#include "kernels.h"
#include "tc_util.cuh"

namespace bg {

using namespace tc;

namespace {

constexpr int kTile = 128;     // rows per tile = UMMA M
constexpr int kSmemLimit = 232448;  // dynamic shared memory one block can have

// Block size S: a 128-row tile sees a window of C1 128-column chunks of the state (and of its
// bit tiles): rows [row0, row0 + 128) only couple to columns in block-rows kr - 1 .. kr + 1 of
// their own block-row kr, which all lie in [ws, ws + 128 C1) with ws = (row0 / S) S - S.
//   S <= 64: C1 = 2 (the tile spans 128 / S block-rows);  S = 128: 3;  S = 256: 6;  S = 512: 12.
__host__ __device__ constexpr int band_chunks(int S) { return S <= 64 ? 2 : 3 * (S / 128); }

// Shapes (block size, state columns per pass) whose forward adds the bias in its epilogue, in-degree
// times b in fp32, dense and gathered alike; at the others it is a product of in-degrees and the bias
// split into two 16-bit parts.
__host__ __device__ constexpr bool bias_in_fp32(int S, int SW) { return S == 512 && SW == 64; }

template <int H, int S, bool BWD = false>
struct Cfg {
  // H > SW runs as H / SW passes over SW-column slices of the state: pass hh contracts the band
  // with columns SW hh .. SW hh + SW - 1 of E and multiplies the result by rows SW hh .. of W_p,
  // into Y.  SW = 64, or 32 at H = 32.
  static constexpr int SW = H < 64 ? 32 : 64;                 // state columns per pass
  // S = 512 at SW = 64: the 1536-node window takes 192 KB, so the kernel keeps nothing else of
  // size in shared memory: the expanders read their mask words straight from global memory (L2)
  // instead of a staged ring, W has one stage, and the bias is added in the epilogue (in-degree
  // times b in fp32) instead of by a product with staged operands
  static constexpr bool GM = bias_in_fp32(S, SW);
  static constexpr int NH = H / SW;
  static constexpr int C1 = band_chunks(S);                   // 128-column chunks per type
  static constexpr int XROW = SW * 2;                         // bytes of one node's slice
  static constexpr int XCHUNK = 128 * XROW;                   // 128 nodes x SW state columns
  static constexpr int XWIN = C1 * XCHUNK;                    // one half's window
  static constexpr int NXB = XWIN <= 48 * 1024 ? 2 : 1;       // state-window buffers
  // W ring stages: at H <= 64, S <= 128 the small window leaves room for a deeper ring (the second
  // issuer's W stages come from L2, and it gates the release of the pre_p units); measured best
  // with four stages forward and three backward, the mask ring giving up the space
  static constexpr bool DW = H <= 64 && S <= 128;
  static constexpr int NW = GM ? 1 : (DW ? (BWD ? 3 : 4) : 2);
  // W stages hold K-columns of W_p^T as fp32 (tf32 operand) in 32-column atoms of H rows: a job's
  // 64 K-columns in one stage, or at H = 256 (64 KB) in two stages of one atom
  static constexpr int WK = H <= 128 ? SW : 32;               // K-columns per stage
  static constexpr int WJ = SW / WK;                          // stages per job
  static constexpr int WSTAGE = (WK / 32) * H * 128;
  static constexpr int DEG = kTile * 128;                     // 128 rows x 64 bf16
  // forward: deg buffers and H rows x 64 bf16 of bias; backward: the dM_p staging tile instead
  static constexpr int NDEG = (GM || BWD) ? 0 : (NH > 1 ? 1 : 2);
  static constexpr int B2 = (GM || BWD) ? 0 : H * 128;
  static constexpr bool DMS = BWD && !(GM && H > 64);         // (no room for it at H = 128, S = 512)
  static constexpr int DM = DMS ? kTile * SW * 2 : 0;
  static constexpr int OFF_X = 0;
  static constexpr int OFF_W = OFF_X + NXB * XWIN;
  static constexpr int OFF_DEG = OFF_W + NW * WSTAGE;
  static constexpr int OFF_B2 = OFF_DEG + NDEG * DEG;
  static constexpr int MSTAGE = C1 * kTile * 16;              // C1 chunks x 128 rows x 128 bits
  // mask ring stages (one job each): as many as fit beside the window, at least two
  static constexpr int NM0 = (C1 <= 3 ? (DW ? (BWD ? 6 : 4) : 8) : 4) / NH;
  static constexpr int NM = GM ? 0 : (C1 > 6 ? 2 : (NM0 > 2 ? NM0 : 2));
  // ring sizes as divisors (the GM shapes have no deg or mask ring; their code paths are off)
  static constexpr int NDEGD = NDEG > 0 ? NDEG : 1, NMD = NM > 0 ? NM : 1;
  static constexpr int OFF_DM = OFF_B2 + B2;
  static constexpr int OFF_M = OFF_DM + DM;
  static constexpr int OFF_BAR = OFF_M + NM * MSTAGE;
  static constexpr int SMEM = OFF_BAR + 1024 + 1024;          // barriers + 1 KB alignment slack
  // TMEM columns: Y (H), two 64-column pre_p units used by the jobs (half, type) in turn, so that
  // a job's band products overlap the previous job's W product, then the A-tile slots
  // (a third unit for the backward at H <= 64, so that the converters' read of one job's dM_p
  // overlaps the band products of the next two, measured 2% slower at packed64: 85.7 vs 84.1 us)
  static constexpr int NB = 2;
  static constexpr int YCOL = 0;
  static constexpr int D1COL0 = H < 64 ? 64 : H;              // units start 64-column aligned
  static constexpr int ACOL = D1COL0 + NB * 64;
  static constexpr int NA = (512 - ACOL) / 64;
  // a job's chunks come in CG-chunk groups (one barrier wait each), G groups per job; a group and
  // one more A tile must fit in the NA slots (H = 256 has two slots: one chunk per group)
  static constexpr int CG = (C1 <= 3 && NA > C1) ? C1 : (NA > 3 ? 3 : NA - 1);
  static constexpr int G = C1 / CG;
  static constexpr int NT = (8 / G) * G;                      // per-group barrier ring
  static constexpr int NE = 2;                                // expander warpgroups
  static constexpr int THREADS = 128 * (2 + NE);
  static_assert(H == 32 || H == 64 || H == 128 || H == 256, "state size");
  static_assert(C1 % CG == 0 && NT % G == 0, "chunk groups");
  // the release of a job's pre_p unit is signalled on the barrier of job + NB's first group: the
  // ring must hold NB jobs' groups, or that barrier would still serve a pending job
  static_assert(NT / G >= NB, "barrier ring");
  static_assert(NA >= CG + 1 && NA <= 8, "one group of A tiles and one more must fit");
  static_assert(GM || (NM >= 2 && NM <= 8), "mask ring");
  static_assert(SMEM <= kSmemLimit, "shared memory");
};

struct Bars {
  uint64_t x_full[2], x_empty[2];
  uint64_t w_full[4], w_empty[4];
  uint64_t deg_full[2], deg_empty[2];
  uint64_t b2_full;
  // release of A slot s for the expander group that uses it next: each group waits only on its
  // own barrier, once per use, so no waiter can fall two phases behind (the groups take jobs in
  // turn, and slot uses alternate between them irregularly)
  uint64_t a_empty[8][2];
  uint64_t d1_full[4];
  uint64_t t_full[8];
  uint64_t y_full, y_empty;
  uint64_t m_full[8], m_empty[8];
  uint64_t drain, drain2;
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ uint32_t expand_pair(uint32_t w, int j) {
  // w holds column 2j at bit j and column 2j+1 at bit 16+j (j < 8); result packs bf16 1.0/0.0
  return (w & (0x00010001u << j)) * (0x3F80u >> j);
}

// Expands one interleaved 32-bit mask word into 16 packed bf16 pairs.
__device__ __forceinline__ void expand_word(uint32_t w, uint32_t* out) {
#pragma unroll
  for (int j = 0; j < 8; ++j) out[j] = expand_pair(w, j);
  const uint32_t w8 = w >> 8;
#pragma unroll
  for (int j = 0; j < 8; ++j) out[8 + j] = expand_pair(w8, j);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// One arrive per warp once every lane of it is done (lanes' earlier operations are ordered
// before lane 0's arrive by the warp barrier).
__device__ __forceinline__ void warp_arrive(uint64_t* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
}

// Bounded wait for every MMA this thread issued (commit to an unused barrier).
__device__ __forceinline__ void drain_mmas(bool leader, uint64_t* bar) {
  if (leader) tc_commit(bar);
  __syncwarp();
  for (uint32_t t = 0; t < (1u << 24) && !mbar_try(bar, 0); ++t) {
  }
}

// Work of one launch.  Items 0 .. n_full-1 are whole tiles; when the tiles do not fill the last
// round of the grid evenly, each remaining tile is split into ksplit items over consecutive ranges
// of its jobs, which write their partial Y (fp32) to their own slice of `part`, and a fix-up
// kernel sums the slices in a fixed order into the outputs.
struct Sched {
  int n_items, n_full, ksplit, part_rows;
  float* part;  // [ksplit][part_rows][H]: partial Y of split items, rows from tile n_full on
  // forward: a row r with slot[r] >= 0 gets addend[slot[r]][:] added to its Y before the outputs
  // are written (the supernode rows' messages); NULL for none
  const float* addend;
  const int32_t* slot;
  // epilogue bias (shapes without the bias product): Y[r] += sum_p deg[r][p] b[p], the in-degrees
  // as 16-bit integers ([n][64], bf16 or, bias_f16, fp16) and b fp32 [P][H]; NULL for none
  const uint16_t* deg;
  const float* bias;
  int bias_f16;
};

// Tile and job range [j0, j1) of item w; part -1 for a whole tile, else its slice.
__device__ __forceinline__ void item_of(const Sched& sc, int w, int jobs, int& tile, int& j0,
                                        int& j1, int& part) {
  if (w < sc.n_full) {
    tile = w, j0 = 0, j1 = jobs, part = -1;
    return;
  }
  const int v = w - sc.n_full;
  tile = sc.n_full + v / sc.ksplit;
  part = v % sc.ksplit;
  j0 = part * jobs / sc.ksplit;
  j1 = (part + 1) * jobs / sc.ksplit;
}

// Lane i of each group of eight holds 16-byte chunks 0 .. 7 (four words each) of its own row; afterwards
// chunk i of the rows of lanes 0 .. 7.  Every lane of the warp calls it.
__device__ __forceinline__ void transpose8(uint32_t (&v)[32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = 4; m; m >>= 1) {
    const bool up = lane & m;
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (!(c & m))
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t a = v[4 * c + k], b = v[4 * (c | m) + k];
          const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? a : b, m);
          v[4 * c + k] = up ? got : a;
          v[4 * (c | m) + k] = up ? b : got;
        }
  }
}

template <int H, int S, bool BWD>
__global__ void __launch_bounds__(Cfg<H, S, BWD>::THREADS, 1)
    k_band_tc(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
              const __grid_constant__ CUtensorMap tm_deg, const __grid_constant__ CUtensorMap tm_b2,
              const __grid_constant__ CUtensorMap tm_dm, const uint32_t* __restrict__ maskI,
              float* __restrict__ out, __nv_bfloat16* __restrict__ outb,
              __nv_bfloat16* __restrict__ outT, int64_t ld_outT, __nv_bfloat16* __restrict__ dM,
              const Sched sc, int P, int has_bias,
              int bias_f16, int accumulate, int* status) {
  using C = Cfg<H, S, BWD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  Bars* bars = reinterpret_cast<Bars*>(smem + C::OFF_BAR);
  uint8_t* xwin = smem + C::OFF_X;
  uint8_t* wring = smem + C::OFF_W;
  uint8_t* degs = smem + C::OFF_DEG;
  uint8_t* b2s = smem + C::OFF_B2;
  uint8_t* mring = smem + C::OFF_M;
  volatile int* abort = &bars->abort;
  // A job is one (half, type) of a tile, in the order tile, half, type; job c writes pre_p unit
  // c % 2.  Chunk group gi = G c + g waits on t_full[gi % NT]: the 4 warps of the expander group
  // once its A tiles are in TMEM, and for first groups (g = 0) the release of the unit: the second
  // issuer's commit and, backward, the 4 converter warps.
  constexpr int kFree = 1 + (BWD ? 4 : 0);
  const int jobs = C::NH * P;  // per tile
  if (C::GM) has_bias = 0;     // the bias enters in the epilogue (sc.bias), not as a product
  // bias: once per tile, by the whole tile or its first slice

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->x_full[i], 1); mbar_init(&bars->x_empty[i], 1);
      mbar_init(&bars->deg_full[i], 1); mbar_init(&bars->deg_empty[i], 1);
    }
    for (int i = 0; i < 4; ++i) mbar_init(&bars->d1_full[i], 1);
    for (int i = 0; i < 4; ++i) { mbar_init(&bars->w_full[i], 1); mbar_init(&bars->w_empty[i], 1); }
    for (int i = 0; i < 8; ++i) { mbar_init(&bars->a_empty[i][0], 1); mbar_init(&bars->a_empty[i][1], 1); }
    for (int i = 0; i < 8; ++i) mbar_init(&bars->t_full[i], 4 + (i % C::G == 0 ? kFree : 0));
    mbar_init(&bars->b2_full, 1);
    mbar_init(&bars->y_full, 1);
    mbar_init(&bars->y_empty, 4);
    mbar_init(&bars->drain, 1);
    mbar_init(&bars->drain2, 1);
    for (int i = 0; i < 8; ++i) { mbar_init(&bars->m_full[i], 1); mbar_init(&bars->m_empty[i], 4); }
    bars->abort = 0;
    fence_mbar_init();
    // the first NB jobs find their pre_p unit free: stand in for the releases; likewise the first
    // use of each A slot (chunk s, job s / C1)
    for (int c = 0; c < C::NB; ++c)
      for (int a = 0; a < kFree; ++a) mbar_arrive(&bars->t_full[(c * C::G) % C::NT]);
    for (int sl = 0; sl < C::NA; ++sl) mbar_arrive(&bars->a_empty[sl][(sl / C::C1) % C::NE]);
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // TMEM is held: the next kernel in the stream may be scheduled on SMs as they free up
  grid_dep_launch();
  const uint32_t tmem = bars->tmem_base;

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------ TMA producer
    tma_prefetch_desc(&tm_x);
    tma_prefetch_desc(&tm_w);
    if (has_bias) tma_prefetch_desc(&tm_deg);
    // the state windows, W and the bias split may be the previous kernel's output (the bit tiles
    // and in-degrees are plan data)
    grid_dep_wait();
    if (has_bias) {
      mbar_expect_tx(&bars->b2_full, C::B2);
      tma_load_2d(b2s, &tm_b2, &bars->b2_full, 0, 0);
    }
    uint32_t widx = 0, xi = 0, di = 0;
    uint32_t n_x[2] = {0, 0}, n_deg[2] = {0, 0}, n_w[4] = {0, 0, 0, 0};
    bool ok = true;
    for (int w = blockIdx.x; w < sc.n_items && ok && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      const int row0 = k * kTile, ws = (row0 / S) * S - S;
      if (has_bias && part <= 0) {
        const int db = di % C::NDEGD;
        if (!mbar_wait(&bars->deg_empty[db], ((di / C::NDEGD) & 1) ^ 1, status, 102, abort, 64)) break;
        ++n_deg[db];
        ++di;
        mbar_expect_tx(&bars->deg_full[db], C::DEG);
        tma_load_2d(degs + db * C::DEG, &tm_deg, &bars->deg_full[db], 0, row0);
      }
      // job jb = P hh + p, stepped without dividing (the issuers' loops are on the MMA issue path)
      int hh = j0 / P, p = j0 - hh * P;
      for (int jb = j0; jb < j1 && ok; ++jb, p = p + 1 == P ? (++hh, 0) : p + 1) {
        if (jb == j0 || p == 0) {
          // the window of the job's state slice: rows ws .. ws + 128 C1 of state columns SW hh ..;
          // rows outside [0, n) arrive as zeros (TMA bounds fill)
          const int xb = xi % C::NXB;
          if (!mbar_wait(&bars->x_empty[xb], ((xi / C::NXB) & 1) ^ 1, status, 101, abort, 64)) {
            ok = false;
            break;
          }
          ++n_x[xb];
          ++xi;
          mbar_expect_tx(&bars->x_full[xb], C::XWIN);
          for (int a = 0; a < C::C1; ++a)
            tma_load_2d(xwin + xb * C::XWIN + a * C::XCHUNK, &tm_x, &bars->x_full[xb], C::SW * hh,
                        ws + a * 128);
        }
        // per job: K-columns SW hh .. of W_p^T in WJ stages of WK / 32 atoms
        {
          for (int wj = 0; wj < C::WJ; ++wj, ++widx) {
            const int ws2 = widx % C::NW;
            if (!mbar_wait(&bars->w_empty[ws2], ((widx / C::NW) & 1) ^ 1, status, 103, abort, 64)) {
              ok = false;
              break;
            }
            ++n_w[ws2];
            mbar_expect_tx(&bars->w_full[ws2], C::WSTAGE);
            for (int a = 0; a < C::WK / 32; ++a)
              tma_load_2d(wring + ws2 * C::WSTAGE + a * H * 128, &tm_w, &bars->w_full[ws2],
                          C::SW * hh + C::WK * wj + 32 * a, p * H);
          }
        }
      }
    }
    if (*abort) {
      // let this CTA's own copies land before shared memory is released (bounded)
      auto settle = [](uint64_t* bar, uint32_t uses) {
        if (!uses) return;
        for (uint32_t t = 0; t < (1u << 22) && !mbar_try(bar, (uses - 1) & 1); ++t) {
        }
      };
      for (int q = 0; q < 2; ++q) { settle(&bars->x_full[q], n_x[q]); settle(&bars->deg_full[q], n_deg[q]); }
      for (int q = 0; q < 4; ++q) settle(&bars->w_full[q], n_w[q]);
      if (has_bias) settle(&bars->b2_full, 1);
    }
  } else if (warp == 2 && lane == 0 && !C::GM) {
    // ------------------------------------------------------------------ mask producer
    // each job's C1 bit chunks (contiguous [C1][128][4] words of its type), NM jobs ahead of the
    // expanders; both halves of a tile read the same bits
    uint32_t midx = 0, n_m[8] = {0};
    for (int w = blockIdx.x; w < sc.n_items && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      bool ok = true;
      int p = j0 % P;
      for (int jb = j0; jb < j1; ++jb, ++midx, p = p + 1 == P ? 0 : p + 1) {
        const int ms = midx % C::NMD;
        if (!mbar_wait(&bars->m_empty[ms], ((midx / C::NMD) & 1) ^ 1, status, 104, abort, 64)) {
          ok = false;
          break;
        }
        ++n_m[ms];
        mbar_expect_tx(&bars->m_full[ms], C::MSTAGE);
        bulk_load(mring + ms * C::MSTAGE, maskI + ((size_t)k * P + p) * C::C1 * kTile * 4,
                  C::MSTAGE, &bars->m_full[ms]);
      }
      if (!ok) break;
    }
    if (*abort)
      for (int q = 0; q < 8; ++q)
        for (uint32_t t = 0; n_m[q] && t < (1u << 22) && !mbar_try(&bars->m_full[q], (n_m[q] - 1) & 1); ++t) {
        }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ band-product issuer
    // pre_p = sum over the window chunks of A_{tile,p,j} X_j (N = SW): one t_full wait per group
    // of chunks, then an unbroken MMA stream
    const bool leader = elect_one_sync();
    // B is the window itself, row-major: N = SW columns contiguous, one row per K index
    constexpr uint32_t idesc = idesc_bf16_f32(kTile, C::SW) | kIdescBMN;
    uint32_t c = 0, slot = 0, gi = 0, xi = 0;
    // expander group of chunk x + NA (the next user of the slot chunk x frees): job (x + NA) / C1
    // mod 2, kept as a group and a position within the job
    uint32_t nx_g = (C::NA / C::C1) & 1, nx_r = C::NA % C::C1;
    bool ok = true;
    for (int w = blockIdx.x; w < sc.n_items && ok; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      // segments of the item's jobs that share a state window (one slice each)
      for (int jb = j0; jb < j1 && ok;) {
        const int seg_end = min(j1, (jb / P + 1) * P);
        const int xb = xi % C::NXB;
        if (!mbar_wait(&bars->x_full[xb], (xi / C::NXB) & 1, status, 204, abort)) { ok = false; break; }
        ++xi;
        // descriptors differ from the window's first one only in the start-address field
        const uint32_t xaddr = smem_u32(xwin + xb * C::XWIN);
        const uint64_t xdesc = C::SW == 64 ? desc_sw128_mnmajor(xaddr, 1024) : desc_sw64_mnmajor(xaddr);
        for (; jb < seg_end && ok; ++jb, ++c) {
          const uint32_t d1 = tmem + C::D1COL0 + (c % C::NB) * 64;
          for (int g = 0; g < C::G; ++g, ++gi) {
            if (!mbar_wait(&bars->t_full[gi % C::NT], (gi / C::NT) & 1, status, 210, abort)) { ok = false; break; }
            tc_fence_after();
            for (int j = g * C::CG; j < (g + 1) * C::CG; ++j) {
              const uint32_t a = tmem + C::ACOL + slot * 64;
              const uint64_t jdesc = xdesc + (uint64_t)((j * C::XCHUNK) >> 4);
              // S = 32: the tile's rows couple to window columns [0, 192) only, so the last four
              // K steps of the second chunk would multiply all-zero A tiles
              const int kk_end = (S == 32 && j == C::C1 - 1) ? 4 : kTile / 16;
#pragma unroll
              for (int kk = 0; kk < kTile / 16; ++kk)
                if (leader && kk < kk_end)
                  mma_ts(d1, a + kk * 8, jdesc + (uint64_t)((kk * 16 * C::XROW) >> 4),
                         idesc, (j == 0 && kk == 0) ? 0u : 1u);
              if (leader) tc_commit(&bars->a_empty[slot][nx_g]);
              slot = slot + 1 == (uint32_t)C::NA ? 0 : slot + 1;
              if (++nx_r == (uint32_t)C::C1) { nx_r = 0; nx_g ^= 1; }
            }
          }
          if (!ok) break;
          if (leader) tc_commit(&bars->d1_full[c % C::NB]);
        }
        if (!ok) break;
        if (leader) tc_commit(&bars->x_empty[xb]);  // the segment's last job is issued
      }
    }
    drain_mmas(leader, &bars->drain);
  } else if (warp == 3) {
    // ------------------------------------------------------------------ second issuer
    // Y (+)= pre_p W_p over the jobs (kind::tf32, A = the fp32 pre_p unit in TMEM, K = the 64 rows
    // of W_p of the job's half), then the bias product
    const bool leader = elect_one_sync();
    // the bias product: in-degrees and bias halves as bf16, or as fp16 when an in-degree exceeds
    // 256 (the plan's hub rows)
    const uint32_t idesc = bias_f16 ? idesc_f16_f32(kTile, H) : idesc_bf16_f32(kTile, H);
    constexpr uint32_t idesc2 = idesc_tf32_f32(kTile, H);
    uint32_t c = 0, widx = 0, di = 0;
    bool ok = true;
    int i = 0;
    for (int w = blockIdx.x; w < sc.n_items && ok; w += gridDim.x, ++i) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      for (int jb = j0; jb < j1 && ok; ++jb, ++c) {
        const int b = c % C::NB;
        if (!mbar_wait(&bars->d1_full[b], (c / C::NB) & 1, status, 208, abort) ||
            (jb == j0 && !mbar_wait(&bars->y_empty, (i & 1) ^ 1, status, 203, abort))) {
          ok = false;
          break;
        }
        for (int wj = 0; wj < C::WJ; ++wj, ++widx) {
          const int ws = widx % C::NW;
          if (!mbar_wait(&bars->w_full[ws], (widx / C::NW) & 1, status, 202, abort)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t wbase = smem_u32(wring + ws * C::WSTAGE);
#pragma unroll
          for (int kk = 0; kk < C::WK / 8; ++kk) {
            const uint64_t bdesc = desc_sw128_kmajor(wbase + (kk / 4) * H * 128 + (kk % 4) * 32);
            if (leader) mma_ts_tf32(tmem + C::YCOL, tmem + C::D1COL0 + b * 64 + C::WK * wj + kk * 8,
                                    bdesc, idesc2, (jb == j0 && wj == 0 && kk == 0) ? 0u : 1u);
          }
          if (leader) tc_commit(&bars->w_empty[ws]);
        }
        if (!ok) break;
        // this unit is free again: part of job c + NB's first group
        if (leader) tc_commit(&bars->t_full[((c + C::NB) * C::G) % C::NT]);
      }
      if (!ok) break;
      if (has_bias && part <= 0) {
        const int db = di % C::NDEGD;
        if (!mbar_wait(&bars->deg_full[db], (di / C::NDEGD) & 1, status, 206, abort)) break;
        if (di == 0 && !mbar_wait(&bars->b2_full, 0, status, 207, abort)) break;
        ++di;
        tc_fence_after();
        const uint32_t dbase = smem_u32(degs + db * C::DEG), bbase = smem_u32(b2s);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          if (leader) mma_ss(tmem + C::YCOL, desc_sw128_kmajor(dbase + kk * 32),
                 desc_sw128_kmajor(bbase + kk * 32), idesc, 1u);
        if (leader) tc_commit(&bars->deg_empty[db]);
      }
      if (leader) tc_commit(&bars->y_full);
    }
    // a CTA whose items were all later slices of split tiles never used the bias rows it loaded:
    // let that copy land before the CTA's shared memory is released
    if (has_bias && di == 0) mbar_wait(&bars->b2_full, 0, status, 209, abort);
    drain_mmas(leader, &bars->drain2);
  } else if (warp >= 4 && warp < 4 + 4 * C::NE) {
    // ------------------------------------------------------------------ expanders
    // the two groups take the jobs in turn
    const int eg = (warp - 4) / 4;
    const int r = (threadIdx.x - 128) % 128;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    uint32_t aidx = 0, midx = 0;
    uint32_t par = 0;  // bit s: parity of this group's waits so far on A slot s
    for (int w = blockIdx.x; w < sc.n_items && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      bool ok = true;
      for (int jb = j0; jb < j1 && ok; ++jb, ++midx) {
        if ((int)(midx % C::NE) != eg) {
          aidx += C::C1;  // the other group's job
          continue;
        }
        // one chunk: wait for its A slot, expand the row's 128 bits into bf16 pairs in TMEM, and
        // after the last chunk of a group signal the band-product issuer
        auto expand_chunk = [&](int j, const uint4 m) -> bool {
          const int slot = aidx % C::NA;
          if (!mbar_wait(&bars->a_empty[slot][eg], (par >> slot) & 1, status, 301, abort))
            return false;
          par ^= 1u << slot;
          tc_fence_after();
          uint32_t v[32];
          expand_word(m.x, v);
          expand_word(m.y, v + 16);
          tmem_st32(tmem + lane_base + C::ACOL + slot * 64, v);
          expand_word(m.z, v);
          expand_word(m.w, v + 16);
          tmem_st32(tmem + lane_base + C::ACOL + slot * 64 + 32, v);
          if ((j + 1) % C::CG == 0) {
            // all of this group's A tiles are in TMEM
            tmem_wait_st();
            tc_fence_before();
            const uint32_t gi = midx * C::G + j / C::CG;
            warp_arrive(&bars->t_full[gi % C::NT]);
          }
          ++aidx;
          return true;
        };
        // this row's mask words of the job's chunks: from the staged ring, or (GM) straight from
        // global memory in groups of four chunks, the next group requested while the current one
        // is expanded (a rolled group loop keeps the code small enough for the instruction cache)
        const int ms = C::GM ? 0 : midx % C::NMD;
        if constexpr (C::GM) {
          constexpr int QG = 4;
          static_assert(C::C1 % QG == 0, "mask prefetch groups");
          const uint4* mg = reinterpret_cast<const uint4*>(maskI) +
                            ((size_t)k * P + (jb % P)) * C::C1 * kTile + r;
          uint4 cur[QG], nxt[QG];
#pragma unroll
          for (int q = 0; q < QG; ++q) cur[q] = __ldg(mg + (size_t)q * kTile);
#pragma unroll 1
          for (int g0 = 0; g0 < C::C1 && ok; g0 += QG) {
            if (g0 + QG < C::C1) {
#pragma unroll
              for (int q = 0; q < QG; ++q) nxt[q] = __ldg(mg + (size_t)(g0 + QG + q) * kTile);
            }
#pragma unroll
            for (int q = 0; q < QG; ++q)
              if (ok && !expand_chunk(g0 + q, cur[q])) ok = false;
#pragma unroll
            for (int q = 0; q < QG; ++q) cur[q] = nxt[q];
          }
        } else {
          if (!mbar_wait(&bars->m_full[ms], (midx / C::NMD) & 1, status, 302, abort, 32)) {
            ok = false;
            break;
          }
          const uint8_t* mrow = mring + ms * C::MSTAGE + r * 16;
          for (int j = 0; j < C::C1; ++j) {
            // the words are read into registers before the slot wait, so that the shared-memory
            // load overlaps it
            const uint4 m = *reinterpret_cast<const uint4*>(mrow + j * kTile * 16);
            if (!expand_chunk(j, m)) {
              ok = false;
              break;
            }
          }
        }
        if (!ok) break;
        if (!C::GM) warp_arrive(&bars->m_empty[ms]);
      }
      if (!ok) break;
    }
  } else if (warp >= 4 + 4 * C::NE) {
    // ------------------------------------------------------------------ converters / epilogue
    grid_dep_wait();  // outputs (and the accumulated dE) may still be in use by the previous kernel
    const int r = threadIdx.x - 128 * (1 + C::NE);
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    uint8_t* dms = smem + C::OFF_DM + (warp & 3) * 32 * C::XROW;
    uint32_t c = 0;
    int i = 0;
    for (int w = blockIdx.x; w < sc.n_items && !*abort; w += gridDim.x, ++i) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      const int row = k * kTile + r;
      const int asl = (!BWD && sc.addend && part < 0) ? sc.slot[row] : -1;
      bool ok = true;
      int hh = j0 / P, p = j0 - hh * P;
      for (int jb = j0; BWD && jb < j1; ++jb, ++c, p = p + 1 == P ? (++hh, 0) : p + 1) {
        const int b = c % C::NB;
        if (!mbar_wait(&bars->d1_full[b], (c / C::NB) & 1, status, 401, abort, 64)) { ok = false; break; }
        tc_fence_after();
        const uint32_t col = tmem + lane_base + C::D1COL0 + b * 64;
        uint32_t v[C::SW];
        tmem_ld32(col, v);
        if constexpr (C::SW > 32) tmem_ld32(col + 32, v + 32);
        tmem_wait_ld();
        // pre_p stays fp32 for the tf32 product: release the unit before the stores
        tc_fence_before();
        warp_arrive(&bars->t_full[((c + C::NB) * C::G) % C::NT]);
        uint32_t pk[C::SW / 2];
#pragma unroll
        for (int j = 0; j < C::SW / 2; ++j)
          pk[j] = pack_bf16(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
        if constexpr (BWD && !C::DMS) {
          // no room for a staging tile: eight lanes swap their rows' 16-byte chunks in registers, so that
          // store j of the group writes row j's slice as one whole line.  (Each lane its own row, 16
          // bytes at a time, was 6% of a GGNN backward: H = 128, 40k nodes, two steps 1,793 us a call;
          // lane pairs swapping halves 1,720; so 1,694.)
          transpose8(pk);
          uint4* d = reinterpret_cast<uint4*>(dM + ((size_t)(row - (lane & 7)) * P + p) * H + C::SW * hh) +
                     (lane & 7);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            d[(size_t)j * (P * H / 8)] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
          continue;
        }
        // dM_p (bf16, row-major) through this warp's 32-row staging tile, one bulk store per job
        // (a thread's own row as 16-byte global stores would touch 32 lines per instruction)
        if (lane == 0) tma_store_wait_read<0>();  // the previous job's copy has left the tile
        __syncwarp();
#pragma unroll
        for (int j = 0; j < C::SW / 8; ++j) {
          const int sw = C::SW == 64 ? (j ^ (lane & 7)) : (j ^ ((lane >> 1) & 3));
          *reinterpret_cast<uint4*>(dms + lane * C::XROW + sw * 16) =
              make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0)
          tma_store_2d(&tm_dm, dms, p * H + C::SW * hh, k * kTile + (warp & 3) * 32);
      }
      if (!ok) break;
      if (!mbar_wait(&bars->y_full, i & 1, status, 402, abort, 64)) break;
      tc_fence_after();
      // Y leaves TMEM in groups, each read completely before any global traffic of its own; after
      // the last group's read the next tile may start accumulating.  Up to H = 64 one group, so
      // the release does not wait on the accumulating backward's reads of the previous dE (wider
      // groups at larger H measured slower: 32 columns there)
      constexpr int YG = H <= 64 ? H : 32;
#pragma unroll
      for (int g0 = 0; g0 < H; g0 += YG) {
        uint32_t vg[YG];
        tmem_ld32(tmem + lane_base + C::YCOL + g0, vg);
        if constexpr (YG > 32) tmem_ld32(tmem + lane_base + C::YCOL + g0 + 32, vg + 32);
        tmem_wait_ld();
        if (g0 + YG >= H) {
          tc_fence_before();
          warp_arrive(&bars->y_empty);
        }
        if (asl >= 0) {
          const float* ad = sc.addend + (size_t)asl * H + g0;
#pragma unroll
          for (int j = 0; j < YG; ++j) vg[j] = __float_as_uint(__uint_as_float(vg[j]) + ad[j]);
        }
        if (C::GM && !BWD && sc.bias && part <= 0) {
          // the bias: in-degree of each type (an exact 16-bit integer) times b_p, in fp32
          const uint16_t* dr = sc.deg + (size_t)row * 64;
          for (int q = 0; q < P; ++q) {
            const uint32_t bits = dr[q];
            if (!bits) continue;
            const float d = sc.bias_f16 ? __half2float(__ushort_as_half((unsigned short)bits))
                                        : __uint_as_float(bits << 16);
            const float* bq = sc.bias + (size_t)q * H + g0;
#pragma unroll
            for (int j = 0; j < YG; ++j) vg[j] = __float_as_uint(fmaf(d, bq[j], __uint_as_float(vg[j])));
          }
        }
#pragma unroll
        for (int h1 = 0; h1 < YG; h1 += 32) {
          const int h0 = g0 + h1;
          const uint32_t* v = vg + h1;
          if (part >= 0) {
            // a slice of a split tile: its partial Y, summed with the other slices' by the fix-up
            float4* o = reinterpret_cast<float4*>(
                sc.part + ((size_t)part * sc.part_rows + (size_t)(k - sc.n_full) * kTile + r) * H + h0);
#pragma unroll
            for (int j = 0; j < 8; ++j)
              o[j] = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                 __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
            continue;
          }
          if (out) {
            float4* o = reinterpret_cast<float4*>(out + (size_t)row * H + h0);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float4 a = make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                     __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
              if (accumulate) {
                const float4 prev = o[j];
                a.x += prev.x; a.y += prev.y; a.z += prev.z; a.w += prev.w;
              }
              o[j] = a;
            }
          }
          if (outb || outT) {
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 16; ++j)
              pk[j] = pack_bf16(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
            if (outb) {
              uint4* ob = reinterpret_cast<uint4*>(outb + (size_t)row * H + h0);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                ob[j] = make_uint4(pk[4 * j], pk[4 * j + 1], pk[4 * j + 2], pk[4 * j + 3]);
            }
            if (outT) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                __nv_bfloat16* d = outT + (size_t)(h0 + 2 * j) * ld_outT + row;
                d[0] = __ushort_as_bfloat16((unsigned short)(pk[j] & 0xFFFFu));
                d[ld_outT] = __ushort_as_bfloat16((unsigned short)(pk[j] >> 16));
              }
            }
          }
        }
      }
    }
    if (BWD && lane == 0) tma_store_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------------------ gathered band
// The same products for a sparse band.  A 128-row tile of a program graph holds a few hundred
// edges per type where the dense product multiplies 128 x 128 C1 entries, so pre_p is summed
// from the edges instead: a warp takes 16 rows and the edges of one type 16 at a time,
//     pre[16 x SW] += T [16 x 16] X[16 x SW],
// where the B operand is the 16 source rows, named one by one in ldmatrix's addresses (a gather
// from the row-major window in shared memory), and T holds a 1 where an edge ends in a row.  The
// accumulator fragment is the register layout of tcgen05.st.16x256b, so pre_p goes to TMEM as the A
// operand of the second product, which is issued exactly as in k_band_tc.  A sum of a few bf16 values
// is nearly always exact in fp32, and the bias is added as the dense kernel adds it, so the results
// agree with the dense kernel's but for the rare sum that is not exact (1e-10 to 3e-7 of the norm).  A GGNN step rounds Y to bf16 and feeds it back, where even
// that grows through the layers; its saved activations and gradients do not depend on how dense a
// plan is, so the GGNN steps stay on the dense kernel.
//
// Bound: latency along each warp's chain (words, ldmatrix, products, TMEM store), with the shared-memory
// and tensor pipes each about half busy at 16 warps of 80 registers.  A step (4 ldmatrix.x4, 8 mma.sync)
// takes 26 cycles of the SM with conflict-free rows, 44 with random ones, which is why the plan deals
// edges into sets of 8 whose rows differ mod 8.  S = 512, H = 64, 131k nodes, 52 edges per node: 113 us
// against the dense kernel's 457; S = 256, H = 128, 20k nodes backward: 61 us against 89 (ncu).
//
// Roles (24 warps, one CTA per SM, persistent over the same items as k_band_tc):
//   warp 0       TMA producer: W tiles
//   warp 2       TMA producer: state windows, deg, bias
//   warp 1       TMEM allocator and issuer of the second product and the bias product
//   warps 4-7    epilogue, Y from TMEM (two accumulators, so it overlaps) and the fp32 bias
//   warps 8-23   gather: 8 warps of 16 rows for the even types, 8 for the odd ones
template <int H, bool BWD>
struct GaCfg {
  static_assert(H == 32 || H == 64 || H == 128, "state sizes with wide bands");
  static constexpr int SW = H < 64 ? 32 : 64;
  static constexpr int NH = H / SW;
  static constexpr int NT = SW / 8;                     // accumulator n-tiles
  static constexpr int YC = H < 64 ? 64 : H;            // TMEM columns of one Y
  static constexpr int NY = 2;
  static constexpr int UC = 64;                         // columns of one pre_p unit
  static constexpr int UCOL = NY * YC;
  static constexpr int NU0 = (512 - UCOL) / UC;
  static constexpr int NU = NU0 > 6 ? 6 : NU0;
  // a W stage as in k_band_tc: SW fp32 K-columns of W_p^T in 32-column atoms of H rows
  static constexpr int WSTAGE = (SW / 32) * H * 128;
  static constexpr bool BIAS = !BWD;                    // bias as a product
  static constexpr int DEG = BIAS ? kTile * 128 : 0;
  static constexpr int B2 = BIAS ? H * 128 : 0;         // the bias split, or b in fp32
  static constexpr int DM = BWD ? 16 * 16 * SW * 2 : 0; // a 16-row staging tile per gather warp
  static constexpr int FIXED = DEG + B2 + DM + 1024 + 1024;
  static constexpr int THREADS = 32 * 24;
  static_assert(NU >= 2, "pre_p units");
};

struct GaBars {
  uint64_t x_full[2], x_empty[2];
  uint64_t w_full[4], w_empty[4];
  uint64_t deg_full, deg_empty;
  uint64_t b2_full;
  uint64_t u_full[6], u_empty[6];
  uint64_t y_full[2], y_empty[2];
  uint64_t drain;
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(GaBars) <= 1024, "barriers");

// Shared-memory split of one launch: window rows (and boxes to load them in), buffers of each ring.
struct GaLayout {
  int lo, rows, box_rows, nxb, nw;
};

// Windows and W stages that fit, or nxb = 0.
template <int H, bool BWD>
GaLayout ga_layout(int lo, int rows) {
  using C = GaCfg<H, BWD>;
  GaLayout g{};
  g.lo = lo;
  g.rows = rows;
  g.box_rows = rows / ((rows + 255) / 256);  // the plan made them equal
  const int win = (rows + 8) * 128;
  // Two windows (the second hides one load per pass) with four or three W stages (their refills come
  // from L2); where that does not fit, the stages before the second window.
  constexpr int kTry[8][2] = {{2, 4}, {2, 3}, {1, 4}, {1, 3}, {2, 2}, {1, 2}, {2, 1}, {1, 1}};
  for (auto& t : kTry)
    if (t[0] * win + t[1] * C::WSTAGE + C::FIXED <= kSmemLimit) {
      g.nxb = t[0];
      g.nw = t[1];
      break;
    }
  return g;
}

__device__ __forceinline__ void ldsm4t(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void stsm4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a),
               "r"(b), "r"(c), "r"(d)
               : "memory");
}
__device__ __forceinline__ void mma16816(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma16816_first(float* c, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// accumulator fragments of 16 rows to 64 / 32 fp32 columns of TMEM
__device__ __forceinline__ void st_16x256b(uint32_t t, const float (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(t),
      "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
      "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]),
      "f"(r[16]), "f"(r[17]), "f"(r[18]), "f"(r[19]), "f"(r[20]), "f"(r[21]), "f"(r[22]),
      "f"(r[23]), "f"(r[24]), "f"(r[25]), "f"(r[26]), "f"(r[27]), "f"(r[28]), "f"(r[29]),
      "f"(r[30]), "f"(r[31])
      : "memory");
}
__device__ __forceinline__ void st_16x256b(uint32_t t, const float (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16};" ::"r"(t),
      "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
      "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
      : "memory");
}
// 16 rows x 32 fp32 columns of TMEM in the same layout
__device__ __forceinline__ void ld_16x256b(uint32_t t, float* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
        "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
      : "r"(t)
      : "memory");
}
// v[0], v[1] += d * b, as one instruction of two fused multiply-adds
__device__ __forceinline__ void fma2(float* v, float d, const float2& b) {
  asm("{\n.reg .b64 x, y, z;\nmov.b64 x, {%0, %1};\nmov.b64 y, {%2, %2};\nmov.b64 z, {%3, %4};\n"
      "fma.rn.f32x2 x, y, z, x;\nmov.b64 {%0, %1}, x;\n}"
      : "+f"(v[0]), "+f"(v[1])
      : "f"(d), "f"(b.x), "f"(b.y));
}
// One gather warp's blocks of four steps in the order of their use: the passes of the CTA's items, one
// per slice of the state.  Lane l holds the block range of pass `held` + l, so that moving on to the
// next pass touches no memory.
struct StepBlocks {
  const uint4* words;  // this lane's words of block 0
  uint32_t at, end;    // next block to request, end of its pass
  int pass, passes;    // pass of `at`, passes in all
  int held;
  uint32_t sb, se;
  __device__ __forceinline__ void fill(const Sched& sc, const uint32_t* off, int P, int jobs, int g,
                                       int b, int first, int lane) {
    int skip = first + lane, n = 0;
    held = first;
    sb = se = 0;
    for (int w = blockIdx.x; w < sc.n_items; w += gridDim.x) {
      int tile, j0, j1, part;
      item_of(sc, w, jobs, tile, j0, j1, part);
      const int h0 = j0 / P, cnt = (j1 - 1) / P - h0 + 1;
      if (skip >= 0 && skip < cnt) {
        const int jh = (h0 + skip) * P, pa = max(j0 - jh, 0), pb = min(j1 - jh, P);
        const int p0 = pa + ((pa ^ g) & 1);
        if (p0 < pb) {
          const uint32_t* o = off + ((size_t)tile * 8 + b) * (P + 1) + (g ? (P + 1) / 2 : 0) + (p0 >> 1);
          sb = o[0];
          se = o[(pb - p0 + 1) >> 1];
        }
      }
      skip -= cnt;
      n += cnt;
    }
    passes = n;
  }
  __device__ __forceinline__ uint4 request(const Sched& sc, const uint32_t* off, int P, int jobs, int g,
                                           int b, int lane) {
    while (at == end) {
      if (++pass >= passes) {
        pass = passes;
        return make_uint4(0u, 0u, 0u, 0u);  // past the end: never used
      }
      if (pass - held == 32) fill(sc, off, P, jobs, g, b, pass, lane);
      __syncwarp();
      at = __shfl_sync(0xffffffffu, sb, pass - held);
      end = __shfl_sync(0xffffffffu, se, pass - held);
    }
    return __ldg(words + (size_t)(at++) * 32);
  }
};

template <int H, bool BWD>
__global__ void __launch_bounds__(GaCfg<H, BWD>::THREADS, 1)
    k_band_gather(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w,
                  const __grid_constant__ CUtensorMap tm_deg,
                  const __grid_constant__ CUtensorMap tm_b2, const uint32_t* __restrict__ words,
                  const uint32_t* __restrict__ off, float* __restrict__ out,
                  __nv_bfloat16* __restrict__ dM, const Sched sc, const GaLayout lay, int P,
                  int has_bias, int bias_f16, int accumulate, int* status) {
  using C = GaCfg<H, BWD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int xbytes = (lay.rows + 8) * 128;
  uint8_t* xwin = smem;
  uint8_t* wring = xwin + lay.nxb * xbytes;
  uint8_t* degs = wring + lay.nw * C::WSTAGE;
  uint8_t* b2s = degs + C::DEG;
  uint8_t* dms = b2s + C::B2;
  GaBars* bars = reinterpret_cast<GaBars*>(dms + C::DM);
  volatile int* abort = &bars->abort;
  const int jobs = C::NH * P;
  const bool bias_mma = C::BIAS && has_bias;
  // the bias in fp32, added by the epilogue: b2s then holds b [P][H] (launch_gather decides)
  const bool bias32 = C::BIAS && C::SW == 64 && sc.bias != nullptr;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->x_full[i], 1); mbar_init(&bars->x_empty[i], 16);
      mbar_init(&bars->y_full[i], 1); mbar_init(&bars->y_empty[i], 4);
    }
    for (int i = 0; i < 4; ++i) { mbar_init(&bars->w_full[i], 1); mbar_init(&bars->w_empty[i], 1); }
    for (int i = 0; i < 6; ++i) { mbar_init(&bars->u_full[i], 8); mbar_init(&bars->u_empty[i], 1); }
    mbar_init(&bars->b2_full, 1);
    mbar_init(&bars->deg_full, 1);
    mbar_init(&bars->deg_empty, bias32 ? 4 : 1);
    mbar_init(&bars->drain, 1);
    bars->abort = 0;
    fence_mbar_init();
  }
  // the zero rows after each window, which padding entries name
  for (int i = threadIdx.x; i < lay.nxb * 64; i += C::THREADS)
    *reinterpret_cast<uint4*>(xwin + (i >> 6) * xbytes + lay.rows * 128 + (i & 63) * 16) =
        make_uint4(0u, 0u, 0u, 0u);
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // TMEM is held: the next kernel in the stream may be scheduled on SMs as they free up
  grid_dep_launch();
  const uint32_t tmem = bars->tmem_base;

  // let this CTA's own copies land before shared memory is released (bounded)
  auto settle = [](uint64_t* bar, uint32_t uses) {
    if (!uses) return;
    for (uint32_t t = 0; t < (1u << 22) && !mbar_try(bar, (uses - 1) & 1); ++t) {
    }
  };
  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------------ W producer
    tma_prefetch_desc(&tm_w);
    grid_dep_wait();  // W may be the previous kernel's output
    uint32_t wi = 0, wph = 0, n_w[4] = {0, 0, 0, 0};
    bool ok = true;
    for (int w = blockIdx.x; w < sc.n_items && ok && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      int hh = j0 / P, p = j0 - hh * P;
      for (int jb = j0; jb < j1 && ok; ++jb, p = p + 1 == P ? (++hh, 0) : p + 1) {
        if (!mbar_wait(&bars->w_empty[wi], (wph & 1) ^ 1, status, 153, abort)) {
          ok = false;
          break;
        }
        ++n_w[wi];
        mbar_expect_tx(&bars->w_full[wi], C::WSTAGE);
        for (int a = 0; a < C::SW / 32; ++a)
          tma_load_2d(wring + wi * C::WSTAGE + a * H * 128, &tm_w, &bars->w_full[wi],
                      C::SW * hh + 32 * a, p * H);
        if (++wi == (uint32_t)lay.nw) wi = 0, ++wph;
      }
    }
    if (*abort)
      for (int q = 0; q < 4; ++q) settle(&bars->w_full[q], n_w[q]);
  } else if (warp == 2 && lane == 0) {
    // ------------------------------------------------------------------ window producer
    // (its own thread: behind the W ring a window was requested only four jobs before its first use,
    // and the gather warps run six jobs ahead of the issuer)
    tma_prefetch_desc(&tm_x);
    // states and the bias split may be the previous kernel's output (in-degrees are plan data)
    grid_dep_wait();
    if (bias_mma) {
      mbar_expect_tx(&bars->b2_full, C::B2);
      tma_load_2d(b2s, &tm_b2, &bars->b2_full, 0, 0);
    } else if (bias32) {
      mbar_expect_tx(&bars->b2_full, (uint32_t)(P * H * 4));  // (P <= 32: no more than C::B2)
      bulk_load(b2s, sc.bias, (uint32_t)(P * H * 4), &bars->b2_full);
    }
    uint32_t xi = 0, di = 0;  // windows and deg tiles so far
    uint32_t n_x[2] = {0, 0}, n_deg = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < sc.n_items && ok && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      const int row0 = k * kTile;
      for (int jb = j0; jb < j1; jb = (jb / P + 1) * P, ++xi) {
        const int xb = lay.nxb == 2 ? (xi & 1) : 0, xn = lay.nxb == 2 ? (xi >> 1) : xi;
        if (!mbar_wait(&bars->x_empty[xb], (xn & 1) ^ 1, status, 151, abort, 32)) {
          ok = false;
          break;
        }
        ++n_x[xb];
        mbar_expect_tx(&bars->x_full[xb], lay.rows * 128);
        for (int r = 0; r < lay.rows; r += lay.box_rows)
          tma_load_2d(xwin + xb * xbytes + r * 128, &tm_x, &bars->x_full[xb], C::SW * (jb / P),
                      row0 - lay.lo + r);
      }
      if (ok && (bias_mma || bias32) && part <= 0) {
        if (!mbar_wait(&bars->deg_empty, (di & 1) ^ 1, status, 152, abort, 32)) break;
        ++n_deg;
        ++di;
        mbar_expect_tx(&bars->deg_full, C::DEG);
        tma_load_2d(degs, &tm_deg, &bars->deg_full, 0, row0);
      }
    }
    if (*abort) {
      for (int q = 0; q < 2; ++q) settle(&bars->x_full[q], n_x[q]);
      settle(&bars->deg_full, n_deg);
      if (bias_mma || bias32) settle(&bars->b2_full, 1);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ issuer
    // Y (+)= pre_p W_p over the jobs (K = the SW rows of W_p of the job's slice), then the bias
    const bool leader = elect_one_sync();
    const uint32_t idescb = bias_f16 ? idesc_f16_f32(kTile, H) : idesc_bf16_f32(kTile, H);
    constexpr uint32_t idesc = idesc_tf32_f32(kTile, H);
    uint32_t u = 0, uph = 0, wi = 0, wph = 0, di = 0;
    bool ok = true;
    int i = 0;
    for (int w = blockIdx.x; w < sc.n_items && ok; w += gridDim.x, ++i) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      const int yb = i % C::NY;
      const uint32_t ycol = tmem + yb * C::YC;
      for (int jb = j0; jb < j1 && ok; ++jb) {
        if (!mbar_wait(&bars->u_full[u], uph & 1, status, 258, abort) ||
            (jb == j0 && !mbar_wait(&bars->y_empty[yb], ((i / C::NY) & 1) ^ 1, status, 253, abort))) {
          ok = false;
          break;
        }
        const uint32_t ucol = tmem + C::UCOL + u * C::UC;
        if (!mbar_wait(&bars->w_full[wi], wph & 1, status, 252, abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t wbase = smem_u32(wring + wi * C::WSTAGE);
#pragma unroll
        for (int kk = 0; kk < C::SW / 8; ++kk)
          if (leader)
            mma_ts_tf32(ycol, ucol + kk * 8,
                        desc_sw128_kmajor(wbase + (kk / 4) * H * 128 + (kk % 4) * 32), idesc,
                        (jb == j0 && kk == 0) ? 0u : 1u);
        if (leader) tc_commit(&bars->w_empty[wi]);
        if (++wi == (uint32_t)lay.nw) wi = 0, ++wph;
        if (leader) tc_commit(&bars->u_empty[u]);
        if (++u == (uint32_t)C::NU) u = 0, ++uph;
      }
      if (!ok) break;
      if (bias_mma && part <= 0) {
        if (!mbar_wait(&bars->deg_full, di & 1, status, 256, abort)) break;
        if (di == 0 && !mbar_wait(&bars->b2_full, 0, status, 257, abort)) break;
        ++di;
        tc_fence_after();
        const uint32_t dbase = smem_u32(degs), bbase = smem_u32(b2s);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          if (leader)
            mma_ss(ycol, desc_sw128_kmajor(dbase + kk * 32), desc_sw128_kmajor(bbase + kk * 32),
                   idescb, 1u);
        if (leader) tc_commit(&bars->deg_empty);
      }
      if (leader) tc_commit(&bars->y_full[yb]);
    }
    // a CTA whose items were all later slices of split tiles never used the bias rows it loaded:
    // let that copy land before the CTA's shared memory is released
    if (bias_mma && di == 0) mbar_wait(&bars->b2_full, 0, status, 259, abort);
    drain_mmas(leader, &bars->drain);
  } else if (warp >= 4 && warp < 8) {
    // ------------------------------------------------------------------ epilogue
    // Y leaves TMEM 16 rows at a time in the fragment layout: lane l holds rows l / 4 and l / 4 + 8 and of
    // each 8 columns the pair 2 (l % 4).  Stores (and the loads of an accumulated dE) then fill whole
    // sectors, and a lane reads the bias of 8 columns for two rows from shared memory instead of 32 for
    // one.  131k nodes, S = 512, H = 64: 115 us a call with a bias and 109 without; with a row per lane 130
    // and 115, and 70 us more when the in-degrees and b came from global memory, where L1 has no room.
    // Accumulating backward at H = 64: 267 us, with a row per lane 296.
    grid_dep_wait();  // outputs (and the accumulated dE) may still be in use by the previous kernel
    const int r0 = (warp & 3) * 32 + (lane >> 2), c0 = 2 * (lane & 3);
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    int i = 0;
    uint32_t di = 0;  // in-degree tiles so far
    for (int w = blockIdx.x; w < sc.n_items && !*abort; w += gridDim.x, ++i) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      const int yb = i % C::NY;
      if (!mbar_wait(&bars->y_full[yb], (i / C::NY) & 1, status, 452, abort, 64)) break;
      tc_fence_after();
      const bool biased = bias32 && part <= 0;
      if (biased) {
        if (!mbar_wait(&bars->deg_full, di & 1, status, 453, abort, 32)) break;
        if (di == 0 && !mbar_wait(&bars->b2_full, 0, status, 454, abort, 32)) break;
        ++di;
      }
      // a slice of a split tile writes its partial Y, summed with the other slices' by the fix-up
      float* dst = part >= 0
          ? sc.part + ((size_t)part * sc.part_rows + (size_t)(k - sc.n_full) * kTile + r0) * H + c0
          : out + ((size_t)k * kTile + r0) * H + c0;
      const bool add = accumulate && part < 0;
#pragma unroll 1
      for (int g = 0; g < H / 16; ++g) {  // 16 rows x 32 columns at a time
        const int h0 = (g >> 1) * 32, rb = (g & 1) * 16;
        __syncwarp();
        float v[16];  // [8-column group][row / 8][pair]
        ld_16x256b(tmem + lane_base + ((uint32_t)rb << 16) + yb * C::YC + h0, v);
        tmem_wait_ld();
        if (g == H / 16 - 1) {
          tc_fence_before();
          warp_arrive(&bars->y_empty[yb]);
        }
        if (biased) {
          // in-degree times b_p, type by type, each a fused multiply-add (an infinite b_p reaches only the
          // rows with such an edge): two types' in-degrees per word of the swizzled tile, 0 beyond the last
          const uint8_t* dr = degs + (r0 + rb) * 128;
          const uint8_t* br = b2s + (h0 + c0) * 4;
#pragma unroll 2
          for (int q = 0; q < P; q += 2, br += 2 * H * 4) {
            uint32_t dw[2];
            float2 b[2][4];
#pragma unroll
            for (int x = 0; x < 2; ++x)  // (row & 7 is the same for both rows)
              dw[x] = *reinterpret_cast<const uint32_t*>(dr + 1024 * x + (((q >> 3) ^ (r0 & 7)) << 4) + 2 * (q & 7));
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
              for (int j = 0; j < 4; ++j) b[t][j] = *reinterpret_cast<const float2*>(br + t * H * 4 + 32 * j);
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
              for (int x = 0; x < 2; ++x) {
                const uint32_t bits = (dw[x] >> (16 * t)) & 0xFFFFu;
                if (bits) {
                  const float d = bias_f16 ? __half2float(__ushort_as_half((unsigned short)bits))
                                           : __uint_as_float(bits << 16);
#pragma unroll
                  for (int j = 0; j < 4; ++j) fma2(v + 4 * j + 2 * x, d, b[t][j]);
                }
              }
          }
          if (g == H / 16 - 1) warp_arrive(&bars->deg_empty);
        }
        float* o = dst + (size_t)rb * H + h0;
        float2 prev[2][4];
        if (add) {
#pragma unroll
          for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int j = 0; j < 4; ++j) prev[x][j] = *reinterpret_cast<const float2*>(o + 8 * x * H + 8 * j);
        }
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float2 a = make_float2(v[4 * j + 2 * x], v[4 * j + 2 * x + 1]);
            if (add) a.x += prev[x][j].x, a.y += prev[x][j].y;
            *reinterpret_cast<float2*>(o + 8 * x * H + 8 * j) = a;
          }
      }
    }
    // (as in the issuer: the bias this CTA loaded and never used must land before it ends)
    if (bias32 && di == 0) mbar_wait(&bars->b2_full, 0, status, 455, abort, 32);
  } else if (warp >= 8) {
    // ------------------------------------------------------------------ gather
    const int gw = warp - 8, g = gw >> 3;            // types of parity g
    const int b = 2 * (warp & 3) + ((gw >> 2) & 1);  // 16-row group within the tile
    const uint32_t tlane = (uint32_t)(16 * b) << 16;
    // staging tile of 16 dM_p rows, and this lane's row and chunk parity in stmatrix's x4 form
    const uint32_t dmw = smem_u32(dms) + gw * 16 * C::SW * 2;
    const int srow = (lane & 7) + (lane & 8), shi = lane >> 4;
    auto swz = [](int row, int ch) { return C::SW == 64 ? (ch ^ (row & 7)) : (ch ^ ((row >> 1) & 3)); };
    StepBlocks sb{reinterpret_cast<const uint4*>(words) + lane, 0, 0, -1, 0, 0, 0, 0};
    sb.fill(sc, off, P, jobs, g, b, 0, lane);
    uint4 nx = sb.request(sc, off, P, jobs, g, b, lane);
    uint4 nx2 = sb.request(sc, off, P, jobs, g, b, lane);
    // the unit of the last job, until its store to TMEM is known to be done: the wait is put off
    // until the next job's first products are under way
    int pending = -1;
    auto flush = [&]() {
      if (pending >= 0) {
        tmem_wait_st();
        tc_fence_before();
        warp_arrive(&bars->u_full[pending]);
        pending = -1;
      }
    };
    uint32_t u = 0, uph = 0, xi = 0;  // the next job's pre_p unit and its phase, windows so far
    auto unit_add = [&](int d) {      // d <= 2 <= NU
      u += d;
      if (u >= (uint32_t)C::NU) u -= C::NU, uph ^= 1;
    };
    bool ok = true;
    for (int w = blockIdx.x; w < sc.n_items && ok && !*abort; w += gridDim.x) {
      int k, j0, j1, part;
      item_of(sc, w, jobs, k, j0, j1, part);
      int hh = j0 / P;
      for (int jb = j0; jb < j1 && ok; ++xi, ++hh) {
        const int pa = jb - hh * P, pb = min(j1 - hh * P, P);
        const int xb = lay.nxb == 2 ? (xi & 1) : 0, xn = lay.nxb == 2 ? (xi >> 1) : xi;
        if (!mbar_wait(&bars->x_full[xb], xn & 1, status, 351, abort, 32)) { ok = false; break; }
        __syncwarp();
        const uint32_t xaddr = smem_u32(xwin + xb * xbytes);
        int p = pa + ((pa ^ g) & 1);
        unit_add(p - pa);
        bool begun = false;
        float acc[4 * C::NT];
        while (p < pb) {
          // up to four steps of 16 edges
          const uint4 cur = nx;
          nx = nx2;
          nx2 = sb.request(sc, off, P, jobs, g, b, lane);
          auto step = [&](uint32_t word, auto first) {
            const uint32_t ad = xaddr + (word & 0x3FFFFu), bits = (word >> 24) * 4097u;
            uint32_t bq[2 * C::NT], a[4];
#pragma unroll
            for (int j = 0; j < C::NT / 2; ++j) ldsm4t(bq + 4 * j, ad ^ (j << 5));
#pragma unroll
            for (int j = 0; j < 4; ++j) a[j] = expand_pair(bits, j);
#pragma unroll
            for (int j = 0; j < C::NT; ++j) {
              if constexpr (decltype(first)::value)
                mma16816_first(acc + 4 * j, a, bq[2 * j], bq[2 * j + 1]);
              else
                mma16816(acc + 4 * j, a, bq[2 * j], bq[2 * j + 1]);
            }
          };
          if (begun) {
            step(cur.x, std::false_type{});
          } else {
            step(cur.x, std::true_type{});
            flush();
          }
          const uint32_t more = (cur.x / kGatherMore) & 3u;
          if (more > 0) {
            step(cur.y, std::false_type{});
            if (more > 1) {
              step(cur.z, std::false_type{});
              if (more > 2) step(cur.w, std::false_type{});
            }
          }
          begun = true;
          if (!(cur.x & kGatherLast)) continue;
          // the type's sums of these 16 rows are complete
          begun = false;
          if constexpr (BWD) {
            // dM_p (bf16) through the warp's staging tile, so that rows leave as whole lines.  (As a
            // bulk store, the proxy fence before it waited for the words on their way.)
#pragma unroll
            for (int j = 0; j < C::NT; j += 2)
              stsm4(dmw + srow * C::SW * 2 + swz(srow, j + shi) * 16, pack_bf16(acc[4 * j], acc[4 * j + 1]),
                    pack_bf16(acc[4 * j + 2], acc[4 * j + 3]), pack_bf16(acc[4 * j + 4], acc[4 * j + 5]),
                    pack_bf16(acc[4 * j + 6], acc[4 * j + 7]));
          }
          if (!mbar_wait(&bars->u_empty[u], uph ^ 1, status, 352, abort, 32)) {
            ok = false;
            break;
          }
          __syncwarp();
          tc_fence_after();
          st_16x256b(tmem + tlane + C::UCOL + u * C::UC, acc);
          pending = (int)u;
          if constexpr (BWD) {
            constexpr int CH = C::SW / 8;  // 16-byte chunks per row
            uint4* d = reinterpret_cast<uint4*>(dM + ((size_t)(k * kTile + 16 * b) * P + p) * H + C::SW * hh);
#pragma unroll
            for (int q = 0; q < C::SW / 16; ++q) {
              const int row = (q * 32 + lane) / CH, ch = lane % CH;
              uint4 v;
              asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                           : "r"(dmw + row * C::SW * 2 + swz(row, ch) * 16)
                           : "memory");
              d[(size_t)row * (P * H / 8) + ch] = v;
            }
            __syncwarp();  // the tile is free for the next 16 rows
          }
          unit_add(min(2, pb - p));
          p += 2;
        }
        if (!ok) break;
        flush();
        warp_arrive(&bars->x_empty[xb]);
        jb += pb - pa;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------------------------ prep
// out[c][r] = bf16(in[r][c]) for an R x Cc row-major input (batched over blockIdx.z)
template <typename T>
__global__ void k_transpose_bf16(const T* __restrict__ in, __nv_bfloat16* __restrict__ out, int R,
                                 int Cc, int64_t in_batch, int64_t out_batch, int64_t ld_out) {
  __shared__ float tile[32][33];
  grid_dep_wait();
  in += blockIdx.z * in_batch;
  out += blockIdx.z * out_batch;
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
    const int r = r0 + dy, c = c0 + threadIdx.x;
    float v = 0.f;
    if (r < R && c < Cc) {
      if constexpr (sizeof(T) == 2)
        v = __bfloat162float(in[(int64_t)r * Cc + c]);
      else
        v = in[(int64_t)r * Cc + c];
    }
    tile[dy][threadIdx.x] = v;
  }
  __syncthreads();
  for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
    const int c = c0 + dy, r = r0 + threadIdx.x;
    if (c < Cc && r < R) out[(int64_t)c * ld_out + r] = __float2bfloat16_rn(tile[threadIdx.x][dy]);
  }
}

// Second-product weights in the band kernel's operand layout, for each type p:
//   forward  out[p][o][i] = W[p][i][o]   (W_p^T, K-major in i)
//   backward out[p][i][o] = W[p][i][o]   (W_p as given, K-major in o)
// as fp32 (the tf32 product's B operand).  Blocks beyond P H H / 256 do the bias split (b2T not
// NULL): one launch instead of two before every propagation.
__device__ void bias_split(const float* b, uint16_t* b2T, int P, int H, int f16, int* status, int t);
__global__ void __launch_bounds__(256) k_prep_w(const __nv_bfloat16* __restrict__ W,
                                                float* __restrict__ out, int P, int H, int transpose,
                                                const float* __restrict__ b,
                                                uint16_t* __restrict__ b2T, int f16, int* status) {
  grid_dep_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x, HH = (uint32_t)(H * H), total = (uint32_t)P * HH;
  if (t < total) {
    const uint32_t p = t / HH, r = t - p * HH, a = r / (uint32_t)H, c = r - a * (uint32_t)H;
    out[t] = __bfloat162float(transpose ? W[p * HH + c * H + a] : W[t]);
  } else if (b2T && t - total < (uint32_t)H * 64u) {
    bias_split(b, b2T, P, H, f16, status, (int)(t - total));
  }
}

// Outputs of the split tiles: Y = sum over the ksplit slices of `part` (fixed order), written like
// the band kernel's own epilogue (fp32 out, accumulating if asked; bf16 row-major; bf16
// transposed).  Rows row0 .. row0 + part_rows.
__global__ void k_band_split_fixup(const float* __restrict__ part, int ksplit, int part_rows,
                                   int row0, int H, float* __restrict__ out,
                                   __nv_bfloat16* __restrict__ outb,
                                   __nv_bfloat16* __restrict__ outT, int64_t ld_outT,
                                   int accumulate, const float* __restrict__ addend,
                                   const int32_t* __restrict__ slot) {
  grid_dep_wait();  // the partials are the band kernel's output
  const int64_t n4 = (int64_t)part_rows * H / 4, slice = (int64_t)part_rows * H;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n4;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = 4 * t;
    float4 y = *reinterpret_cast<const float4*>(part + e);
    for (int q = 1; q < ksplit; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(part + q * slice + e);
      y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
    }
    const int row = row0 + (int)(e / H), h = (int)(e % H);
    if (addend && slot[row] >= 0) {
      const float4 a = *reinterpret_cast<const float4*>(addend + (size_t)slot[row] * H + h);
      y.x += a.x; y.y += a.y; y.z += a.z; y.w += a.w;
    }
    if (out) {
      float4* o = reinterpret_cast<float4*>(out + (size_t)row * H + h);
      if (accumulate) {
        const float4 prev = *o;
        y.x += prev.x; y.y += prev.y; y.z += prev.z; y.w += prev.w;
      }
      *o = y;
    }
    const uint32_t p0 = pack_bf16(y.x, y.y), p1 = pack_bf16(y.z, y.w);
    if (outb) *reinterpret_cast<uint2*>(outb + (size_t)row * H + h) = make_uint2(p0, p1);
    if (outT) {
      outT[(size_t)h * ld_outT + row] = __ushort_as_bfloat16((unsigned short)(p0 & 0xFFFFu));
      outT[(size_t)(h + 1) * ld_outT + row] = __ushort_as_bfloat16((unsigned short)(p0 >> 16));
      outT[(size_t)(h + 2) * ld_outT + row] = __ushort_as_bfloat16((unsigned short)(p1 & 0xFFFFu));
      outT[(size_t)(h + 3) * ld_outT + row] = __ushort_as_bfloat16((unsigned short)(p1 >> 16));
    }
  }
}

// b2T[h][p] = high part of b[p][h], b2T[h][32 + p] = the remainder (zero beyond P), both bf16, or
// both fp16 (f16 != 0; the in-degrees are then fp16 too).  fp16 holds magnitudes up to 65504: a
// finite bias beyond that is recorded in the status word (code 2, site 120) and the product is
// then not to be trusted.
__device__ void bias_split(const float* __restrict__ b, uint16_t* __restrict__ b2T, int P, int H,
                           int f16, int* status, int t) {
  const int h = t / 64, q = t % 64, p = q % 32;
  float x = 0.f;
  if (p < P && b) x = b[p * H + h];
  if (f16) {
    if (fabsf(x) > 65504.f && isfinite(x) && atomicCAS(status, 0, 2) == 0) atomicExch(status + 1, 120);
    const __half hi = __float2half_rn(x);
    b2T[t] = __half_as_ushort(q < 32 ? hi : __float2half_rn(x - __half2float(hi)));
  } else {
    const __nv_bfloat16 hi = __float2bfloat16_rn(x);
    b2T[t] = __bfloat16_as_ushort(q < 32 ? hi : __float2bfloat16_rn(x - __bfloat162float(hi)));
  }
}

// ------------------------------------------------------------------------------------ host
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

bool make_map(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  return make_map_ld(m, base, rows, cols, cols, box_rows);
}

// The W map of the band kernel: fp32 (the tf32 second product), boxes of 32 columns x H rows.
bool make_map_w(CUtensorMap* m, const void* Wk, int P, int H) {
  return make_map_f32(m, Wk, (uint64_t)P * H, H, H);
}

int num_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

inline size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// State columns per pass of the band kernel (Cfg::SW) and so its jobs per tile.
int band_jobs(int H, int S, int P) {
  (void)S;
  return H / (H < 64 ? 32 : 64) * P;
}

// Work items of a launch over n_tiles tiles on `sms` SMs, one CTA per SM: whole tiles, and when
// the last round of the grid would be mostly idle, its tiles split over k in {2, 4} job ranges
// (rounds of a k-th of a tile: ceil(k tail / sms) / k).  A split tile costs extra window loads,
// partial-sum traffic and the fix-up launch, measured at about half a tile round, so the split is
// taken only when the tail then lasts less than half a round (single20k: 158 tiles on 152 SMs,
// +28%; a tail of 110 of 152 tiles split four ways measured 9% slower).
Sched make_sched(int n_tiles, int jobs, int sms, bool can_split) {
  Sched sc{};
  sc.n_items = sc.n_full = n_tiles;
  sc.ksplit = 1;
  const int full = (n_tiles / sms) * sms, tail = n_tiles - full;
  if (!can_split || tail == 0) return sc;
  int best = 1;
  double best_t = 1.0;
  for (int k = 2; k <= 4 && k <= jobs; k *= 2) {
    const double t = (double)((k * tail + sms - 1) / sms) / k;
    if (t < best_t - 1e-9) best_t = t, best = k;
  }
  if (best == 1 || best_t >= 0.5) return sc;
  sc.n_full = full;
  sc.ksplit = best;
  sc.n_items = full + best * tail;
  sc.part_rows = tail * kTile;
  return sc;
}

template <int H, int S, bool BWD>
cudaError_t launch_s(const bg_plan* p, const CUtensorMap& tx, const CUtensorMap& tw,
                     const CUtensorMap& tdeg, const CUtensorMap& tb2, const CUtensorMap& tdm,
                     float* out, __nv_bfloat16* outb, __nv_bfloat16* outT, int64_t ld_outT,
                     __nv_bfloat16* dM, int has_bias, int accumulate,
                     float* split, const float* addend, const float* b32, int* status,
                     cudaStream_t st) {
  using C = Cfg<H, S, BWD>;
  cudaError_t e = cudaFuncSetAttribute(k_band_tc<H, S, BWD>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
  if (e != cudaSuccess) return e;
  const int n_tiles = p->n_pad() / kTile, sms = num_sms();
  Sched sc = make_sched(n_tiles, C::NH * p->P, sms, split != nullptr);
  sc.part = split;
  sc.addend = BWD ? nullptr : addend;
  sc.slot = p->d_sin_slot;
  sc.deg = reinterpret_cast<const uint16_t*>(p->d_deg2);
  sc.bias = (C::GM && !BWD && has_bias) ? b32 : nullptr;
  sc.bias_f16 = p->max_deg > 256 ? 1 : 0;
  const int grid = std::min(sc.n_items, sms);
  e = launch_pdl(k_band_tc<H, S, BWD>, dim3(grid), dim3(C::THREADS), C::SMEM, st, tx, tw, tdeg,
                 tb2, tdm, BWD ? p->d_maskTI : p->d_maskI, out, outb, outT, ld_outT, dM, sc,
                 p->P, has_bias, p->max_deg > 256 ? 1 : 0, accumulate, status);
  note_launch();
  if (e != cudaSuccess || sc.ksplit == 1) return e;
  const int64_t n4 = (int64_t)sc.part_rows * H / 4;
  e = launch_pdl(k_band_split_fixup, dim3((unsigned)std::min<int64_t>((n4 + 255) / 256, 2048)),
                 dim3(256), 0, st, (const float*)split, sc.ksplit, sc.part_rows,
                 sc.n_full * kTile, H, out, outb, outT, ld_outT, accumulate, sc.addend, sc.slot);
  note_launch();
  return e;
}

// The shapes with a tensor-core kernel: H in {32, 64, 128} at S in {32, 64, 128, 256, 512}; H = 256
// at S in {32, 64, 128} (its state-slice window at S = 256 leaves no room for the mask ring).
template <int H, bool BWD>
cudaError_t launch(const bg_plan* p, const CUtensorMap& tx, const CUtensorMap& tw,
                   const CUtensorMap& tdeg, const CUtensorMap& tb2, const CUtensorMap& tdm,
                   float* out, __nv_bfloat16* outb, __nv_bfloat16* outT, int64_t ld_outT,
                   __nv_bfloat16* dM, int has_bias, int accumulate, float* split,
                   const float* addend, const float* b32, int* status, cudaStream_t st) {
#define BG_BAND_S(SV)                                                                            \
  return launch_s<H, SV, BWD>(p, tx, tw, tdeg, tb2, tdm, out, outb, outT, ld_outT, dM, has_bias, \
                              accumulate, split, addend, b32, status, st);
  switch (p->S) {
    case 32: BG_BAND_S(32)
    case 64: BG_BAND_S(64)
    case 256:
      if constexpr (H <= 128) { BG_BAND_S(256) }
      return cudaErrorInvalidValue;
    case 512:
      if constexpr (H <= 128) { BG_BAND_S(512) }
      return cudaErrorInvalidValue;
    default: BG_BAND_S(128)
  }
#undef BG_BAND_S
}

// Operands of a launch of the gathered kernel (band_tc.h gives their meanings).
struct GaOps {
  const __nv_bfloat16* X;
  const void* Wk;
  const __nv_bfloat16* b2T;
  const float* b32;
  float* out;
  __nv_bfloat16* dM;
  int accumulate;
  float* split;
};

template <int H, bool BWD>
cudaError_t launch_gather(const bg_plan* p, const GaOps& o, int* status, cudaStream_t st) {
  using C = GaCfg<H, BWD>;
  const int n = p->n_pad(), P = p->P;
  const GaLayout lay = ga_layout<H, BWD>(p->g_lo[BWD], p->g_rows[BWD]);
  if (!lay.nxb) return cudaErrorInvalidValue;
  CUtensorMap tx, tw, tdeg, tb2;
  if (!make_map_ld(&tx, o.X, n, H, H, lay.box_rows) ||
      !make_map_w(&tw, o.Wk, P, H))
    return cudaErrorInvalidValue;
  // the bias in fp32 from the epilogue wherever the dense kernel adds it so (Cfg::GM), else as a product
  const bool bias32 = !BWD && o.b32 && bias_in_fp32(p->S, C::SW);
  const bool bias_mma = C::BIAS && o.b2T != nullptr && !bias32;
  tdeg = tb2 = tx;
  if ((bias_mma || bias32) && !make_map(&tdeg, p->d_deg2, n, 64, kTile)) return cudaErrorInvalidValue;
  if (bias_mma && !make_map(&tb2, o.b2T, H, 64, H)) return cudaErrorInvalidValue;
  const int smem = lay.nxb * (lay.rows + 8) * 128 + lay.nw * C::WSTAGE + C::FIXED;
  // the attribute belongs to the kernel, not to this launch: with the plan's own size, a thread with a
  // smaller plan could lower it between another thread's setting and launch
  cudaError_t e = cudaFuncSetAttribute(k_band_gather<H, BWD>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit);
  if (e != cudaSuccess) return e;
  const int sms = num_sms();
  Sched sc = make_sched(n / kTile, C::NH * P, sms, o.split != nullptr);
  sc.part = o.split;
  sc.bias = bias32 ? o.b32 : nullptr;
  e = launch_pdl(k_band_gather<H, BWD>, dim3(std::min(sc.n_items, sms)), dim3(C::THREADS),
                 smem, st, tx, tw, tdeg, tb2, (const uint32_t*)p->d_glist[BWD],
                 (const uint32_t*)p->d_goff[BWD], o.out, o.dM, sc, lay, P, bias_mma ? 1 : 0,
                 p->max_deg > 256 ? 1 : 0, o.accumulate, status);
  note_launch();
  if (e != cudaSuccess || sc.ksplit == 1) return e;
  const int64_t n4 = (int64_t)sc.part_rows * H / 4;
  e = launch_pdl(k_band_split_fixup, dim3((unsigned)std::min<int64_t>((n4 + 255) / 256, 2048)),
                 dim3(256), 0, st, (const float*)o.split, sc.ksplit, sc.part_rows,
                 sc.n_full * kTile, H, o.out, (__nv_bfloat16*)nullptr, (__nv_bfloat16*)nullptr, (int64_t)0,
                 o.accumulate, (const float*)nullptr, (const int32_t*)nullptr);
  note_launch();
  return e;
}

template <bool BWD>
cudaError_t launch_gather_h(const bg_plan* p, int H, const GaOps& o, int* status, cudaStream_t st) {
  switch (H) {
    case 32: return launch_gather<32, BWD>(p, o, status, st);
    case 64: return launch_gather<64, BWD>(p, o, status, st);
    case 128: return launch_gather<128, BWD>(p, o, status, st);
    default: return cudaErrorInvalidValue;
  }
}

template <bool BWD>
bool gather_fits(int lo, int rows, int H) {
  switch (H) {
    case 32: return ga_layout<32, BWD>(lo, rows).nxb > 0;
    case 64: return ga_layout<64, BWD>(lo, rows).nxb > 0;
    case 128: return ga_layout<128, BWD>(lo, rows).nxb > 0;
    default: return false;
  }
}

// The average number of gather steps per (tile, type) up to which the edge lists are used (0: never).
// The gathered kernel's time follows the steps and hardly the block size, the dense one's follows the
// window's chunks and not the edges.  Measured on 48 graphs, 61.7k nodes, 20 types, at 20 and 160
// edges per node, lists against chunks in us a launch: S = 256 forward 34 and 68 against 93 (H = 32),
// 49 and 104 against 101 (64), 94 and 211 against 225 (128), backward 47 and 76 against 95, 65 and 115
// against 103, 125 and 238 against 222; S = 512 forward 37 and 74 against 183, 50 and 107 against 225,
// 100 and 214 against 495, backward 50 and 82 against 186, 68 and 120 against 187, 146 and 241 against
// 560.  The entries lie where the measured lines cross, or at S = 512 at half the distance beyond the
// last measured point (about 80 steps); there, at 20k nodes and about 150 steps, the lists still take 60 us
// a call against 80 at H = 32, 87 against 105 at H = 64 and 158 against 218 at H = 128 forward, 89 against
// 107 and 238 against 300 backward at H = 32 and 128.  At S = 128 the two are within 7% of one another at H = 64 and
// 52 edges per node, and the lists are not built there.
int gather_max_steps(int S, int H, bool bwd) {
  if (S != 256 && S != 512) return 0;
  const int h = H == 32 ? 0 : H == 64 ? 1 : 2;
  static constexpr int kMax[2][2][3] = {{{100, 70, 80}, {80, 60, 68}},      // S = 256
                                        {{200, 160, 200}, {200, 110, 200}}};  // S = 512
  return kMax[S == 512][bwd][h];
}

// Shapes whose propagation runs on the fused tensor-core kernels (and rounds where they round).
bool tc_shape_ok(int S, int H) {
  return ((H == 32 || H == 64 || H == 128) &&
          (S == 32 || S == 64 || S == 128 || S == 256 || S == 512)) ||
         (H == 256 && (S == 32 || S == 64 || S == 128));
}

}  // namespace

// Row-major fp32 [rows][cols], boxes of 32 columns (one 128-byte swizzle row) x box_rows.
bool make_map_f32(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols,
                  uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 4};
  cuuint32_t box[2] = {32, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool make_map_ld(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
                 uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool make_map_box(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
                  uint32_t box_cols, uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn || (box_cols != 64 && box_cols != 32)) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {box_cols, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  box_cols == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

int gemm_tn_num_sms() { return num_sms(); }

bool make_map_3d(CUtensorMap* m, const void* base, uint64_t batch, uint64_t rows, uint64_t cols,
                 uint64_t ld, uint64_t sbatch, uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {cols, rows, batch};
  cuuint64_t strides[2] = {ld * 2, sbatch * 2};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool band_tc_supported(const bg_plan* p, int dtype, int H) {
  if (!p || dtype != 1 || p->P > 32 || p->n_pad() % kTile || !tc_shape_ok(p->S, H)) return false;
  return p->d_maskI && p->d_maskTI && p->d_deg2 && p->max_deg < 2048 && encode_fn() != nullptr;
}

namespace {
bool use_lists(const bg_plan* p, int H, bool bwd) { return p->list_h[bwd] >> (H / 32) & 1; }
}  // namespace

bool band_tc_uses_lists(const bg_plan* p, int dtype, int H, bool bwd) {
  return band_tc_supported(p, dtype, H) && use_lists(p, H, bwd);
}

size_t band_tc_w_bytes(const bg_plan* p, int H) {
  return al256((size_t)p->P * H * H * 4);
}

cudaError_t band_tc_prep_w(const bg_plan* p, int H, const void* W, int bwd, void* Wk,
                           const float* b, __nv_bfloat16* b2T, int* status, cudaStream_t st) {
  const int64_t n = (int64_t)p->P * H * H + (b ? H * 64 : 0);
  cudaError_t e = launch_pdl(k_prep_w, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, st,
                             static_cast<const __nv_bfloat16*>(W), static_cast<float*>(Wk), p->P, H,
                             bwd ? 0 : 1, b, b ? reinterpret_cast<uint16_t*>(b2T) : nullptr,
                             p->max_deg > 256 ? 1 : 0, status);
  note_launch();
  return e;
}

// (The first n H bf16 elements are not used; the size is what callers have always been asked for,
// and what the allocation-free entry point's limit is checked against.)
size_t band_tc_fwd_ws_bytes(const bg_plan* p, int dtype, int H) {
  if (!p || dtype != 1) return 0;
  const size_t n = (size_t)p->n_pad();
  return al256(n * H * 2) + band_tc_w_bytes(p, H) + al256((size_t)H * 64 * 2) +
         al256(sizeof(float) * band_tc_split_floats(p, H));
}

size_t band_tc_bwd_ws_bytes(const bg_plan* p, int dtype, int H) {
  if (!p || dtype != 1) return 0;
  const size_t n = (size_t)p->n_pad();
  return al256(n * H * 2) + al256((size_t)p->P * H * n * 2) + al256((size_t)(H + 16) * n * 2) +
         band_tc_w_bytes(p, H) +
         al256(sizeof(float) * gemm_tn_part_floats(p->P * H, H + 16, (int64_t)n)) +
         al256(sizeof(float) * band_tc_split_floats(p, H));
}

size_t band_tc_split_floats(const bg_plan* p, int H) {
  const Sched sc = make_sched(p->n_pad() / kTile, band_jobs(H, p->S, p->P), num_sms(), true);
  return sc.ksplit > 1 ? (size_t)sc.ksplit * sc.part_rows * H : 0;
}

cudaError_t band_tc_fwd_core(const bg_plan* p, int H, const __nv_bfloat16* X, const void* Wk,
                             const __nv_bfloat16* b2T, const float* b32, float* out,
                             __nv_bfloat16* outb, __nv_bfloat16* outT, int64_t ld_outT,
                             float* split, const float* addend, int* status, cudaStream_t st,
                             bool lists) {
  const int n = p->n_pad(), P = p->P;
  if (lists && use_lists(p, H, false) && !outb && !outT && !addend)
    return launch_gather_h<false>(p, H, GaOps{X, Wk, b2T, b32, out, nullptr, 0, split}, status, st);
  CUtensorMap tx, tw, tdeg, tb2;
  if (!make_map_box(&tx, X, n, H, H, H < 64 ? 32 : 64, kTile) ||
      !make_map_w(&tw, Wk, P, H) || !make_map(&tdeg, p->d_deg2, n, 64, kTile) ||
      !make_map(&tb2, b2T ? b2T : X, H, 64, H))
    return cudaErrorInvalidValue;
  const int hb = b2T != nullptr;
#define BG_FWD(HV)                                                                                \
  return launch<HV, false>(p, tx, tw, tdeg, tb2, tw, out, outb, outT, ld_outT, nullptr, hb, 0,    \
                           split, addend, b32, status, st);
  switch (H) {
    case 32: BG_FWD(32)
    case 64: BG_FWD(64)
    case 128: BG_FWD(128)
    default: BG_FWD(256)
  }
#undef BG_FWD
}

cudaError_t band_tc_bwd_core(const bg_plan* p, int H, const __nv_bfloat16* dY, const void* Wk,
                             float* dE, int accumulate, __nv_bfloat16* dM, float* split,
                             int* status, cudaStream_t st, bool lists) {
  const int n = p->n_pad(), P = p->P;
  if (lists && use_lists(p, H, true))
    return launch_gather_h<true>(p, H, GaOps{dY, Wk, nullptr, nullptr, dE, dM, accumulate, split},
                                 status, st);
  CUtensorMap tx, tw, tdm;
  const int sw = H < 64 ? 32 : 64;
  if (!make_map_box(&tx, dY, n, H, H, sw, kTile) || !make_map_w(&tw, Wk, P, H) ||
      !make_map_box(&tdm, dM, n, (uint64_t)P * H, (uint64_t)P * H, sw, 32))
    return cudaErrorInvalidValue;
#define BG_BWD(HV)                                                                                \
  return launch<HV, true>(p, tx, tw, tw, tw, tdm, dE, nullptr, nullptr, 0, dM, 0, accumulate,     \
                          split, nullptr, nullptr, status, st);
  switch (H) {
    case 32: BG_BWD(32)
    case 64: BG_BWD(64)
    case 128: BG_BWD(128)
    default: BG_BWD(256)
  }
#undef BG_BWD
}

cudaError_t prep_transpose_bf16(const void* in, int in_is_f32, __nv_bfloat16* out, int R, int Cc,
                                int batch, cudaStream_t st, int64_t ld_out) {
  dim3 grid((Cc + 31) / 32, (R + 31) / 32, batch);
  if (ld_out <= 0) ld_out = R;
  const int64_t sb = (int64_t)R * Cc;
  cudaError_t e;
  if (in_is_f32)
    e = launch_pdl(k_transpose_bf16<float>, grid, dim3(32, 8), 0, st, static_cast<const float*>(in),
                   out, R, Cc, sb, sb, ld_out);
  else
    e = launch_pdl(k_transpose_bf16<__nv_bfloat16>, grid, dim3(32, 8), 0, st,
                   static_cast<const __nv_bfloat16*>(in), out, R, Cc, sb, sb, ld_out);
  note_launch();
  return e;
}

cudaError_t band_tc_fwd(const bg_plan* p, int H, const void* E, const void* W, const float* b,
                        float* Y, char* ws, size_t ws_bytes, int* status, cudaStream_t st,
                        bool lists) {
  if (ws_bytes < band_tc_fwd_ws_bytes(p, 1, H)) return cudaErrorInvalidValue;
  const int n = p->n_pad();
  void* WT = ws + al256((size_t)n * H * 2);
  __nv_bfloat16* b2T = reinterpret_cast<__nv_bfloat16*>(ws + al256((size_t)n * H * 2) +
                                                        band_tc_w_bytes(p, H));
  float* split = reinterpret_cast<float*>(ws + al256((size_t)n * H * 2) + band_tc_w_bytes(p, H) +
                                          al256((size_t)H * 64 * 2));
  // W_p [H_in][H_out] -> W_p^T in the kernel's operand type;  bias split
  cudaError_t e = band_tc_prep_w(p, H, W, 0, WT, b, b2T, status, st);
  if (e != cudaSuccess) return e;
  ProfSpan span(BG_KID_BAND_FWD, st);
  return band_tc_fwd_core(p, H, static_cast<const __nv_bfloat16*>(E), WT, b ? b2T : nullptr, b, Y,
                          nullptr, nullptr, 0, band_tc_split_floats(p, H) ? split : nullptr, nullptr, status, st,
                          lists);
}

cudaError_t band_tc_bwd(const bg_plan* p, int H, const void* E, const void* W, const float* dY,
                        float* dE, float* dW, float* db, int accum, char* ws, size_t ws_bytes,
                        int* status, cudaStream_t st, bool lists) {
  if (ws_bytes < band_tc_bwd_ws_bytes(p, 1, H)) return cudaErrorInvalidValue;
  const int n = p->n_pad(), P = p->P;
  size_t o = 0;
  __nv_bfloat16* dYb = reinterpret_cast<__nv_bfloat16*>(ws + o);
  o += al256((size_t)n * H * 2);
  __nv_bfloat16* dM = reinterpret_cast<__nv_bfloat16*>(ws + o);
  o += al256((size_t)P * H * n * 2);
  __nv_bfloat16* ETa = reinterpret_cast<__nv_bfloat16*>(ws + o);
  o += al256((size_t)(H + 16) * n * 2);
  void* Wk = ws + o;
  o += band_tc_w_bytes(p, H);
  float* part = reinterpret_cast<float*>(ws + o);
  const size_t part_floats = gemm_tn_part_floats(P * H, H + 16, (int64_t)n);
  o += al256(sizeof(float) * part_floats);
  float* split = band_tc_split_floats(p, H) ? reinterpret_cast<float*>(ws + o) : nullptr;
  cudaError_t e = f32_to_bf16(dY, dYb, (int64_t)n * H, st);
  if (e == cudaSuccess) e = band_tc_prep_w(p, H, W, 1, Wk, nullptr, nullptr, status, st);
  if (e == cudaSuccess) {
    ProfSpan span(BG_KID_BAND_BWD, st);
    e = band_tc_bwd_core(p, H, dYb, Wk, dE, accum, dM, split, status, st, lists);
  }
  if (e != cudaSuccess) return e;
  // E^T; the weight-gradient product appends its ones row, which turns the bias gradient into
  // column H of the same product
  e = prep_transpose_bf16(E, 0, ETa, n, H, 1, st);
  if (e != cudaSuccess) return e;
  // dW_p[h][h'] (+)= sum_nodes E[node][h] dM_p[node][h'],  db_p[h'] (+)= sum_nodes dM_p[node][h']
  ProfSpan span(BG_KID_DW, st);
  return gemm_tn(dM, (int64_t)P * H, 1, ETa, n, P * H, H, n, 1, dW, db, accum, part, part_floats,
                 status, st);
}

namespace {
template <typename T>
bool upload_to(const std::vector<T>& v, T** d, cudaStream_t st) {
  const size_t bytes = v.size() * sizeof(T);
  return cudaMalloc(d, std::max<size_t>(bytes, 16)) == cudaSuccess &&
         (bytes == 0 || cudaMemcpyAsync(*d, v.data(), bytes, cudaMemcpyHostToDevice, st) == cudaSuccess);
}
}  // namespace

static cudaError_t upload_lists(bg_plan* p, cudaStream_t st) {
  const int S = p->S;
  const double cells = (double)(p->n_pad() / kTile) * p->P;  // (tile, type) pairs
  uint32_t want[2] = {0, 0};
  // state sizes whose rule `steps` gather steps per (tile, type) meet
  auto rule = [&](int d, double steps) {
    uint32_t w = 0;
    for (int H : {32, 64, 128})
      if (steps <= gather_max_steps(S, H, d)) w |= 1u << (H / 32);
    return w;
  };
  unsigned dirs = 0;
  for (int d = 0; d < 2; ++d)
    if (rule(d, std::max(8.0, (double)p->band_edges / 16 / cells))) dirs |= 1u << d;  // full steps at best
  if (!dirs) return cudaSuccess;
  // the edges per (tile, group, type) counted on the device, in the place of their offsets
  const size_t n_off = (size_t)p->n_pad() / 16 * (p->P + 1), off_bytes = al256(n_off * 4);
  auto alloc = [](char** d, size_t bytes) {
    if (cudaMalloc(d, bytes) == cudaSuccess) return true;
    *d = nullptr;
    cudaGetLastError();  // taken off the runtime's record: the caller goes on without lists
    return false;
  };
  if (!alloc(&p->d_list_off, 2 * off_bytes + 256)) return cudaErrorMemoryAllocation;
  int* d_reach = reinterpret_cast<int*>(p->d_list_off + 2 * off_bytes);
  cudaError_t e = cudaMemsetAsync(d_reach, 0, 16, st);
  int reach[4];
  GatherLists l[2];
  for (int d = 0; d < 2 && e == cudaSuccess; ++d) {
    if (!(dirs >> d & 1)) continue;
    p->d_goff[d] = reinterpret_cast<uint32_t*>(p->d_list_off + d * off_bytes);
    l[d].off.resize(n_off);
    e = list_count(p, d, p->d_goff[d], d_reach + 2 * d, st);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(l[d].off.data(), p->d_goff[d], n_off * 4, cudaMemcpyDeviceToHost, st);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(reach, d_reach, 16, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  size_t at[2], bytes = 0;
  for (int d = 0; d < 2; ++d) {
    if (!(dirs >> d & 1)) continue;
    list_layout(p, reach + 2 * d, l[d]);
    want[d] = (l[d].blocks >> 31) ? 0 : rule(d, (double)l[d].steps / cells);
    for (int H : {32, 64, 128})
      if (!(d ? gather_fits<true>(l[d].lo, l[d].rows, H) : gather_fits<false>(l[d].lo, l[d].rows, H)))
        want[d] &= ~(1u << (H / 32));
    if (!want[d]) {
      dirs &= ~(1u << d);
      continue;
    }
    at[d] = bytes;
    bytes += al256((size_t)l[d].blocks * 32 * kGatherBlock * 4);
  }
  if (!dirs) return cudaSuccess;
  if (!alloc(&p->d_lists, bytes)) return cudaErrorMemoryAllocation;
  for (int d = 0; d < 2 && e == cudaSuccess; ++d) {
    if (!(dirs >> d & 1)) continue;
    p->d_glist[d] = reinterpret_cast<uint32_t*>(p->d_lists + at[d]);
    p->g_lo[d] = l[d].lo;
    p->g_rows[d] = l[d].rows;
    e = cudaMemcpyAsync(p->d_goff[d], l[d].off.data(), n_off * 4, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = list_emit(p, d, p->d_goff[d], l[d].lo, l[d].rows, p->d_glist[d], st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  for (int d = 0; d < 2; ++d) p->list_h[d] = want[d];
  return cudaSuccess;
}

static void free_lists(bg_plan* p) {
  cudaFree(p->d_lists);
  cudaFree(p->d_list_off);
  p->d_lists = p->d_list_off = nullptr;
  for (int d = 0; d < 2; ++d) p->d_glist[d] = p->d_goff[d] = nullptr;
  p->list_h[0] = p->list_h[1] = 0;
}

cudaError_t band_tc_upload_lists(bg_plan* p, cudaStream_t st) {
  if (!p->d_deg2 || p->max_deg >= 2048) return cudaSuccess;  // no tensor-core path
  cudaError_t e = cudaErrorMemoryAllocation;
  try {
    e = upload_lists(p, st);
  } catch (const std::bad_alloc&) {
  }
  if (!p->list_h[0] && !p->list_h[1]) free_lists(p);
  return e == cudaErrorMemoryAllocation ? cudaSuccess : e;
}

int band_tc_upload(bg_plan* p, cudaStream_t st) {
  const int S = p->S;
  if (p->P > 32 || (S != 32 && S != 64 && S != 128 && S != 256 && S != 512)) return 0;
  const size_t n = (size_t)p->K * S;
  if (n % kTile) return 0;
  std::vector<uint16_t> deg;
  p->max_deg = band_tc_host_degrees(p, deg, &p->band_edges);
  if (!upload_to(deg, &p->d_deg2, st)) return -1;
  const size_t words = n / kTile * p->P * band_chunks(S) * kTile * 4;
  for (int d = 0; d < 2; ++d) {
    std::unique_ptr<uint32_t[]> m(new uint32_t[words]);
    band_tc_host_chunks(p, band_chunks(S), d, m.get());
    uint32_t** dst = d ? &p->d_maskTI : &p->d_maskI;
    if (cudaMalloc(dst, std::max<size_t>(words * 4, 16)) != cudaSuccess ||
        cudaMemcpyAsync(*dst, m.get(), words * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return -1;
  }
  return cudaStreamSynchronize(st) == cudaSuccess ? 0 : -1;
}

cudaError_t band_tc_preload_fwd(const bg_plan* p) {
  if (!encode_fn()) return cudaErrorNotSupported;
  cudaFuncAttributes a;
  cudaError_t e = cudaSuccess;
  auto take = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  take(cudaFuncGetAttributes(&a, k_prep_w));
  take(cudaFuncGetAttributes(&a, k_band_split_fixup));
#define BG_PRELOAD(HV, SV) take(cudaFuncGetAttributes(&a, k_band_tc<HV, SV, false>));
#define BG_PRELOAD_S(SV) BG_PRELOAD(32, SV) BG_PRELOAD(64, SV) BG_PRELOAD(128, SV)
  switch (p->S) {
    case 32: BG_PRELOAD_S(32) BG_PRELOAD(256, 32) break;
    case 64: BG_PRELOAD_S(64) BG_PRELOAD(256, 64) break;
    case 128: BG_PRELOAD_S(128) BG_PRELOAD(256, 128) break;
    case 256: BG_PRELOAD_S(256) break;
    case 512: BG_PRELOAD_S(512) break;
    default: break;
  }
#undef BG_PRELOAD_S
#undef BG_PRELOAD
  take(cudaFuncGetAttributes(&a, k_band_gather<32, false>));
  take(cudaFuncGetAttributes(&a, k_band_gather<64, false>));
  take(cudaFuncGetAttributes(&a, k_band_gather<128, false>));
  return e;
}

void band_tc_release(bg_plan* p) {
  cudaFree(p->d_maskI);
  cudaFree(p->d_maskTI);
  cudaFree(p->d_deg2);
  free_lists(p);
  p->d_maskI = p->d_maskTI = nullptr;
  p->d_deg2 = nullptr;
}

}  // namespace bg
