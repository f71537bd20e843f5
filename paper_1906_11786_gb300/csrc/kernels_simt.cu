// SIMT kernels of the band-GGNN path: generic strided GEMM, band aggregation over bit tiles,
// GRU gates, layout conversion, readout and Adam.  Every kernel is bounds-checked by its index
// arithmetic; none waits on another block.
#include <atomic>
#include <type_traits>

#include "kernels.h"
#include "tc_util.cuh"

namespace bg {

using tc::grid_dep_wait;

static std::atomic<long long> g_launches{0};
void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
long long launch_total() { return g_launches.load(); }

namespace {

__device__ __forceinline__ float ld(const float* p, int64_t i) { return p[i]; }
__device__ __forceinline__ float ld(const __nv_bfloat16* p, int64_t i) {
  return __bfloat162float(p[i]);
}
__device__ __forceinline__ void st(float* p, int64_t i, float v) { p[i] = v; }
__device__ __forceinline__ void st(__nv_bfloat16* p, int64_t i, float v) {
  p[i] = __float2bfloat16_rn(v);
}

inline int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b > (1 << 20)) b = 1 << 20;
  return (int)(b < 1 ? 1 : b);
}

// ------------------------------------------------------------------------------------ GEMM
constexpr int GK = 16;   // k step

// 16 TM x 16 TN tile, TM x TN outputs per thread.  The next K step's operands are on their way in
// registers while the current one is multiplied from shared memory (two buffers, one barrier a step):
// with the loads in front of each step the loop was latency-bound (four 512 x 64 x 64 products 15.4 us
// against 8.2, ncu).  Eight rows a thread do 32 or 48 FMAs per 3 or 3.5 16-byte shared loads instead of
// 16 per 2; six columns fit a width of 96 without an idle quarter (a two-step fp32 batch of 3,001 nodes
// at H = 96, mostly these products: 157 us a pass with 4 x 4, 137 so).
template <int N>
__device__ __forceinline__ void lds_vec(float (&v)[N], const float* p) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 x = *reinterpret_cast<const float4*>(p + i);
      v[i] = x.x; v[i + 1] = x.y; v[i + 2] = x.z; v[i + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < N; i += 2) {
      const float2 x = *reinterpret_cast<const float2*>(p + i);
      v[i] = x.x; v[i + 1] = x.y;
    }
  }
}

template <int TM, int TN, typename TA, typename TB>
__global__ void __launch_bounds__(256) k_gemm(Gemm g, int splits, int kchunk, float* part) {
  constexpr int BM = 16 * TM, BN = 16 * TN;
  __shared__ __align__(16) float As[2][GK][BM + 4];
  __shared__ __align__(16) float Bs[2][GK][BN + 4];
  grid_dep_wait();
  const TA* A = static_cast<const TA*>(g.A);
  const TB* B = static_cast<const TB*>(g.B);
  const int b = blockIdx.z / splits, s = blockIdx.z % splits;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int kbeg = s * kchunk;
  const int kend = min(g.K, kbeg + kchunk);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const bool a_k_fast = (g.sAk == 1);
  const bool b_n_fast = (g.sBn == 1);
  float acc[TM][TN];
#pragma unroll
  for (int r = 0; r < TM; ++r)
#pragma unroll
    for (int c = 0; c < TN; ++c) acc[r][c] = 0.f;
  float ra[TM], rb[TN];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < TM; ++q) {
      const int idx = tid + 256 * q;
      const int am = a_k_fast ? idx / GK : idx % BM, ak = a_k_fast ? idx % GK : idx / BM;
      const int m = m0 + am, k = k0 + ak;
      ra[q] = (m < g.M && k < kend) ? ld(A, b * g.sAb + m * g.sAm + k * g.sAk) : 0.f;
    }
#pragma unroll
    for (int q = 0; q < TN; ++q) {
      const int idx = tid + 256 * q;
      const int bn = b_n_fast ? idx % BN : idx / GK, bk = b_n_fast ? idx / BN : idx % GK;
      const int n = n0 + bn, k = k0 + bk;
      rb[q] = (n < g.N && k < kend) ? ld(B, b * g.sBb + k * g.sBk + n * g.sBn) : 0.f;
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < TM; ++q) {
      const int idx = tid + 256 * q;
      As[buf][a_k_fast ? idx % GK : idx / BM][a_k_fast ? idx / GK : idx % BM] = ra[q];
    }
#pragma unroll
    for (int q = 0; q < TN; ++q) {
      const int idx = tid + 256 * q;
      Bs[buf][b_n_fast ? idx / BN : idx % GK][b_n_fast ? idx % BN : idx / GK] = rb[q];
    }
  };
  if (kbeg < kend) {
    fetch(kbeg);
    stage(0);
  }
  __syncthreads();
  for (int k0 = kbeg, buf = 0; k0 < kend; k0 += GK, buf ^= 1) {
    const bool more = k0 + GK < kend;
    if (more) fetch(k0 + GK);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      float a[TM], bb[TN];
      lds_vec(a, &As[buf][kk][ty * TM]);
      lds_vec(bb, &Bs[buf][kk][tx * TN]);
#pragma unroll
      for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) acc[r][c] += a[r] * bb[c];
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int r = 0; r < TM; ++r) {
    int m = m0 + ty * TM + r;
    if (m >= g.M) continue;
#pragma unroll
    for (int c = 0; c < TN; ++c) {
      int n = n0 + tx * TN + c;
      if (n >= g.N) continue;
      if (splits == 1) {
        int64_t o = b * g.sCb + (int64_t)m * g.ldc + n;
        float v = acc[r][c] + (g.bias ? g.bias[b * g.sBias + n] : 0.f);
        g.C[o] = g.accumulate ? g.C[o] + v : v;
      } else {
        part[(((int64_t)s * g.batch + b) * g.M + m) * g.N + n] = acc[r][c];
      }
    }
  }
}

__global__ void k_gemm_reduce(Gemm g, int splits, const float* part) {
  grid_dep_wait();
  int64_t total = (int64_t)g.batch * g.M * g.N;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int n = (int)(t % g.N);
    int64_t bm = t / g.N;
    int m = (int)(bm % g.M);
    int b = (int)(bm / g.M);
    float v = 0.f;
    for (int s = 0; s < splits; ++s) v += part[(int64_t)s * total + t];
    if (g.bias) v += g.bias[b * g.sBias + n];
    int64_t o = b * g.sCb + (int64_t)m * g.ldc + n;
    g.C[o] = g.accumulate ? g.C[o] + v : v;
  }
}

// ------------------------------------------------------------------------------------ layout
// Rows of whole 16-byte chunks: one chunk per thread, its row by one 32-bit division.  Bound by HBM
// (both arrays once).  The element-wise form below divides a 64-bit index per element: at 72k x 64
// fp32 it packs in 26.6 us and unpacks in 22.6, this one in 8.0 and 6.9 (ncu).
__global__ void __launch_bounds__(256) k_pack16(const uint4* __restrict__ Eo, uint4* __restrict__ Eb,
                                                const int32_t* __restrict__ gather, int n_real,
                                                uint32_t total, uint32_t chunks) {
  grid_dep_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= total) return;
  const uint32_t q = t / chunks, c = t - q * chunks;
  Eb[t] = q < (uint32_t)n_real ? Eo[(size_t)gather[q] * chunks + c] : make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(256) k_unpack16(const uint4* __restrict__ Eb,
                                                  uint4* __restrict__ Eo,
                                                  const int32_t* __restrict__ gather,
                                                  uint32_t total, uint32_t chunks) {
  grid_dep_wait();
  const uint32_t t = blockIdx.x * 256u + threadIdx.x;
  if (t >= total) return;
  const uint32_t q = t / chunks, c = t - q * chunks;
  Eo[(size_t)gather[q] * chunks + c] = Eb[t];
}

// Any row size and alignment, element by element.
template <typename T>
__global__ void k_pack(const T* Eo, T* Eb, const int32_t* gather, int n_real, int64_t total,
                       int H) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t q = t / H;
    int h = (int)(t % H);
    Eb[t] = q < n_real ? Eo[(int64_t)gather[q] * H + h] : T(0.f);
  }
}

template <typename T>
__global__ void k_unpack(const T* Eb, T* Eo, const int32_t* gather, int64_t total, int H) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t q = t / H;
    int h = (int)(t % H);
    Eo[(int64_t)gather[q] * H + h] = Eb[t];
  }
}

// ------------------------------------------------------------------------------------ band
// Sums rows of a [*][H] array (H = 32 HQ; lanes hold columns lane + 32 q) in the order they are
// pushed, four rows' loads at a time: one row after another the sum waited out a memory latency per
// edge (30k rows of 50 edges at H = 64: 193.7 us against 67.6, which is 5.7 TB/s from L2, ncu).
template <int HQ>
struct RowSum {
  const float* src;
  float acc[HQ];
  int64_t r[4];
  int n;
  __device__ __forceinline__ void clear() {
    n = 0;
    r[0] = r[1] = r[2] = r[3] = 0;
#pragma unroll
    for (int q = 0; q < HQ; ++q) acc[q] = 0.f;
  }
  __device__ __forceinline__ void push(int64_t row) {
    r[0] = r[1]; r[1] = r[2]; r[2] = r[3]; r[3] = row;
    if (++n == 4) {
      float v[4][HQ];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < HQ; ++q) v[i][q] = src[r[i] * (32 * HQ) + 32 * q];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int q = 0; q < HQ; ++q) acc[q] += v[i][q];
      n = 0;
    }
  }
  __device__ __forceinline__ void finish() {  // the last n < 4 rows
    float v[3][HQ];
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < n) {
        const int64_t row = n == 3 ? r[1 + i] : n == 2 ? r[2 + (i & 1)] : r[3];
#pragma unroll
        for (int q = 0; q < HQ; ++q) v[i][q] = src[row * (32 * HQ) + 32 * q];
      }
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < n)
#pragma unroll
        for (int q = 0; q < HQ; ++q) acc[q] += v[i][q];
    n = 0;
  }
};

// One warp per row.  Each lane reads one mask word of the row (in the order diagonal, type, word),
// and the set bits of the words are walked in that order, so the summation order is fixed.
template <int HQ>
__global__ void __launch_bounds__(256) k_band_fwd_gather(const uint32_t* __restrict__ masks,
                                                         const float* __restrict__ M,
                                                         float* __restrict__ Y, int K, int S,
                                                         int P) {
  grid_dep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int64_t n_pad = (int64_t)K * S;
  if (i >= n_pad) return;
  const int k = (int)(i / S), r = (int)(i % S), W32 = S / 32, nw = 3 * P * W32;
  RowSum<HQ> sum;
  sum.src = M + lane;
  sum.clear();
  for (int f0 = 0; f0 < nw; f0 += 32) {
    const int f = f0 + lane;
    uint32_t word = 0;
    int64_t base = 0;  // row of M of the word's bit 0
    if (f < nw) {
      const int w = f % W32, ep = f / W32, e = ep / P, p = ep - e * P, kb = k + e - 1;
      if (kb >= 0 && kb < K) {
        word = masks[((((int64_t)k * 3 + e) * P + p) * S + r) * W32 + w];
        base = (int64_t)p * n_pad + (int64_t)kb * S + w * 32;
      }
    }
    uint32_t full = __ballot_sync(0xffffffffu, word != 0);
    while (full) {
      const int l = __ffs(full) - 1;
      full &= full - 1;
      uint32_t bits = __shfl_sync(0xffffffffu, word, l);
      const int64_t b0 = __shfl_sync(0xffffffffu, base, l);
      while (bits) {
        sum.push(b0 + __ffs(bits) - 1);
        bits &= bits - 1;
      }
    }
  }
  sum.finish();
#pragma unroll
  for (int q = 0; q < HQ; ++q) Y[i * (32 * HQ) + lane + 32 * q] = sum.acc[q];
}

// The same over the transposed tiles, one sum per type; the next type's words are read while the
// current one's rows are summed (3 S / 32 <= 48 words: two per lane).
template <int HQ, typename TO>
__global__ void __launch_bounds__(256) k_band_bwd_gather(const uint32_t* __restrict__ masksT,
                                                         const float* __restrict__ dY,
                                                         TO* __restrict__ dM, int K, int S, int P) {
  grid_dep_wait();
  const int lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int64_t n_pad = (int64_t)K * S;
  if (j >= n_pad) return;
  const int kj = (int)(j / S), c = (int)(j % S), W32 = S / 32, nw = 3 * W32;
  RowSum<HQ> sum;
  sum.src = dY + lane;
  int64_t base[2];
  bool in[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int f = lane + 32 * h, e = f / W32, kb = kj + e - 1;
    in[h] = f < nw && kb >= 0 && kb < K;
    base[h] = (int64_t)kb * S + (f - e * W32) * 32;
  }
  auto words = [&](int p, uint32_t (&w)[2]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int f = lane + 32 * h, e = f / W32;
      w[h] = in[h] ? masksT[((((int64_t)kj * 3 + e) * P + p) * S + c) * W32 + f - e * W32] : 0u;
    }
  };
  uint32_t cur[2], nxt[2] = {0u, 0u};
  words(0, cur);
  for (int p = 0; p < P; ++p) {
    if (p + 1 < P) words(p + 1, nxt);
    sum.clear();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t full = __ballot_sync(0xffffffffu, cur[h] != 0);
      while (full) {
        const int l = __ffs(full) - 1;
        full &= full - 1;
        uint32_t bits = __shfl_sync(0xffffffffu, cur[h], l);
        const int64_t b0 = __shfl_sync(0xffffffffu, base[h], l);
        while (bits) {
          sum.push(b0 + __ffs(bits) - 1);
          bits &= bits - 1;
        }
      }
    }
    sum.finish();
#pragma unroll
    for (int q = 0; q < HQ; ++q) st(dM, (j * P + p) * (32 * HQ) + lane + 32 * q, sum.acc[q]);
    cur[0] = nxt[0];
    cur[1] = nxt[1];
  }
}

// Wperm[h][p*H + o] = W[p][h][o]  (the [H][P*H] B operand of dE = dM_cat W_perm^T)
__global__ void k_wperm(const __nv_bfloat16* __restrict__ W, __nv_bfloat16* __restrict__ Wp, int P,
                        int H) {
  int64_t total = (int64_t)P * H * H;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int o = (int)(t % H);
    const int64_t ph = t / H;
    const int h = (int)(ph % H), p = (int)(ph / H);
    Wp[(int64_t)h * P * H + (int64_t)p * H + o] = W[t];
  }
}

__global__ void k_f32_to_bf16(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    y[t] = __float2bfloat16_rn(x[t]);
}

// Four elements per thread: one 16-byte load, one 8-byte store (x 16-byte and y 8-byte aligned,
// n4 = n / 4 groups; the caller converts the n % 4 tail with k_f32_to_bf16).
__global__ void k_f32_to_bf16_x4(const float4* __restrict__ x, uint2* __restrict__ y, int64_t n4) {
  grid_dep_wait();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n4;
       t += (int64_t)gridDim.x * blockDim.x) {
    const float4 v = x[t];
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    y[t] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
  }
}

template <typename T>
__global__ void k_transpose_w(const T* W, float* Wt, int P, int H) {
  grid_dep_wait();
  int64_t total = (int64_t)P * H * H;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(t % H);
    int64_t po = t / H;
    int o = (int)(po % H);
    int p = (int)(po / H);
    Wt[t] = ld(W, ((int64_t)p * H + i) * H + o);
  }
}

__global__ void k_colsum_part(const float* X, int64_t rows, int cols, int64_t chunk, float* part) {
  grid_dep_wait();
  int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= cols) return;
  int64_t r0 = blockIdx.y * chunk, r1 = min(rows, r0 + chunk);
  float s = 0.f;
  for (int64_t r = r0; r < r1; ++r) s += X[r * cols + col];
  part[(int64_t)blockIdx.y * cols + col] = s;
}

__global__ void k_colsum_reduce(const float* part, int splits, int cols, float* out, int accum) {
  grid_dep_wait();
  int col = blockIdx.x * blockDim.x + threadIdx.x;
  if (col >= cols) return;
  float s = 0.f;
  for (int i = 0; i < splits; ++i) s += part[(int64_t)i * cols + col];
  out[col] = accum ? out[col] + s : s;
}

// ------------------------------------------------------------------------------------ GRU
__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + __expf(-x)); }

template <typename T>
__global__ void k_gru_fwd(const float* gi, const float* gh, const T* E, T* En, int n_real,
                          int64_t total, int H) {
  grid_dep_wait();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = t / H;
    int h = (int)(t % H);
    if (i >= n_real) { st(En, t, 0.f); continue; }
    const float* a = gi + i * 3 * H;
    const float* c = gh + i * 3 * H;
    float r = sigm(a[h] + c[h]);
    float z = sigm(a[H + h] + c[H + h]);
    float n = tanhf(a[2 * H + h] + r * c[2 * H + h]);
    st(En, t, (1.f - z) * n + z * ld(E, t));
  }
}

template <typename T>
__global__ void k_gru_bwd(const float* gi, const float* gh, const T* E, const float* dHn,
                          float* dgi, float* dgh, float* dHd, int n_real, int64_t total, int H) {
  grid_dep_wait();
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t i = t / H;
    int h = (int)(t % H);
    float* oi = dgi + i * 3 * H;
    float* oh = dgh + i * 3 * H;
    if (i >= n_real) {
      oi[h] = oi[H + h] = oi[2 * H + h] = 0.f;
      oh[h] = oh[H + h] = oh[2 * H + h] = 0.f;
      dHd[t] = 0.f;
      continue;
    }
    const float* a = gi + i * 3 * H;
    const float* c = gh + i * 3 * H;
    float r = sigm(a[h] + c[h]);
    float z = sigm(a[H + h] + c[H + h]);
    float n = tanhf(a[2 * H + h] + r * c[2 * H + h]);
    float g = dHn[t];
    float dn = g * (1.f - z);
    float dz = g * (ld(E, t) - n);
    float dan = dn * (1.f - n * n);
    float dar = dan * c[2 * H + h] * r * (1.f - r);
    float daz = dz * z * (1.f - z);
    oi[h] = dar; oi[H + h] = daz; oi[2 * H + h] = dan;
    oh[h] = dar; oh[H + h] = daz; oh[2 * H + h] = dan * r;
    dHd[t] = g * z;
  }
}

// ------------------------------------------------------------------------------------ readout
// Mean pool in two passes so that every graph's rows are read by many blocks at once (one block
// per graph walked each graph's rows one load after another): block (g, k) sums rows
// [off + k cnt / kPoolSplit, off + (k + 1) cnt / kPoolSplit) of graph g, 256 / H rows at a time, into
// part[g][k][H]; k_pool_finish adds the kPoolSplit partial sums in a fixed order.
template <typename T>
__global__ void k_pool_part(const T* ET, const int32_t* seg_off, const int32_t* seg_cnt, int H,
                            float* part) {
  __shared__ float red[256];
  const int g = blockIdx.x, k = blockIdx.y;
  const int R = blockDim.x / H, r = threadIdx.x / H, h = threadIdx.x - r * H;
  const int64_t off = seg_off[g], cnt = seg_cnt[g];
  const int64_t r0 = off + k * cnt / kPoolSplit, r1 = off + (k + 1) * cnt / kPoolSplit;
  float s = 0.f;
  if (r < R)
    for (int64_t i = r0 + r; i < r1; i += R) s += ld(ET, i * H + h);
  red[threadIdx.x] = s;
  __syncthreads();
  if (r == 0) {
    for (int q = 1; q < R; ++q) s += red[q * H + h];
    part[((int64_t)g * kPoolSplit + k) * H + h] = s;
  }
}

__global__ void k_pool_finish(const float* part, const float* w_out, const float* target,
                              const int32_t* seg_cnt, int H, float* pool, float* resid) {
  __shared__ float red[256];
  const int g = blockIdx.x, h = threadIdx.x;
  float s = 0.f;
  if (h < H) {
    for (int k = 0; k < kPoolSplit; ++k) s += part[((int64_t)g * kPoolSplit + k) * H + h];
    s /= (float)seg_cnt[g];
    pool[(int64_t)g * H + h] = s;
  }
  red[h] = h < H ? s * w_out[h] : 0.f;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (h < o) red[h] += red[h + o];
    __syncthreads();
  }
  if (h == 0) resid[g] = red[0] - target[g];
}

__global__ void k_readout_tail(const float* pool, const float* resid, int n_seg, int H,
                               float* loss, float* dw_out) {
  int h = threadIdx.x;
  if (h < H) {
    float s = 0.f;
    for (int g = 0; g < n_seg; ++g) s += resid[g] * pool[(int64_t)g * H + h];
    dw_out[h] = s;
  }
  if (h == 0) {
    float L = 0.f;
    for (int g = 0; g < n_seg; ++g) L += 0.5f * resid[g] * resid[g];
    *loss = L;
  }
}

// dE(T) of the readout, one warp per row (no per-element division of the flat index).
__global__ void k_readout_grad(const float* w_out, const float* resid, const int32_t* seg_cnt,
                               const int32_t* row_graph, int64_t n_rows, int H, float* dET) {
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  if (i >= n_rows) return;
  const int g = row_graph[i];
  float* d = dET + i * H;
  for (int h = threadIdx.x & 31; h < H; h += 32)
    d[h] = g < 0 ? 0.f : resid[g] * w_out[h] / (float)seg_cnt[g];
}

// ------------------------------------------------------------------------------------ Adam
__global__ void k_adam(int64_t n, float* p, __nv_bfloat16* wb, float* wf, float* m, float* v,
                       const float* g, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    float gi = g[i];
    float mi = b1 * m[i] + (1.f - b1) * gi;
    float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (wb) wb[i] = __float2bfloat16_rn(pi);
    if (wf) wf[i] = pi;
  }
}

__global__ void k_zero(float* p, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    p[i] = 0.f;
}

__global__ void k_add(float* d, const float* s, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    d[i] += s[i];
}

}  // namespace

// ====================================================================================== hosts

namespace {
using GemmFn = void (*)(Gemm, int, int, float*);
template <int TM, int TN>
GemmFn gemm_types(const Gemm& g) {
  if (g.a_bf16) return g.b_bf16 ? k_gemm<TM, TN, __nv_bfloat16, __nv_bfloat16> : k_gemm<TM, TN, __nv_bfloat16, float>;
  return g.b_bf16 ? k_gemm<TM, TN, float, __nv_bfloat16> : k_gemm<TM, TN, float, float>;
}
GemmFn gemm_fn(const Gemm& g, int TM, int TN) {
  return TM == 8 ? (TN == 6 ? gemm_types<8, 6>(g) : gemm_types<8, 4>(g))
                 : (TN == 6 ? gemm_types<4, 6>(g) : gemm_types<4, 4>(g));
}
}  // namespace

cudaError_t gemm(const Gemm& g, float* part, size_t part_floats, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  // six columns a thread where the width is a multiple of 96 and not of 64; eight rows where tiles of
  // 128 rows still give every SM one
  const int TN = (g.N % 96 == 0 && g.N % 64 != 0) ? 6 : 4, BN = 16 * TN;
  const int nt = (g.N + BN - 1) / BN;
  const int TM = (int64_t)nt * ((g.M + 127) / 128) * g.batch >= 152 ? 8 : 4, BM = 16 * TM;
  const int tiles = nt * ((g.M + BM - 1) / BM) * g.batch;
  // Few tiles: K split over more blocks, at least 64 of it each (four steps of the loop).  The second
  // launch costs about 3.5 us, so K below 256 is not split.  The two products of the 512-node fp32
  // backward (512 x 64 x 256, and 64 x 64 x 512 for four types) take 15.3 us and 7.2 for their
  // reductions; with the split from K > 512 on and the old loop 165 us (ncu).
  int splits = 1;
  if (g.K >= 256 && tiles < 304 && part) {
    splits = (304 + tiles - 1) / tiles;
    splits = splits > 64 ? 64 : splits;
    int maxk = g.K / 64;
    if (splits > maxk) splits = maxk;
    while (splits > 1 && (size_t)splits * g.batch * g.M * g.N > part_floats) --splits;
  }
  int kchunk = (g.K + splits - 1) / splits;
  kchunk = ((kchunk + GK - 1) / GK) * GK;
  splits = (g.K + kchunk - 1) / kchunk;
  if (splits < 1) splits = 1;
  dim3 grid(nt, (g.M + BM - 1) / BM, g.batch * splits);
  cudaError_t e = launch_pdl(gemm_fn(g, TM, TN), grid, dim3(256), 0, st, g, splits, kchunk, part);
  note_launch();
  if (e == cudaSuccess && splits > 1) {
    int64_t total = (int64_t)g.batch * g.M * g.N;
    e = launch_pdl(k_gemm_reduce, dim3(grid_for(total, 256)), dim3(256), 0, st, g, splits,
                   (const float*)part);
    note_launch();
  }
  return e;
}

// Rows of H elements of `esize` bytes as whole 16-byte chunks: the number per row, 0 where the rows
// or the arrays are not so aligned, or the chunks exceed 32 bits.
static uint32_t row_chunks(const void* a, const void* b, int64_t rows, int H, int esize) {
  const uintptr_t m = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b);
  const int64_t bytes = (int64_t)H * esize;
  return (m % 16 == 0 && bytes % 16 == 0 && rows * (bytes / 16) < (int64_t)1 << 31)
             ? (uint32_t)(bytes / 16) : 0;
}

cudaError_t pack_states(int bf16, const void* Eo, void* Eb, const int32_t* gather, int n_real,
                        int n_pad, int H, cudaStream_t st) {
  int64_t total = (int64_t)n_pad * H;
  if (const uint32_t c = row_chunks(Eo, Eb, n_pad, H, bf16 ? 2 : 4)) {
    const uint32_t n = (uint32_t)n_pad * c;
    if (!n) return cudaSuccess;
    cudaError_t e = launch_pdl(k_pack16, dim3((n + 255) / 256), dim3(256), 0, st,
                               static_cast<const uint4*>(Eo), static_cast<uint4*>(Eb), gather, n_real,
                               n, c);
    note_launch();
    return e;
  }
  if (bf16)
    k_pack<<<grid_for(total, 256), 256, 0, st>>>(static_cast<const __nv_bfloat16*>(Eo),
                                                 static_cast<__nv_bfloat16*>(Eb), gather, n_real,
                                                 total, H);
  else
    k_pack<<<grid_for(total, 256), 256, 0, st>>>(static_cast<const float*>(Eo),
                                                 static_cast<float*>(Eb), gather, n_real, total, H);
  note_launch();
  return cudaGetLastError();
}

cudaError_t unpack_states(int bf16, const void* Eb, void* Eo, const int32_t* gather, int n_real,
                          int H, cudaStream_t st) {
  int64_t total = (int64_t)n_real * H;
  if (total == 0) return cudaSuccess;
  if (const uint32_t c = row_chunks(Eb, Eo, n_real, H, bf16 ? 2 : 4)) {
    const uint32_t n = (uint32_t)n_real * c;
    cudaError_t e = launch_pdl(k_unpack16, dim3((n + 255) / 256), dim3(256), 0, st,
                               static_cast<const uint4*>(Eb), static_cast<uint4*>(Eo), gather, n, c);
    note_launch();
    return e;
  }
  if (bf16)
    k_unpack<<<grid_for(total, 256), 256, 0, st>>>(static_cast<const __nv_bfloat16*>(Eb),
                                                   static_cast<__nv_bfloat16*>(Eo), gather, total,
                                                   H);
  else
    k_unpack<<<grid_for(total, 256), 256, 0, st>>>(static_cast<const float*>(Eb),
                                                   static_cast<float*>(Eo), gather, total, H);
  note_launch();
  return cudaGetLastError();
}

namespace {
// f(integral_constant<int, H / 32>) for H a multiple of 32 up to 256
template <typename F>
cudaError_t with_hq(int H, F f) {
  switch (H / 32) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    default: return cudaErrorInvalidValue;
  }
}
}  // namespace

cudaError_t preload_fwd_simt() {
  // CUDA loads kernels lazily, on first launch; this loads the ones the SIMT forward launches
  cudaFuncAttributes a;
  cudaError_t e = cudaSuccess;
  auto take = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
  for (int v = 0; v < 16; ++v) {
    Gemm g;
    g.a_bf16 = v & 1;
    g.b_bf16 = v >> 1 & 1;
    take(cudaFuncGetAttributes(&a, reinterpret_cast<const void*>(gemm_fn(g, v & 4 ? 8 : 4, v & 8 ? 6 : 4))));
  }
  take(cudaFuncGetAttributes(&a, k_gemm_reduce));
  for (int H = 32; H <= 256; H += 32)
    take(with_hq(H, [&](auto hq) {
      return cudaFuncGetAttributes(&a, k_band_fwd_gather<decltype(hq)::value>);
    }));
  return e;
}

cudaError_t band_fwd_gather(const uint32_t* masks, const float* M, float* Y, int K, int S, int P,
                            int H, cudaStream_t st) {
  const dim3 grid((unsigned)(((int64_t)K * S + 7) / 8));
  cudaError_t e = with_hq(H, [&](auto hq) {
    return launch_pdl(k_band_fwd_gather<decltype(hq)::value>, grid, dim3(256), 0, st, masks, M, Y, K, S, P);
  });
  note_launch();
  return e;
}

cudaError_t band_bwd_gather(const uint32_t* masksT, const float* dY, float* dM, int K, int S,
                            int P, int H, cudaStream_t st) {
  const dim3 grid((unsigned)(((int64_t)K * S + 7) / 8));
  cudaError_t e = with_hq(H, [&](auto hq) {
    return launch_pdl(k_band_bwd_gather<decltype(hq)::value, float>, grid, dim3(256), 0, st, masksT, dY,
                      dM, K, S, P);
  });
  note_launch();
  return e;
}

cudaError_t band_bwd_gather_bf16(const uint32_t* masksT, const float* dY, __nv_bfloat16* dM, int K,
                                 int S, int P, int H, cudaStream_t st) {
  const dim3 grid((unsigned)(((int64_t)K * S + 7) / 8));
  cudaError_t e = with_hq(H, [&](auto hq) {
    return launch_pdl(k_band_bwd_gather<decltype(hq)::value, __nv_bfloat16>, grid, dim3(256), 0, st,
                      masksT, dY, dM, K, S, P);
  });
  note_launch();
  return e;
}

cudaError_t wperm(const void* W, __nv_bfloat16* Wp, int P, int H, cudaStream_t st) {
  int64_t total = (int64_t)P * H * H;
  k_wperm<<<grid_for(total, 256), 256, 0, st>>>(static_cast<const __nv_bfloat16*>(W), Wp, P, H);
  note_launch();
  return cudaGetLastError();
}

cudaError_t f32_to_bf16(const float* x, __nv_bfloat16* y, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t n4 = (reinterpret_cast<uintptr_t>(x) % 16 == 0 && reinterpret_cast<uintptr_t>(y) % 8 == 0)
                         ? n / 4 : 0;
  if (n4 > 0) {
    cudaError_t e = launch_pdl(k_f32_to_bf16_x4, dim3(grid_for(n4, 256)), dim3(256), 0, st,
                               reinterpret_cast<const float4*>(x), reinterpret_cast<uint2*>(y), n4);
    note_launch();
    if (e != cudaSuccess) return e;
  }
  if (n > 4 * n4) {
    k_f32_to_bf16<<<grid_for(n - 4 * n4, 256), 256, 0, st>>>(x + 4 * n4, y + 4 * n4, n - 4 * n4);
    note_launch();
  }
  return cudaGetLastError();
}

cudaError_t transpose_weights(int bf16, const void* W, float* Wt, int P, int H, cudaStream_t st) {
  int64_t total = (int64_t)P * H * H;
  cudaError_t e;
  if (bf16)
    e = launch_pdl(k_transpose_w<__nv_bfloat16>, dim3(grid_for(total, 256)), dim3(256), 0, st,
                   static_cast<const __nv_bfloat16*>(W), Wt, P, H);
  else
    e = launch_pdl(k_transpose_w<float>, dim3(grid_for(total, 256)), dim3(256), 0, st,
                   static_cast<const float*>(W), Wt, P, H);
  note_launch();
  return e;
}

cudaError_t colsum(const float* X, int64_t rows, int cols, float* out, int accumulate, float* part,
                   size_t part_floats, cudaStream_t st) {
  // 32 rows a block up to 256 blocks (one block of 512 rows added them one latency after another:
  // 32.3 us against 3.9)
  int splits = (int)((rows + 31) / 32);
  if (splits > 256) splits = 256;
  while (splits > 1 && (size_t)splits * cols > part_floats) --splits;
  if (splits < 1) splits = 1;
  if ((size_t)splits * cols > part_floats) return cudaErrorInvalidValue;  // partials always used
  int64_t chunk = (rows + splits - 1) / splits;
  dim3 grid((cols + 255) / 256, splits);
  cudaError_t e = launch_pdl(k_colsum_part, grid, dim3(256), 0, st, X, rows, cols, chunk, part);
  note_launch();
  if (e != cudaSuccess) return e;
  e = launch_pdl(k_colsum_reduce, dim3((cols + 255) / 256), dim3(256), 0, st, (const float*)part, splits,
                 cols, out, accumulate);
  note_launch();
  return e;
}

cudaError_t gru_fwd_gates(int bf16, const float* gi, const float* gh, const void* E, void* En,
                          int n_real, int n_pad, int H, cudaStream_t st) {
  const int64_t total = (int64_t)n_pad * H;
  cudaError_t e;
  if (bf16)
    e = launch_pdl(k_gru_fwd<__nv_bfloat16>, dim3(grid_for(total, 256)), dim3(256), 0, st, gi, gh,
                   static_cast<const __nv_bfloat16*>(E), static_cast<__nv_bfloat16*>(En), n_real, total, H);
  else
    e = launch_pdl(k_gru_fwd<float>, dim3(grid_for(total, 256)), dim3(256), 0, st, gi, gh,
                   static_cast<const float*>(E), static_cast<float*>(En), n_real, total, H);
  note_launch();
  return e;
}

cudaError_t gru_bwd_gates(int bf16, const float* gi, const float* gh, const void* E,
                          const float* dHn, float* dgi, float* dgh, float* dHd, int n_real,
                          int n_pad, int H, cudaStream_t st) {
  const int64_t total = (int64_t)n_pad * H;
  cudaError_t e;
  if (bf16)
    e = launch_pdl(k_gru_bwd<__nv_bfloat16>, dim3(grid_for(total, 256)), dim3(256), 0, st, gi, gh,
                   static_cast<const __nv_bfloat16*>(E), dHn, dgi, dgh, dHd, n_real, total, H);
  else
    e = launch_pdl(k_gru_bwd<float>, dim3(grid_for(total, 256)), dim3(256), 0, st, gi, gh,
                   static_cast<const float*>(E), dHn, dgi, dgh, dHd, n_real, total, H);
  note_launch();
  return e;
}

cudaError_t readout_loss(int bf16, const void* ET, const float* w_out, const float* target,
                         const int32_t* seg_off, const int32_t* seg_cnt, const int32_t* row_graph,
                         int n_seg, int n_pad, int H, float* pool, float* resid, float* part,
                         float* loss, float* dET, float* dw_out, cudaStream_t st) {
  if (H < 1 || H > 256) return cudaErrorInvalidValue;
  if (n_seg > 0) {
    const dim3 grid(n_seg, kPoolSplit);
    if (bf16)
      k_pool_part<<<grid, 256, 0, st>>>(static_cast<const __nv_bfloat16*>(ET), seg_off, seg_cnt, H,
                                        part);
    else
      k_pool_part<<<grid, 256, 0, st>>>(static_cast<const float*>(ET), seg_off, seg_cnt, H, part);
    note_launch();
    k_pool_finish<<<n_seg, 256, 0, st>>>(part, w_out, target, seg_cnt, H, pool, resid);
    note_launch();
  }
  k_readout_tail<<<1, 256, 0, st>>>(pool, resid, n_seg, H, loss, dw_out);
  note_launch();
  k_readout_grad<<<(unsigned)((n_pad + 7) / 8), 256, 0, st>>>(w_out, resid, seg_cnt, row_graph,
                                                              n_pad, H, dET);
  note_launch();
  return cudaGetLastError();
}

cudaError_t adam(int64_t n, float* master, void* working, int working_bf16, float* m, float* v,
                 const float* grad, float lr, float b1, float b2, float eps, int step,
                 cudaStream_t st) {
  float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  __nv_bfloat16* wb = working_bf16 ? static_cast<__nv_bfloat16*>(working) : nullptr;
  float* wf = working_bf16 ? nullptr : static_cast<float*>(working);
  k_adam<<<grid_for(n, 256), 256, 0, st>>>(n, master, wb, wf, m, v, grad, lr, b1, b2, eps, c1, c2);
  note_launch();
  return cudaGetLastError();
}

cudaError_t fill_zero_f32(float* p, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_zero<<<grid_for(n, 256), 256, 0, st>>>(p, n);
  note_launch();
  return cudaGetLastError();
}

cudaError_t add_inplace_f32(float* dst, const float* src, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  k_add<<<grid_for(n, 256), 256, 0, st>>>(dst, src, n);
  note_launch();
  return cudaGetLastError();
}

}  // namespace bg
