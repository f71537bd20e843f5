// Host side of the tensor-core path's plan data (band_tc.cu uploads what this builds).
//
// For every 128-row tile and edge type: the C1 128-column chunks of the tile's state window
// [ws, ws + 128 C1), ws = (row0 / S) S - S, as 4 words per row and chunk, in both orientations,
// with the bits of each word interleaved (column 2j at bit j, column 2j+1 at bit 16+j) so that the
// kernel turns a word into packed bf16 pairs with one AND and one multiply; words outside the three
// block diagonals of the row's block-row are zero.  And per row and type the in-degree over the
// three diagonals (columns p and 32 + p), the bias product's A operand: bf16 integers when every
// in-degree is at most 256, fp16 integers otherwise (a hub node; fp16 is exact up to 2048).
#include <algorithm>
#include <atomic>
#include <cstring>
#include <new>
#include <numeric>
#include <thread>
#include <vector>

#include "band_tc.h"
#include "internal.h"

namespace bg {

namespace {

// Bits 0, 2, 4, ... of x packed into bits 0..15 (even-bit compaction by shifts and masks).
inline uint32_t even_bits(uint32_t x) {
  x &= 0x55555555u;
  x = (x | (x >> 1)) & 0x33333333u;
  x = (x | (x >> 2)) & 0x0F0F0F0Fu;
  x = (x | (x >> 4)) & 0x00FF00FFu;
  x = (x | (x >> 8)) & 0x0000FFFFu;
  return x;
}

// Column 2j -> bit j, column 2j+1 -> bit 16+j.
inline uint32_t interleave(uint32_t w) {
  return w == 0 ? 0u : even_bits(w) | (even_bits(w >> 1) << 16);
}

// Items of `bytes` of masks or chunks each that make a thread's range worth its start (about 50 us).
inline int64_t grain_of(int64_t bytes) { return std::max<int64_t>(1, (int64_t)(1 << 18) / std::max<int64_t>(1, bytes)); }

// Runs f(lo, hi) over [0, n) split into contiguous ranges of at least `grain` on up to 16 host threads.
// An exception in any of them (an allocation that failed) is thrown here as bad_alloc once all have
// ended.
template <typename F>
void parallel_ranges(int64_t n, F f, int64_t grain) {
  unsigned nt = std::max(1u, std::min(std::thread::hardware_concurrency(), 16u));
  nt = (unsigned)std::max<int64_t>(1, std::min<int64_t>(nt, n / grain));
  std::atomic<bool> failed{false};
  auto run = [&failed, &f](int64_t lo, int64_t hi) {
    try {
      f(lo, hi);
    } catch (...) {
      failed = true;
    }
  };
  std::vector<std::thread> pool;
  for (unsigned t = 1; t < nt; ++t) {
    const int64_t lo = n * t / nt, hi = n * (t + 1) / nt;
    try {
      pool.emplace_back(run, lo, hi);
    } catch (...) {  // no thread to be had: this range here
      run(lo, hi);
    }
  }
  run(0, n / nt);
  for (auto& th : pool) th.join();
  if (failed) throw std::bad_alloc();
}

// bf16 bit pattern of a count (exact up to 256).
inline uint16_t bf16_bits_of_count(int c) {
  const float f = (float)c;
  uint32_t u;
  std::memcpy(&u, &f, 4);
  return (uint16_t)(u >> 16);
}

// IEEE fp16 bit pattern of a count in [0, 2048) (exact: at most 11 significant bits).
inline uint16_t f16_bits_of_count(int c) {
  if (c == 0) return 0;
  int e = 0;
  while ((c >> (e + 1)) != 0) ++e;  // floor(log2 c)
  const uint32_t mant = ((uint32_t)c << (10 - e)) & 0x3FFu;
  return (uint16_t)(((uint32_t)(e + 15) << 10) | mant);
}

}  // namespace

// One orientation's chunks, [n_tiles][P][C1][128][4] words, every word written (out needs no
// clearing: at S = 512 the arrays are 1 GB, and one thread zeroing them took longer than the threads
// that fill them).
void band_tc_host_chunks(const bg_plan* p, int C1, bool transposed, uint32_t* out) {
  constexpr int kTile = 128;
  const int S = p->S, K = p->K, P = p->P, W32 = p->W32;
  const int64_t n = (int64_t)K * S, n_tiles = n / kTile;
  const std::vector<uint32_t>& masks = transposed ? p->masksT : p->masks;
  const int SB = std::min(S, kTile);  // rows of one block-row within a tile
  parallel_ranges(n_tiles, [&](int64_t t0, int64_t t1) {
    for (int64_t t = t0; t < t1; ++t) {
      const int64_t row0 = t * kTile, ws = (row0 / S) * S - S;
      for (int q = 0; q < P; ++q)
        for (int j = 0; j < C1; ++j)
          for (int r0 = 0; r0 < kTile; r0 += SB) {
            const int64_t R = row0 + r0, kr = R / S;
            uint32_t* o = out + ((((size_t)t * P + q) * C1 + j) * kTile + r0) * 4;
            const uint32_t* src[4];
            for (int w = 0; w < 4; ++w) {
              const int64_t Cc = ws + j * kTile + 32 * w, kc = Cc >= 0 && Cc < n ? Cc / S : -2;
              const int64_t d = kc - kr + 1;
              src[w] = kc < 0 || d < 0 || d > 2 ? nullptr
                       : &masks[((((size_t)kr * 3 + d) * P + q) * S + R % S) * W32 + (Cc % S) / 32];
            }
            for (int r = 0; r < SB; ++r)
              for (int w = 0; w < 4; ++w)
                o[4 * r + w] = src[w] ? interleave(src[w][(size_t)r * W32]) : 0u;
          }
    }
  }, grain_of((int64_t)P * C1 * kTile * 16));
}

// mi, mti: [n_tiles][P][C1][128][4] words; deg: [n_pad][64] in-degrees (type q at columns q and
// 32 + q) as bf16 when the largest is at most 256, else as fp16.  Returns the largest in-degree.
int band_tc_host_tiles(const bg_plan* p, int C1, std::vector<uint32_t>& mi,
                       std::vector<uint32_t>& mti, std::vector<uint16_t>& deg) {
  const size_t words = (size_t)p->K * p->S / 128 * p->P * C1 * 128 * 4;
  mi.resize(words);
  mti.resize(words);
  band_tc_host_chunks(p, C1, false, mi.data());
  band_tc_host_chunks(p, C1, true, mti.data());
  return band_tc_host_degrees(p, deg);
}

// deg: [n_pad][64], see above; returns the largest in-degree of one type.
int band_tc_host_degrees(const bg_plan* p, std::vector<uint16_t>& deg, int64_t* edges) {
  const int S = p->S, K = p->K, P = p->P, W32 = p->W32;
  const int64_t n = (int64_t)K * S;
  deg.assign((size_t)n * 64, 0);
  // in-degrees first, then their encoding: bf16 while every count is at most 256 (exact), else
  // fp16 (exact up to 2048 > 3 S for every block size)
  std::vector<uint16_t> cnt((size_t)n * P, 0);
  std::vector<int> part_max(K, 0);
  std::vector<int64_t> part_sum(K, 0);
  parallel_ranges(K, [&](int64_t k0, int64_t k1) {
    for (int64_t k = k0; k < k1; ++k) {
      int mx = 0;
      int64_t sum = 0;
      for (int q = 0; q < P; ++q)
        for (int r = 0; r < S; ++r) {
          int c = 0;
          for (int d = 0; d < 3; ++d)
            for (int w = 0; w < W32; ++w)  // (nearly every word is zero)
              if (const uint32_t m = p->masks[((((size_t)k * 3 + d) * P + q) * S + r) * W32 + w])
                c += __builtin_popcount(m);
          mx = std::max(mx, c);
          sum += c;
          cnt[((size_t)k * S + r) * P + q] = (uint16_t)c;
        }
      part_max[k] = mx;
      part_sum[k] = sum;
    }
  }, grain_of((int64_t)12 * P * S * W32));
  const int max_deg = *std::max_element(part_max.begin(), part_max.end());
  if (edges) *edges = std::accumulate(part_sum.begin(), part_sum.end(), (int64_t)0);
  const bool f16 = max_deg > 256;
  parallel_ranges(n, [&](int64_t r0, int64_t r1) {
    for (int64_t r = r0; r < r1; ++r)
      for (int q = 0; q < P; ++q) {
        const uint16_t v = f16 ? f16_bits_of_count(cnt[(size_t)r * P + q])
                               : bf16_bits_of_count(cnt[(size_t)r * P + q]);
        deg[(size_t)r * 64 + q] = v;
        deg[(size_t)r * 64 + 32 + q] = v;
      }
  }, grain_of(256));
  return max_deg;
}


namespace {
// Gather steps of one type of a 16-row group (at least one).
inline uint32_t list_steps(uint32_t edges) { return std::max<uint32_t>(1, (edges + 15) / 16); }
}  // namespace

void list_layout(const bg_plan* p, const int* reach, GatherLists& out) {
  const int P = p->P;
  auto up8 = [](int x) { return (x + 7) & ~7; };
  out.lo = up8(reach[0]);
  out.rows = out.lo + 128 + up8(reach[1]);
  // a whole number of equal TMA boxes of at most 256 rows
  const int boxes = (out.rows + 255) / 256;
  out.rows = up8((out.rows + boxes - 1) / boxes) * boxes;
  // per 16-row group: the even types, then the odd ones (the kernel's two classes of warps), each
  // type's steps padded to whole blocks
  uint64_t total = 0;
  out.steps = 0;
  for (size_t o = 0; o < out.off.size(); o += P + 1) {
    for (int i = 0; i < P; ++i) {
      const uint32_t ns = list_steps(out.off[o + i]);
      out.off[o + i] = (uint32_t)total;
      out.steps += ns;
      total += (ns + kGatherBlock - 1) / kGatherBlock;
    }
    out.off[o + P] = (uint32_t)total;
  }
  out.blocks = (int64_t)total;
}

namespace {

// One 16-row group's edges of one type (row within the group << 16 | window row) as gather steps of
// 16: `words` gets 32 words per step (see band_tc_host_lists).  ldmatrix reads 8 window rows at
// once from one 16-byte column, so a set of 8 edges whose window rows differ mod 8 reads all 32
// banks and one whose rows agree serialises: the edges are dealt into sets by taking the fullest
// residues first, and padding entries take a zero row of an unused residue.
void emit_steps(const uint32_t* e, int n, int zero_row, uint32_t* words,
                std::vector<uint32_t>& tmp) {
  const int steps = (int)list_steps((uint32_t)n);
  int cnt[8] = {0}, pos[8];
  for (int i = 0; i < n; ++i) ++cnt[e[i] & 7];
  for (int r = 0, o = 0; r < 8; ++r) { pos[r] = o; o += cnt[r]; }
  tmp.resize((size_t)std::max(n, 1));
  {
    int at[8];
    std::copy(pos, pos + 8, at);
    for (int i = 0; i < n; ++i) tmp[at[e[i] & 7]++] = e[i];
  }
  int rem = n;
  for (int s = 0; s < steps; ++s) {
    uint32_t ent[16];
    bool real[16];
    for (int half = 0; half < 2; ++half) {
      const int sets_after = 2 * (steps - s) - half - 1;
      const int need = std::max(0, rem - 8 * sets_after);
      int order[8] = {0, 1, 2, 3, 4, 5, 6, 7};
      for (int i = 1; i < 8; ++i)
        for (int j = i; j > 0 && cnt[order[j]] > cnt[order[j - 1]]; --j) std::swap(order[j], order[j - 1]);
      bool used[8] = {false};
      int k = 0;
      for (int i = 0; i < 8; ++i)
        if (cnt[order[i]] > 0) {
          const int r = order[i];
          ent[8 * half + k] = tmp[pos[r]++];
          real[8 * half + k++] = true;
          --cnt[r];
          used[r] = true;
        }
      while (k < need) {
        const int r = (int)(std::max_element(cnt, cnt + 8) - cnt);
        ent[8 * half + k] = tmp[pos[r]++];
        real[8 * half + k++] = true;
        --cnt[r];
      }
      rem -= k;
      for (int r = 0; k < 8; r = (r + 1) & 7)
        if (!used[r]) {
          ent[8 * half + k] = (uint32_t)(zero_row + r);
          real[8 * half + k++] = false;
          used[r] = true;
        } else if (std::all_of(used, used + 8, [](bool u) { return u; })) {
          std::fill(used, used + 8, false);
        }
    }
    uint32_t* w = words + (size_t)s * 32;
    for (int l = 0; l < 32; ++l) {
      const uint32_t row = ent[l & 15] & 0xFFFFu, hi = (uint32_t)(l >> 4);
      w[l] = row * 128u + ((hi ^ (row & 7u)) << 4);
    }
    for (int k = 0; k < 16; ++k)
      if (real[k]) {
        const int r = (int)(ent[k] >> 16);
        w[(r & 7) * 4 + (k & 7) / 2] |= 1u << (24 + (r >> 3) + 2 * (k >> 3) + 4 * (k & 1));
      }
  }
}

}  // namespace

int64_t band_tc_list_steps(const bg_plan* p, bool transposed) {
  const int S = p->S, K = p->K, P = p->P, W32 = p->W32;
  const std::vector<uint32_t>& masks = transposed ? p->masksT : p->masks;
  std::vector<int64_t> part((size_t)K, 0);  // S is a multiple of 16: no group spans two block-rows
  parallel_ranges(K, [&](int64_t k0, int64_t k1) {
    for (int64_t k = k0; k < k1; ++k)
      for (int q = 0; q < P; ++q)
        for (int r0 = 0; r0 < S; r0 += 16) {
          int m = 0;
          for (int d = 0; d < 3; ++d) {
            const uint32_t* w = &masks[((((size_t)k * 3 + d) * P + q) * S + r0) * W32];
            for (int j = 0; j < 16 * W32; ++j) m += __builtin_popcount(w[j]);
          }
          part[(size_t)k] += list_steps((uint32_t)m);
        }
  }, grain_of((int64_t)12 * P * S * W32));
  // the groups beyond the last row of a last tile that is not whole have one empty step per type
  const int64_t n = (int64_t)K * S;
  int64_t steps = ((n + 127) / 128 * 8 - n / 16) * P;
  for (int64_t x : part) steps += x;
  return steps;
}

void band_tc_host_lists(const bg_plan* p, bool transposed, GatherLists& out) {
  constexpr int kTile = 128;
  const int S = p->S, K = p->K, P = p->P, W32 = p->W32;
  const int64_t n = (int64_t)K * S, n_tiles = (n + kTile - 1) / kTile;
  const std::vector<uint32_t>& masks = transposed ? p->masksT : p->masks;
  const int NB = kTile / 16;
  // edges of every tile, as (16-row group, type), row in the group, column; reach beyond the tile
  std::vector<std::vector<uint32_t>> edges((size_t)n_tiles);  // col - row0 + 2048 | row << 16
  std::vector<std::vector<uint32_t>> start((size_t)n_tiles);  // (group, type) ranges, [NB * P + 1]
  std::vector<int> lo((size_t)n_tiles, 0), hi((size_t)n_tiles, 0);
  parallel_ranges(n_tiles, [&](int64_t t0, int64_t t1) {
    for (int64_t t = t0; t < t1; ++t) {
      const int64_t row0 = t * kTile;
      auto& ed = edges[t];
      auto& st = start[t];
      st.reserve((size_t)NB * P + 1);
      for (int b = 0; b < NB; ++b)
        for (int q = 0; q < P; ++q) {
          st.push_back((uint32_t)ed.size());
          for (int i = 0; i < 16; ++i) {
            const int64_t R = row0 + 16 * b + i;
            if (R >= n) break;
            const int64_t kr = R / S;
            for (int d = 0; d < 3; ++d) {
              const int64_t kc = kr + d - 1;
              if (kc < 0 || kc >= K) continue;
              const uint32_t* w = &masks[((((size_t)kr * 3 + d) * P + q) * S + R % S) * W32];
              for (int j = 0; j < W32; ++j)
                for (uint32_t m = w[j]; m; m &= m - 1) {
                  const int rel = (int)(kc * S + 32 * j + __builtin_ctz(m) - row0);
                  lo[t] = std::max(lo[t], -rel);
                  hi[t] = std::max(hi[t], rel - (kTile - 1));
                  ed.push_back((uint32_t)i << 16 | (uint32_t)(rel + 2048));
                }
            }
          }
        }
      st.push_back((uint32_t)ed.size());
    }
  }, 1);
  auto type_at = [&](int i) { return i < (P + 1) / 2 ? 2 * i : 2 * (i - (P + 1) / 2) + 1; };
  out.off.assign((size_t)n_tiles * NB * (P + 1), 0);
  for (int64_t t = 0; t < n_tiles; ++t)
    for (int b = 0; b < NB; ++b)
      for (int i = 0; i < P; ++i) {
        const uint32_t* at = &start[t][(size_t)b * P + type_at(i)];
        out.off[((size_t)t * NB + b) * (P + 1) + i] = at[1] - at[0];
      }
  const int reach[2] = {*std::max_element(lo.begin(), lo.end()), *std::max_element(hi.begin(), hi.end())};
  list_layout(p, reach, out);
  if (out.blocks >> 31) return;  // the caller checks `blocks`
  out.words.assign((size_t)out.blocks * 32 * kGatherBlock, 0u);
  parallel_ranges(n_tiles, [&](int64_t t0, int64_t t1) {
    std::vector<uint32_t> tmp, words;
    for (int64_t t = t0; t < t1; ++t) {
      for (auto& e : edges[t]) e += (uint32_t)(out.lo - 2048);  // window row in the low half
      for (int b = 0; b < NB; ++b)
        for (int i = 0; i < P; ++i) {
          const int q = type_at(i);
          const uint32_t e0 = start[t][(size_t)b * P + q], e1 = start[t][(size_t)b * P + q + 1];
          const int ns = (int)list_steps(e1 - e0);
          words.assign((size_t)ns * 32, 0u);
          emit_steps(edges[t].data() + e0, (int)(e1 - e0), out.rows, words.data(), tmp);
          uint32_t* o = &out.words[(size_t)out.off[((size_t)t * NB + b) * (P + 1) + i] * 32 * kGatherBlock];
          for (int s = 0; s < ns; ++s) {
            const int s0 = s / kGatherBlock * kGatherBlock, in = std::min(kGatherBlock, ns - s0);
            const uint32_t flags = (uint32_t)(in - 1) * kGatherMore + (s0 + in == ns ? kGatherLast : 0u);
            for (int l = 0; l < 32; ++l)
              o[((size_t)(s / kGatherBlock) * 32 + l) * kGatherBlock + s % kGatherBlock] =
                  words[(size_t)s * 32 + l] | flags;
          }
        }
    }
  }, 1);
}

}  // namespace bg
