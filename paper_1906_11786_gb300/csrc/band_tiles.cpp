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

constexpr int kListTile = 128, kGroups = kListTile / 16;  // rows of a tile, 16-row groups of one

// Position of the i-th type in a group's order: the even types, then the odd ones (the kernel's two
// classes of warps).
inline int type_at(int i, int P) { return i < (P + 1) / 2 ? 2 * i : 2 * (i - (P + 1) / 2) + 1; }
inline uint32_t steps_of(uint32_t edges) { return std::max<uint32_t>(1, (edges + 15) / 16); }

// One 16-row group's edges of one type (row within the group << 16 | column - tile + 2048) as blocks of
// gather steps of 16 edges at `out` (the format: band_tc.h).  `add` turns the low half into the window
// row.  ldmatrix reads 8 window rows at once from one 16-byte column, so a set of 8 edges whose window
// rows differ mod 8 reads all 32 banks and one whose rows agree serialises: the edges are dealt into
// sets by taking the fullest residues first, and padding entries take a zero row of an unused residue.
void emit_type(const uint32_t* e, int n, uint32_t add, uint32_t zero_row, uint32_t* out,
               std::vector<uint32_t>& tmp) {
  const int steps = (int)steps_of((uint32_t)n);
  uint32_t cnt[8] = {0}, pos[8], at[8];
  for (int i = 0; i < n; ++i) ++cnt[e[i] & 7];  // (add is a multiple of 8)
  for (uint32_t r = 0, o = 0; r < 8; ++r) { pos[r] = at[r] = o; o += cnt[r]; }
  if (tmp.size() < (size_t)n) tmp.resize((size_t)n);
  for (int i = 0; i < n; ++i) tmp[at[e[i] & 7]++] = e[i] + add;
  int rem = n;
  uint32_t blk[32][kGatherBlock];
  for (int s = 0; s < steps; ++s) {
    const int in_blk = s % kGatherBlock;
    if (in_blk == 0) std::memset(blk, 0, sizeof(blk));
    uint32_t ent[16], bits[32] = {0};
    for (int half = 0; half < 2; ++half) {
      const int need = std::max(0, rem - 8 * (2 * (steps - s) - half - 1));
      uint32_t* x = ent + 8 * half;
      int k = 0;
      unsigned used = 0;
      auto take = [&](int r) {
        const uint32_t v = x[k] = tmp[pos[r]++], row = v >> 16;
        --cnt[r];
        bits[(row & 7) * 4 + k / 2] |= 1u << (24 + (row >> 3) + 2 * half + 4 * (k & 1));
        ++k;
      };
      if (rem) {
        // one edge of every residue left, the fullest first (by residue where equal)
        uint32_t key[8];
        for (uint32_t r = 0; r < 8; ++r) key[r] = cnt[r] << 3 | (7 - r);
        auto order = [&](int a, int b) {
          const uint32_t hi = std::max(key[a], key[b]), lo = std::min(key[a], key[b]);
          key[a] = hi, key[b] = lo;
        };
        order(0, 1); order(2, 3); order(4, 5); order(6, 7);
        order(0, 2); order(1, 3); order(4, 6); order(5, 7);
        order(1, 2); order(5, 6);
        order(0, 4); order(1, 5); order(2, 6); order(3, 7);
        order(2, 4); order(3, 5);
        order(1, 2); order(3, 4); order(5, 6);
        for (int i = 0; i < 8 && key[i] >= 8; ++i) {
          const int r = 7 - (int)(key[i] & 7);
          take(r);
          used |= 1u << r;
        }
        while (k < need) take((int)(std::max_element(cnt, cnt + 8) - cnt));
        rem -= k;
      }
      for (int r = 0; k < 8; r = (r + 1) & 7) {
        if (!(used >> r & 1)) {
          x[k++] = zero_row + r;
          used |= 1u << r;
        } else if (used == 0xFF) {
          used = 0;
        }
      }
    }
    const int s0 = s - in_blk, in = std::min(kGatherBlock, steps - s0);
    const uint32_t flags = (uint32_t)(in - 1) * kGatherMore + (s0 + in == steps ? kGatherLast : 0u);
    for (int k = 0; k < 16; ++k) {
      const uint32_t row = ent[k] & 0xFFFFu, w = row * 128u + ((row & 7u) << 4);
      blk[k][in_blk] = w | flags | bits[k];
      blk[k + 16][in_blk] = (w ^ 16u) | flags | bits[k + 16];
    }
    if (in_blk == in - 1) std::memcpy(out + (size_t)(s / kGatherBlock) * 32 * kGatherBlock, blk, sizeof(blk));
  }
}

// The set bits of `words` 32-bit mask words, in order: f(bit).  Two words at a time where they pair up.
template <typename F>
inline void for_bits(const uint32_t* w, int words, F f) {
  int j = 0;
  for (; j + 1 < words; j += 2) {
    uint64_t m;
    std::memcpy(&m, w + j, 8);  // (both hosts are little-endian)
    for (; m; m &= m - 1) f(32 * j + __builtin_ctzll(m));
  }
  if (j < words)
    for (uint32_t m = w[j]; m; m &= m - 1) f(32 * j + __builtin_ctz(m));
}

}  // namespace

// Edges of one orientation by tile, 16-row group and type, and where their steps will stand.
void band_tc_scan_lists(const bg_plan* p, unsigned orientations, ListScan* out) {
  const int S = p->S, K = p->K, P = p->P, W32 = p->W32;
  const int64_t n = (int64_t)K * S, n_tiles = (n + kListTile - 1) / kListTile;
  // a unit of tiles shares one array of edges (row in the group << 16 | column - tile + 2048)
  const int unit = (int)std::min<int64_t>(std::max<int64_t>(1, n_tiles / 64), 64);
  const int64_t units = (n_tiles + unit - 1) / unit;
  std::vector<int> todo;
  for (int d = 0; d < 2; ++d)
    if (orientations >> d & 1) {
      todo.push_back(d);
      out[d].unit = unit;
      out[d].edges.resize((size_t)units);
      out[d].start.resize((size_t)n_tiles * (kGroups * P + 1));
    }
  const int64_t jobs = units * (int64_t)todo.size();
  std::vector<int> lo((size_t)jobs, 0), hi((size_t)jobs, 0);
  parallel_ranges(jobs, [&](int64_t w0, int64_t w1) {
    for (int64_t w = w0; w < w1; ++w) {
      const int tr = todo[(size_t)(w / units)];
      const int64_t u = w % units;
      const std::vector<uint32_t>& masks = tr ? p->masksT : p->masks;
      std::vector<uint32_t>& ed = out[tr].edges[(size_t)u];
      int l = 0, h = 0;
      for (int64_t t = u * unit; t < std::min(n_tiles, (u + 1) * unit); ++t) {
        const int64_t row0 = t * kListTile;
        uint32_t* st = &out[tr].start[(size_t)t * (kGroups * P + 1)];
        for (int b = 0; b < kGroups; ++b)
          for (int q = 0; q < P; ++q) {
            *st++ = (uint32_t)ed.size();
            for (int i = 0; i < 16; ++i) {
              const int64_t R = row0 + 16 * b + i;
              if (R >= n) break;
              const int64_t kr = R / S;
              for (int d = 0; d < 3; ++d) {
                const int64_t kc = kr + d - 1;
                if (kc < 0 || kc >= K) continue;
                const int c0 = (int)(kc * S - row0);
                for_bits(&masks[((((size_t)kr * 3 + d) * P + q) * S + R % S) * W32], W32, [&](int c) {
                  const int rel = c0 + c;
                  l = std::max(l, -rel);
                  h = std::max(h, rel - (kListTile - 1));
                  ed.push_back((uint32_t)i << 16 | (uint32_t)(rel + 2048));
                });
              }
            }
          }
        *st = (uint32_t)ed.size();
      }
      lo[(size_t)w] = l;
      hi[(size_t)w] = h;
    }
  }, grain_of((int64_t)unit * kListTile * P * 3 * W32 * 4));
  auto up8 = [](int x) { return (x + 7) & ~7; };
  for (size_t j = 0; j < todo.size(); ++j) {
    ListScan& s = out[todo[j]];
    const auto at = (int64_t)j * units;
    s.lo = up8(*std::max_element(lo.begin() + at, lo.begin() + at + units));
    s.rows = s.lo + kListTile + up8(*std::max_element(hi.begin() + at, hi.begin() + at + units));
    // a whole number of equal TMA boxes of at most 256 rows
    const int boxes = (s.rows + 255) / 256;
    s.rows = up8((s.rows + boxes - 1) / boxes) * boxes;
    // each type's steps padded to whole blocks
    s.off.resize((size_t)n_tiles * kGroups * (P + 1));
    uint64_t total = 0;
    s.steps = 0;
    uint32_t* o = s.off.data();
    for (int64_t t = 0; t < n_tiles; ++t)
      for (int b = 0; b < kGroups; ++b) {
        const uint32_t* st = &s.start[(size_t)t * (kGroups * P + 1) + (size_t)b * P];
        for (int i = 0; i <= P; ++i) {
          *o++ = (uint32_t)total;
          if (i == P) break;
          const int q = type_at(i, P);
          const uint32_t ns = steps_of(st[q + 1] - st[q]);
          s.steps += ns;
          total += (ns + kGatherBlock - 1) / kGatherBlock;
        }
      }
    s.blocks = (int64_t)total;
  }
}

void band_tc_emit_lists(const bg_plan* p, unsigned orientations, const ListScan* s,
                        uint32_t* const* out) {
  const int P = p->P;
  const int64_t n_tiles = ((int64_t)p->K * p->S + kListTile - 1) / kListTile;
  std::vector<int> todo;
  int64_t steps = 0;
  for (int d = 0; d < 2; ++d)
    if (orientations >> d & 1) todo.push_back(d), steps += s[d].steps;
  const int64_t jobs = n_tiles * (int64_t)todo.size();
  parallel_ranges(jobs, [&](int64_t w0, int64_t w1) {
    std::vector<uint32_t> tmp;
    for (int64_t w = w0; w < w1; ++w) {
      const int tr = todo[(size_t)(w / n_tiles)];
      const int64_t t = w % n_tiles;
      const ListScan& c = s[tr];
      const uint32_t* ed = c.edges[(size_t)(t / c.unit)].data();
      const uint32_t add = (uint32_t)(c.lo - 2048);
      for (int b = 0; b < kGroups; ++b) {
        const uint32_t* st = &c.start[(size_t)t * (kGroups * P + 1) + (size_t)b * P];
        const uint32_t* off = &c.off[((size_t)t * kGroups + b) * (P + 1)];
        for (int i = 0; i < P; ++i) {
          const int q = type_at(i, P);
          emit_type(ed + st[q], (int)(st[q + 1] - st[q]), add, (uint32_t)c.rows,
                    out[tr] + (size_t)off[i] * 32 * kGatherBlock, tmp);
        }
      }
    }
  }, grain_of(jobs ? 512 * steps / jobs : 1));
}

int64_t band_tc_list_steps(const bg_plan* p, bool transposed) {
  ListScan s[2];
  band_tc_scan_lists(p, 1u << transposed, s);
  return s[transposed].steps;
}

void band_tc_host_lists(const bg_plan* p, bool transposed, GatherLists& out) {
  ListScan s[2];
  band_tc_scan_lists(p, 1u << transposed, s);
  ListScan& c = s[transposed];
  out.lo = c.lo, out.rows = c.rows, out.steps = c.steps, out.blocks = c.blocks;
  if (c.blocks >> 31) return;  // the caller checks `blocks`
  out.words.resize((size_t)c.blocks * 32 * kGatherBlock);
  uint32_t* const to[2] = {out.words.data(), out.words.data()};
  band_tc_emit_lists(p, 1u << transposed, s, to);
  out.off = std::move(c.off);
}

}  // namespace bg
