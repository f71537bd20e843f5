// Test helper for tests/test_edge_lists.py: plans the graphs of a binary file and writes the plan's
// bit tiles of one orientation together with the edge lists built from them.
//
//   lists_probe IN OUT P S TRANSPOSED
//   IN:  int32 n_graphs, then per graph int32 n_nodes, int64 n_edges, int32 src[], dst[], etype[]
//   OUT: int32 K, lo, rows; int64 steps, blocks, steps as counted ahead, word counts (masks, words,
//        off); then the arrays
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "band_tc.h"

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  const int P = std::atoi(argv[3]), S = std::atoi(argv[4]), tr = std::atoi(argv[5]);
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 3;
  int32_t ng = 0;
  if (std::fread(&ng, 4, 1, f) != 1 || ng < 1) return 4;
  std::vector<std::vector<int32_t>> a(3 * (size_t)ng);
  std::vector<bg_graph> gs(ng);
  for (int g = 0; g < ng; ++g) {
    int32_t n = 0;
    int64_t m = 0;
    if (std::fread(&n, 4, 1, f) != 1 || std::fread(&m, 8, 1, f) != 1 || m < 0) return 5;
    for (int k = 0; k < 3; ++k) {
      a[3 * g + k].resize(m);
      if (m && std::fread(a[3 * g + k].data(), 4, m, f) != (size_t)m) return 6;
    }
    gs[g] = bg_graph{n, m, a[3 * g].data(), a[3 * g + 1].data(), a[3 * g + 2].data()};
  }
  std::fclose(f);
  bg_plan* pl = nullptr;
  if (bg_band_plan(gs.data(), ng, P, S, 0, BG_RCM | BG_KEEP_IF_BETTER, &pl) != BG_OK) return 7;
  bg::GatherLists l;
  bg::band_tc_host_lists(pl, tr != 0, l);
  const auto& m = tr ? pl->masksT : pl->masks;
  FILE* o = std::fopen(argv[2], "wb");
  if (!o) return 8;
  const int32_t head[3] = {pl->K, l.lo, l.rows};
  const int64_t counts[6] = {l.steps, l.blocks, bg::band_tc_list_steps(pl, tr != 0),
                             (int64_t)m.size(), (int64_t)l.words.size(), (int64_t)l.off.size()};
  std::fwrite(head, 4, 3, o);
  std::fwrite(counts, 8, 6, o);
  std::fwrite(m.data(), 4, m.size(), o);
  std::fwrite(l.words.data(), 4, l.words.size(), o);
  std::fwrite(l.off.data(), 4, l.off.size(), o);
  std::fclose(o);
  bg_plan_free(pl);
  return 0;
}
