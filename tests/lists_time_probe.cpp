// Test helper for tests/test_edge_lists.py: plans the graphs of a binary file (as lists_probe.cpp) and
// prints the least time, of several runs in turn, of the host work an upload does with and without
// edge lists: degrees and chunks of both orientations, and the lists of both.
//
//   lists_time_probe IN P S C1 RUNS
#include <algorithm>
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <memory>
#include <vector>

#include "band_tc.h"

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  const int P = std::atoi(argv[2]), S = std::atoi(argv[3]), C1 = std::atoi(argv[4]), runs = std::atoi(argv[5]);
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
  using clk = std::chrono::steady_clock;
  auto ms = [](clk::time_point t) { return std::chrono::duration<double, std::milli>(clk::now() - t).count(); };
  double tiles = 1e30, lists = 1e30;
  for (int r = 0; r < runs; ++r) {
    auto t = clk::now();
    std::vector<uint16_t> deg;
    bg::band_tc_host_degrees(pl, deg);
    const size_t words = (size_t)pl->K * S / 128 * P * C1 * 128 * 4;
    for (int d = 0; d < 2; ++d) {
      std::unique_ptr<uint32_t[]> m(new uint32_t[words]);
      bg::band_tc_host_chunks(pl, C1, d != 0, m.get());
    }
    tiles = std::min(tiles, ms(t));
    t = clk::now();
    for (int d = 0; d < 2; ++d) {
      bg::GatherLists l;
      bg::band_tc_host_lists(pl, d != 0, l);
    }
    lists = std::min(lists, ms(t));
  }
  std::printf("%.6f %.6f\n", tiles, lists);
  bg_plan_free(pl);
  return 0;
}
