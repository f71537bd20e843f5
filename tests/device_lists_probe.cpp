// Test helper for tests/test_edge_lists.py: plans the graphs of a binary file (as lists_probe.cpp),
// uploads the plan and compares the edge lists the device built with those the host builds.
//
//   device_lists_probe IN P S
//   prints, per orientation: 1 if the plan has lists on the device (0: nothing to compare), words that
//   differ, offsets that differ, 1 if window and sizes agree, blocks
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <vector>

#include "band_tc.h"

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  const int P = std::atoi(argv[2]), S = std::atoi(argv[3]);
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
  bg_plan* p = nullptr;
  if (bg_band_plan(gs.data(), ng, P, S, 0, BG_RCM | BG_KEEP_IF_BETTER, &p) != BG_OK) return 7;
  if (bg_plan_upload(p, nullptr) != BG_OK) return 8;
  for (int d = 0; d < 2; ++d) {
    if (!p->list_h[d]) {
      std::printf("0 0 0 0 0 ");
      continue;
    }
    bg::GatherLists l;
    bg::band_tc_host_lists(p, d != 0, l);
    std::vector<uint32_t> words(l.words.size()), off(l.off.size());
    if (cudaMemcpy(words.data(), p->d_glist[d], words.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess ||
        cudaMemcpy(off.data(), p->d_goff[d], off.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
      return 9;
    size_t dw = 0, doff = 0;
    for (size_t i = 0; i < words.size(); ++i) dw += words[i] != l.words[i];
    for (size_t i = 0; i < off.size(); ++i) doff += off[i] != l.off[i];
    std::printf("1 %zu %zu %d %lld ", dw, doff, p->g_lo[d] == l.lo && p->g_rows[d] == l.rows, (long long)l.blocks);
  }
  std::printf("\n");
  bg_plan_free(p);
  return 0;
}
