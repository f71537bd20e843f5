// Test helper for tests/test_edge_lists.py: bg_plan_upload on a fake of the CUDA runtime calls it makes
// (linked with --wrap), device memory being host memory, so that an allocation can be made to fail
// without a GPU.
//
//   upload_probe S FAIL_ALLOC    (the FAIL_ALLOC-th device allocation fails; 0: none)
//   prints: status, allocations made, uses tensor cores, lists forward, lists backward, runtime error
//   left behind, bytes of device memory still held after bg_plan_free beyond the library's own word
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <iterator>
#include <map>
#include <random>
#include <vector>

#include "bandggnn.h"

namespace {
int g_fail_alloc = 0, g_allocs = 0;
cudaError_t g_last = cudaSuccess;
std::map<char*, size_t> g_held;
cudaError_t err(cudaError_t e) { return e == cudaSuccess ? e : (g_last = e); }
alignas(256) char g_symbol[1024];
int fake_encode() { return 0; }
}  // namespace

extern "C" {
cudaError_t __wrap_cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t __wrap_cudaSetDevice(int) { return cudaSuccess; }
cudaError_t __wrap_cudaMalloc(void** p, size_t n) {
  if (++g_allocs == g_fail_alloc) return err(cudaErrorMemoryAllocation);
  char* q = static_cast<char*>(std::aligned_alloc(256, (n + 255) / 256 * 256));
  std::memset(q, 0, n);
  g_held[q] = n;
  *p = q;
  return cudaSuccess;
}
cudaError_t __wrap_cudaFree(void* p) {
  if (p && !g_held.erase(static_cast<char*>(p))) return err(cudaErrorInvalidValue);
  std::free(p);
  return cudaSuccess;
}
cudaError_t __wrap_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  char* dev = static_cast<char*>(kind == cudaMemcpyDeviceToHost ? const_cast<void*>(s) : d);
  auto it = g_held.upper_bound(dev);
  if (it == g_held.begin() || dev + n > std::prev(it)->first + std::prev(it)->second)
    return err(cudaErrorInvalidValue);
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t __wrap_cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t __wrap_cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
// kernels do nothing: the edge counts stay as the allocation is, 0
cudaError_t __wrap_cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t __wrap_cudaGetLastError() { cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t __wrap_cudaGetSymbolAddress(void** p, const void*) { *p = g_symbol; return cudaSuccess; }
cudaError_t __wrap_cudaFuncGetAttributes(cudaFuncAttributes*, const void*) { return cudaSuccess; }
cudaError_t __wrap_cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                                    cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&fake_encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  const int S = std::atoi(argv[1]);
  const int P = 4, n = 900, m = 4000;
  std::mt19937 r(5);
  std::vector<int32_t> src(m), dst(m), et(m);
  for (int e = 0; e < m; ++e) {
    src[e] = (int32_t)(r() % n);
    dst[e] = std::min(n - 1, std::max(0, src[e] + (int32_t)(r() % 81) - 40));
    et[e] = (int32_t)(r() % P);
  }
  const bg_graph g{n, m, src.data(), dst.data(), et.data()};
  bg_plan* p = nullptr;
  if (bg_band_plan(&g, 1, P, S, 0, BG_RCM | BG_KEEP_IF_BETTER, &p) != BG_OK) return 3;
  g_fail_alloc = std::atoi(argv[2]);
  const int rc = bg_plan_upload(p, nullptr);
  const cudaError_t left = __wrap_cudaGetLastError();
  std::printf("%d %d %d %d %d %d ", rc, g_allocs, bg_band_uses_tensor_cores(p, BG_BF16, 64),
              bg_band_uses_lists(p, BG_BF16, 64, BG_OP_PROPAGATE_FWD),
              bg_band_uses_lists(p, BG_BF16, 64, BG_OP_PROPAGATE_BWD), (int)left);
  bg_plan_free(p);
  size_t held = 0;
  for (auto& h : g_held) held += h.second == 256 ? 0 : h.second;
  std::printf("%zu\n", held);
  return 0;
}
