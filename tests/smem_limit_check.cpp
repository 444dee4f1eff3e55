// A kernel's dynamic shared-memory limit is one value for the process: a call that set it to what it
// needs itself would take it away from a call in another thread that has set it and not yet launched.
// launch_dense_inverse with the runtime's calls answered here: every call sets the same limit for a
// kernel, and no launch needs more.  Built and run by tests/test_smem_limit_cpu.py.
#include <cstdio>
#include <map>

#include "../paper_1805_12344_gb300/csrc/abip_internal.h"

static std::map<const void*, int> g_limit;
static bool g_ok = true;

extern "C" {
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (g_limit.count(f) && g_limit[f] != v) g_ok = false;
    g_limit[f] = v;
  }
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) {
  if (smem > 48 * 1024 && (!g_limit.count(f) || (size_t)g_limit[f] < smem)) g_ok = false;
  return cudaSuccess;
}
}

int main() {
  // instances and rows: four, eight and 32 columns a CTA, up to the rows that the shared-matrix batch takes
  for (int count : {1, 3, 40, 400})
    for (int m : {1, 33, 400, 1600, 3200, 6400})
      if (abip::launch_dense_inverse(nullptr, count, m, 152, 0) != cudaSuccess) g_ok = false;
  std::printf(g_ok && g_limit.size() == 3 ? "ok\n" : "FAIL limits that differ, or too small, for %zu kernels\n", g_limit.size());
  return g_ok && g_limit.size() == 3 ? 0 : 1;
}
