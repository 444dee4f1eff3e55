// SharedVectors of the shared-A batch with the runtime's calls answered here (device memory is host
// memory): what read() staged on the device is the same after to_host(), which gives the device's room
// back; without device memory read() stages on the host.  Built and run by
// tests/test_shared_inputs_cpu.py.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../paper_1805_12344_gb300/csrc/abip_internal.h"

static bool g_room = true;
static int g_held = 0;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) {
  if (!g_room) return cudaErrorMemoryAllocation;
  *p = std::malloc(n);
  ++g_held;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::free(p);
  --g_held;
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
}

int main() {
  const int count = 70, m = 3, n = 5;
  std::vector<std::vector<double>> bv(count), cv(count);
  std::vector<const double*> b, c;
  for (int k = 0; k < count; ++k) {
    for (int i = 0; i < m; ++i) bv[k].push_back(100.0 * k + i);
    for (int j = 0; j < n; ++j) cv[k].push_back(-100.0 * k - j);
    b.push_back(bv[k].data());
    c.push_back(cv[k].data());
  }
  for (int room = 0; room < 2; ++room) {
    g_room = room != 0;
    abip::SharedVectors v;
    int bad = 0;
    if (v.read(count, m, n, b.data(), c.data(), 0, bad) != cudaSuccess || bad != -1 || v.on_host != !g_room) return std::puts("FAIL read"), 1;
    if (v.to_host(count, m, n) != g_room || !v.on_host || g_held != 0) return std::puts("FAIL to_host"), 1;
    for (int k = 0; k < count; ++k)
      if (std::memcmp(v.b + k * m, b[k], m * 8) != 0 || std::memcmp(v.c + k * n, c[k], n * 8) != 0) return std::puts("FAIL values"), 1;
  }
  std::puts("ok");
  return 0;
}
