// What the dense paths do on a device that holds no cluster of 16 CTAs (or of 8, 4, 2): the planning
// and launching routines of the library's objects, with the runtime calls that ask the device replaced
// by the ones below.  Built and run by tests/test_cluster_plan_cpu.py; prints "ok" and exits 0, or
// names what broke and exits 1.
#include <cstdio>
#include <string>
#include <vector>

#include "../paper_1805_12344_gb300/csrc/abip_internal.h"

static int g_most = 16;        // CTAs of the largest cluster that the device holds
static int g_launched = 0;     // cluster size of the last launch
static size_t g_smem = 0;

static int cluster_of(const cudaLaunchConfig_t* c) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)c->attrs[i].val.clusterDim.x;
  return 1;
}

extern "C" {
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  const int size = cluster_of(c);
  *n = size <= g_most ? 152 / size : 0;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**) {
  g_launched = cluster_of(c);
  g_smem = c->dynamicSmemBytes;
  return g_launched <= g_most ? cudaSuccess : cudaErrorInvalidConfiguration;
}
}

static int fail(const std::string& what, int m, int n) {
  std::printf("FAIL %s (%d x %d, clusters up to %d)\n", what.c_str(), m, n, g_most);
  return 1;
}

int main() {
  const std::vector<std::pair<int, int>> sizes = {{2, 3}, {50, 120}, {97, 97}, {201, 611}, {512, 1154}, {1, 3001}, {100, 5000}, {1500, 3000}};
  for (g_most = 16; g_most >= 4; g_most /= 2)
    for (auto [m, n] : sizes) {
      abip::DenseGroupPlan f64{}, mixed{};
      // FP64: the vectors of these sizes fit clusters of 4 and more
      if (!abip::plan_dense_cluster(&m, &n, 1, 16, 223 * 1024, f64)) return fail("no plan in FP64", m, n);
      if (f64.ctas > g_most) return fail("FP64 plan larger than the device's clusters", m, n);
      g_launched = 0;
      if (abip::launch_dense_group(nullptr, 1, abip::DenseParams{}, nullptr, nullptr, f64, abip::GroupSparse{}, 0, nullptr, 0, 0, 0) !=
              cudaSuccess || g_launched != f64.ctas)
        return fail("FP64 launch", m, n);
      if (48 * m + 40 * n <= 200 * 1024) {
        if (!abip::plan_dense_mixed(&m, &n, 1, 16, 223 * 1024, mixed)) return fail("no plan in mixed precision", m, n);
        if (mixed.ctas > g_most) return fail("mixed plan larger than the device's clusters", m, n);
        g_launched = 0;
        if (abip::launch_dense_mixed(nullptr, 1, abip::DenseParams{}, nullptr, nullptr, mixed, 0, 0) != cudaSuccess || g_launched != mixed.ctas)
          return fail("mixed launch", m, n);
        if (g_smem != mixed.smem) return fail("mixed shared memory", m, n);
      }
    }
  for (g_most = 16; g_most >= 1; g_most /= 2) {
    g_launched = 0;
    if (abip::launch_dense_factor(nullptr, 1, 512, 152, 0) != cudaSuccess || g_launched < 1 || g_launched > g_most)
      return fail("factorisation", 512, 1154);
    // small LPs need no cluster at all
    int m = 50, n = 120;
    abip::DenseGroupPlan p{};
    if (!abip::plan_dense_cluster(&m, &n, 1, 8, 100 * 1024, p) || p.ctas > g_most) return fail("small FP64 plan", m, n);
    if (!abip::plan_dense_mixed(&m, &n, 1, 8, 100 * 1024, p) || p.ctas > g_most) return fail("small mixed plan", m, n);
    std::vector<int32_t> rp(256), cp(961);
    for (int i = 0; i <= 255; ++i) rp[i] = 8 * i;
    for (int j = 0; j <= 960; ++j) cp[j] = (int)(2040ll * j / 960);
    abip::GroupSparse sp{};
    int parts = 0;
    if (!abip::plan_sparse_group(255, 960, rp.data(), cp.data(), 152, sp, p, parts) || p.ctas > g_most) return fail("sparse plan", 255, 960);
  }
  g_most = 0;   // not even single CTAs of a cluster launch: no plan, and the caller's other path
  int m = 50, n = 120;
  abip::DenseGroupPlan p{};
  if (abip::plan_dense_cluster(&m, &n, 1, 8, 100 * 1024, p) || abip::plan_dense_mixed(&m, &n, 1, 8, 100 * 1024, p))
    return fail("a plan without a launch", m, n);
  std::printf("ok\n");
  return 0;
}
