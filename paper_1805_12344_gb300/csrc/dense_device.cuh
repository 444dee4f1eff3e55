// Device routines shared by the dense kernels of one CTA per LP and of a group of CTAs.
#pragma once

#include "abip_device.cuh"

namespace abip {
namespace dense {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// Sums of P per-lane values over the warp, P a power of two <= 32: halving exchanges, then a
// butterfly over the rest.  Lane l receives the sum of value l >> (5 - log2 P).  Every sum is
// formed by the additions of warp_sum's butterfly, in its order, so the bits are the same; P
// sums take P - 1 + 5 - log2 P additions where P butterflies take 5 P.
template <int P, typename T>
__device__ __forceinline__ T sum_together(T (&a)[P], int lane) {
  int o = 16;
#pragma unroll
  for (int h = P / 2; h > 0; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const T send = up ? a[k] : a[k + h];
      const T keep = up ? a[k + h] : a[k];
      a[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  T v = a[0];
#pragma unroll
  for (; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// w <- L^{-1} w, L lower triangular (row-major, leading dimension m), w in shared memory.
template <typename T>
__device__ void trsv_lower(const T* __restrict__ L, int m, T* w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int kb = 0; kb < m; kb += 32) {
    const int nb = min(32, m - kb);
    if (wid == 0) {
      T wl = lane < nb ? w[kb + lane] : T(0);
      for (int j = 0; j < nb; ++j) {
        if (lane == j) wl = wl / L[(size_t)(kb + j) * m + kb + j];
        const T wj = __shfl_sync(0xffffffffu, wl, j);
        if (lane > j && lane < nb) wl -= L[(size_t)(kb + lane) * m + kb + j] * wj;
      }
      if (lane < nb) w[kb + lane] = wl;
    }
    __syncthreads();
    const T wb = lane < nb ? w[kb + lane] : T(0);
    for (int i = kb + nb + wid; i < m; i += kWarps) {
      T a = lane < nb ? L[(size_t)i * m + kb + lane] * wb : T(0);
      a = warp_sum(a);
      if (lane == 0) w[i] -= a;
    }
    __syncthreads();
  }
}

// w <- L^{-T} w.
template <typename T>
__device__ void trsv_lower_t(const T* __restrict__ L, int m, T* w) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nblk = (m + 31) / 32;
  for (int bk = nblk - 1; bk >= 0; --bk) {
    const int kb = bk * 32;
    const int nb = min(32, m - kb);
    if (wid == 0) {
      T wl = lane < nb ? w[kb + lane] : T(0);
      for (int j = nb - 1; j >= 0; --j) {
        if (lane == j) wl = wl / L[(size_t)(kb + j) * m + kb + j];
        const T zj = __shfl_sync(0xffffffffu, wl, j);
        if (lane < j) wl -= L[(size_t)(kb + j) * m + kb + lane] * zj;
      }
      if (lane < nb) w[kb + lane] = wl;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kb; i += kThreads) {
      T a = T(0);
      for (int j = 0; j < nb; ++j) a += L[(size_t)(kb + j) * m + i] * w[kb + j];
      w[i] -= a;
    }
    __syncthreads();
  }
}

}  // namespace dense
}  // namespace abip
