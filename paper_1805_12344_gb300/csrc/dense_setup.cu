// Setup of the dense path spread over the SMs: G = I + A A^T (Sec. 4.4) by output tiles,
// its Cholesky factor by a thread-block cluster per instance, and by column tiles the FP32
// explicit inverse of the mixed-precision path or the inverse of the factor of the FP64 path.
//
// What bounds it: the FP64 pipe (2 FMA per clock and SM).  A Gram of 512 x 1154 is 151 MFMA:
// 36 ms on one SM, 0.3 ms on 136 tiles over the SMs.  Every value is formed by the operations
// of the one-CTA routines (dense_solver.cu: gram, cholesky, trsv_lower, trsv_lower_t) in their
// order -- one chain of multiply-adds per entry -- so the factor and the inverse are the same
// bits whatever the split: the mixed path rounds its changes to FP32, and a last-bit
// difference in the factor would move those roundings.
// Measured, setup of one 512 x 1154 L1-SVM, one CTA -> this split: FP64 91 -> 7 ms, mixed
// precision (with the inverse) 585 -> 9 ms.
#include <algorithm>

#include <cooperative_groups.h>

#include "abip_device.cuh"
#include "abip_internal.h"

namespace cg = cooperative_groups;

namespace abip {
namespace {

constexpr int kThr = 256;
constexpr int kNB = 32;   // block columns of the factorisation and of the solves

// ---------------------------------------------------------------------------
// G = I + A A^T, lower triangle: 32 x 32 output tiles, 4 outputs per thread, each one chain
// over the columns of A in increasing order.  blockIdx.y: instance; the CTAs of a row share
// its tiles.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThr) gram_tiles_kernel(const DenseInst* __restrict__ insts) {
  constexpr int JC = 64;   // columns of A staged at a time
  __shared__ double Ti[32][JC + 1], Tk[32][JC + 1];
  const DenseInst& I = insts[blockIdx.y];
  const int m = I.m, n = I.n;
  const int64_t ld = I.ld;
  const double* __restrict__ A = I.A;
  const int nt = (m + 31) / 32, tiles = nt * (nt + 1) / 2;
  const int tr = threadIdx.x / 32, tc = threadIdx.x % 32;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
    int bi = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
    while ((bi + 1) * (bi + 2) / 2 <= t) ++bi;
    while (bi * (bi + 1) / 2 > t) --bi;
    const int bk = t - bi * (bi + 1) / 2;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j0 = 0; j0 < n; j0 += JC) {
      for (int e = threadIdx.x; e < 32 * JC; e += kThr) {
        const int r = e / JC, c = e % JC;
        const int gi = bi * 32 + r, gk = bk * 32 + r, gj = j0 + c;
        Ti[r][c] = (gi < m && gj < n) ? A[(size_t)gi * ld + gj] : 0.0;
        Tk[r][c] = (gk < m && gj < n) ? A[(size_t)gk * ld + gj] : 0.0;
      }
      __syncthreads();
#pragma unroll 8
      for (int c = 0; c < JC; ++c) {
        const double kv = Tk[tc][c];
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] += Ti[tr * 4 + q][c] * kv;
      }
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gi = bi * 32 + tr * 4 + q, gk = bk * 32 + tc;
      if (gi < m && gk <= gi) I.L[(size_t)gi * m + gk] = acc[q] + (gi == gk ? 1.0 : 0.0);
    }
  }
}

// G of a sparse A, lower triangle of the zeroed L: a warp per row i, over the entries (i, j) of
// the row in order, its lanes over the entries (k, j) of column j (k distinct: no duplicates)
__global__ void __launch_bounds__(kThr) gram_sparse_kernel(const DenseInst* __restrict__ inst, GroupSparse sp) {
  const int m = inst->m, lane = threadIdx.x & 31;
  for (int i = blockIdx.x * (kThr / 32) + (threadIdx.x >> 5); i < m; i += gridDim.x * (kThr / 32)) {
    double* row = inst->L + (size_t)i * m;
    for (int e = sp.rp[i]; e < sp.rp[i + 1]; ++e) {
      const int j = sp.ci[e];
      const double a = sp.va[e];
      for (int t = sp.cp[j] + lane; t < sp.cp[j + 1]; t += 32) {
        const int k = sp.ri[t];
        if (k <= i) row[k] += a * sp.cv[t];
      }
      __syncwarp();
    }
    if (lane == 0) row[i] += 1.0;
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Cholesky G = L L^T in place, one cluster per instance, right-looking by 32-wide block
// columns: every CTA factors the diagonal block for itself (a warp, one row per lane), the
// rows below and then the trailing 32 x 32 tiles are dealt out to the CTAs, two cluster
// barriers per block column.  Entry (i, j) receives -L_il L_jl for l = 0, 1, ..., j - 1 in
// that order as fused multiply-adds on the entry itself, as in the unblocked factorisation.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThr) chol_cluster_kernel(DenseInst* insts, int count) {
  __shared__ double D[kNB][kNB + 1];
  __shared__ double Pi[kNB][kNB + 1], Pj[kNB][kNB + 1];
  __shared__ int s_ok;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int nclusters = gridDim.x / C;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int id = blockIdx.x / C; id < count; id += nclusters) {
    DenseInst& I = insts[id];
    const int m = I.m;
    double* L = I.L;
    bool ok = true;
    for (int k0 = 0; k0 < m; k0 += kNB) {
      const int nb = min(kNB, m - k0);
      for (int e = threadIdx.x; e < kNB * kNB; e += kThr) {
        const int r = e / kNB, c = e % kNB;
        D[r][c] = (r < nb && c <= r) ? __ldcg(L + (size_t)(k0 + r) * m + k0 + c) : 0.0;
      }
      if (threadIdx.x == 0) s_ok = 1;
      __syncthreads();
      if (wid == 0) {
        for (int k = 0; k < nb; ++k) {
          const double d = D[k][k];
          if (!(d > 0.0) || !isfinite(d)) {
            if (lane == 0) s_ok = 0;
            break;
          }
          const double dk = sqrt(d);
          double lik = 0.0;
          if (lane > k && lane < nb) lik = D[lane][k] / dk;
          __syncwarp();
          if (lane == k) D[k][k] = dk;
          else if (lane > k && lane < nb) D[lane][k] = lik;
          __syncwarp();
          if (lane > k && lane < nb)
            for (int j = k + 1; j <= lane; ++j) D[lane][j] -= lik * D[j][k];
          __syncwarp();
        }
      }
      __syncthreads();
      ok = s_ok != 0;
      if (!ok) break;   // the same in every CTA: all factor the same block
      const int r0 = k0 + nb, rest = m - r0;
      // rows below the block: one thread per row, the rows dealt out by cluster rank
      for (int i = rank + C * threadIdx.x; i < rest; i += C * kThr) {
        double row[kNB];
        double* p = L + (size_t)(r0 + i) * m + k0;
#pragma unroll
        for (int k = 0; k < kNB; ++k) row[k] = k < nb ? __ldcg(p + k) : 0.0;
#pragma unroll
        for (int k = 0; k < kNB; ++k) {
          if (k >= nb) break;
          const double v = row[k] / D[k][k];
          row[k] = v;
#pragma unroll
          for (int j = k + 1; j < kNB; ++j) row[j] -= v * D[j][k];
        }
#pragma unroll
        for (int k = 0; k < kNB; ++k)
          if (k < nb) __stcg(p + k, row[k]);
      }
      cl.sync();   // the panel is complete; every CTA has read the old diagonal block
      if (rank == 0)
        for (int e = threadIdx.x; e < nb * nb; e += kThr) {
          const int r = e / nb, c = e % nb;
          if (c <= r) __stcg(L + (size_t)(k0 + r) * m + k0 + c, D[r][c]);
        }
      // trailing tiles (bi >= bj)
      const int nt = (rest + kNB - 1) / kNB, tiles = nt * (nt + 1) / 2;
      const int tr = threadIdx.x / 32, tc = threadIdx.x % 32;
      int bi = 0, bj = 0, at = 0;
      for (int t = rank; t < tiles; t += C) {
        for (; at < t; ++at) {
          if (bj == bi) { ++bi; bj = 0; }
          else ++bj;
        }
        const int i0 = r0 + bi * kNB, j0 = r0 + bj * kNB;
        for (int e = threadIdx.x; e < kNB * kNB; e += kThr) {
          const int r = e / kNB, c = e % kNB;
          Pi[r][c] = (i0 + r < m && c < nb) ? __ldcg(L + (size_t)(i0 + r) * m + k0 + c) : 0.0;
          Pj[r][c] = (j0 + r < m && c < nb) ? __ldcg(L + (size_t)(j0 + r) * m + k0 + c) : 0.0;
        }
        __syncthreads();
        double acc[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + tr * 4 + q, j = j0 + tc;
          acc[q] = (i < m && j <= i) ? __ldcg(L + (size_t)i * m + j) : 0.0;
        }
        for (int l = 0; l < nb; ++l) {
          const double b = Pj[tc][l];
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q] -= Pi[tr * 4 + q][l] * b;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int i = i0 + tr * 4 + q, j = j0 + tc;
          if (i < m && j <= i) __stcg(L + (size_t)i * m + j, acc[q]);
        }
        __syncthreads();
      }
      cl.sync();
    }
    if (!ok) {
      if (rank == 0 && threadIdx.x == 0) { I.err = DEV_ERR_CHOLESKY; I.status = 0; }
    } else {   // zero the strict upper triangle (kept clean for readers)
      const int64_t mm = (int64_t)m * m;
      for (int64_t e = (int64_t)rank * kThr + threadIdx.x; e < mm; e += (int64_t)C * kThr) {
        const int i = (int)(e / m), j = (int)(e % m);
        if (j > i) L[e] = 0.0;
      }
    }
    cl.sync();   // the shared tiles are free for the next instance
  }
}

// ---------------------------------------------------------------------------
// Inverses from L, Q columns per CTA: L z = e_col (L^{-1}) and L^T g = z (G^{-1}), one column per
// lane (32 / Q rows side by side in a warp).  Same operations per column as trsv_lower and
// trsv_lower_t: the 32 products of a block are summed in the order of their butterfly.
// ---------------------------------------------------------------------------
// the butterfly's sum over l of p(l): T(l, 16) = p(l) + p(l + 16), T(l, o) = T(l, 2o) + T(l + o, 2o)
// (p rounds its products, as the values that a butterfly exchanges are)
template <int O, typename P>
__device__ __forceinline__ double tree_sum(int l, P p) {
  if constexpr (O == 16) return p(l) + p(l + 16);
  else return tree_sum<2 * O>(l, p) + tree_sum<2 * O>(l + O, p);
}

template <int Q>
__global__ void __launch_bounds__(kThr) inverse_tiles_kernel(const DenseInst* __restrict__ insts) {
  constexpr int S = 32 / Q;                     // rows side by side in a warp
  constexpr int RL = Q == 32 ? 4 : Q == 8 ? 2 : 1;
  constexpr int ROWS = S * RL;                  // rows a warp takes at once, RL per lane; divides kNB
  extern __shared__ double W[];                 // m x Q
  __shared__ double Lb[kNB][kNB + 1];           // the diagonal block
  __shared__ double Lr[kThr / 32][ROWS][kNB];   // rows of the block column in flight, per warp
  const DenseInst& I = insts[blockIdx.y];
  if (I.err != 0) return;
  const int m = I.m;
  const double* __restrict__ L = I.L;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int col = lane % Q, sub = lane / Q;
  constexpr int kW = kThr / 32;
  for (int c0 = blockIdx.x * Q; c0 < m; c0 += gridDim.x * Q) {
    for (int e = threadIdx.x; e < m * Q; e += kThr) W[e] = (e / Q == c0 + e % Q) ? 1.0 : 0.0;
    __syncthreads();
    // L z = e_col: z is zero above the tile's block
    for (int kb = (c0 / kNB) * kNB; kb < m; kb += kNB) {
      const int nb = min(kNB, m - kb);
      for (int e = threadIdx.x; e < nb * nb; e += kThr) Lb[e / nb][e % nb] = L[(size_t)(kb + e / nb) * m + kb + e % nb];
      __syncthreads();
      if (wid == 0 && sub == 0) {
        double w[kNB];
#pragma unroll
        for (int r = 0; r < kNB; ++r) w[r] = r < nb ? W[(kb + r) * Q + col] : 0.0;
#pragma unroll
        for (int j = 0; j < kNB; ++j) {
          if (j >= nb) break;
          w[j] = w[j] / Lb[j][j];
#pragma unroll
          for (int r = j + 1; r < kNB; ++r)
            if (r < nb) w[r] -= Lb[r][j] * w[j];
        }
#pragma unroll
        for (int r = 0; r < kNB; ++r)
          if (r < nb) W[(kb + r) * Q + col] = w[r];
      }
      __syncthreads();
      // rows below exist only under a full block (nb = 32)
      for (int i0 = kb + nb + wid * ROWS; i0 < m; i0 += kW * ROWS) {
#pragma unroll
        for (int q = 0; q < ROWS; ++q) Lr[wid][q][lane] = i0 + q < m ? L[(size_t)(i0 + q) * m + kb + lane] : 0.0;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < RL; ++u) {
          const double* lr = Lr[wid][u * S + sub];
          const double a = tree_sum<1>(0, [&](int l) { return __dmul_rn(lr[l], W[(kb + l) * Q + col]); });
          const int i = i0 + u * S + sub;
          if (i < m) W[i * Q + col] -= a;
        }
        __syncwarp();
      }
      __syncthreads();
    }
    if (I.Li) {   // column c0 + q of L^{-1} is z
      const int mp = m + (m & 1);
      for (int e = threadIdx.x; e < m * Q; e += kThr) {
        if (c0 + e % Q < m) I.Li[(size_t)(e / Q) * mp + c0 + e % Q] = W[e];
        const int q = e / m, i = e % m;
        if (c0 + q < m) I.LiT[(size_t)(c0 + q) * mp + i] = W[i * Q + q];
      }
      __syncthreads();
      continue;
    }
    // L^T g = z
    for (int kb = ((m - 1) / kNB) * kNB; kb >= 0; kb -= kNB) {
      const int nb = min(kNB, m - kb);
      for (int e = threadIdx.x; e < nb * nb; e += kThr) Lb[e / nb][e % nb] = L[(size_t)(kb + e / nb) * m + kb + e % nb];
      __syncthreads();
      if (wid == 0 && sub == 0) {
        double w[kNB];
#pragma unroll
        for (int r = 0; r < kNB; ++r) w[r] = r < nb ? W[(kb + r) * Q + col] : 0.0;
#pragma unroll
        for (int j = kNB - 1; j >= 0; --j) {
          if (j < nb) {
            w[j] = w[j] / Lb[j][j];
#pragma unroll
            for (int r = 0; r < j; ++r) w[r] -= Lb[j][r] * w[j];
          }
        }
#pragma unroll
        for (int r = 0; r < kNB; ++r)
          if (r < nb) W[(kb + r) * Q + col] = w[r];
      }
      __syncthreads();
      for (int i0 = wid * ROWS; i0 < kb; i0 += kW * ROWS) {
        // columns i0 .. of the block's rows: kb is a multiple of ROWS, so i0 + q < kb
#pragma unroll
        for (int q = 0; q < ROWS; ++q) Lr[wid][q][lane] = lane < nb ? L[(size_t)(kb + lane) * m + i0 + q] : 0.0;
        __syncwarp();
        double a[RL];
#pragma unroll
        for (int u = 0; u < RL; ++u) a[u] = 0.0;
        for (int j = 0; j < nb; ++j) {
          const double wj = W[(kb + j) * Q + col];
#pragma unroll
          for (int u = 0; u < RL; ++u) a[u] += Lr[wid][u * S + sub][j] * wj;
        }
#pragma unroll
        for (int u = 0; u < RL; ++u) W[(i0 + u * S + sub) * Q + col] -= a[u];
        __syncwarp();
      }
      __syncthreads();
    }
    for (int e = threadIdx.x; e < m * Q; e += kThr) {
      const int q = e / m, i = e % m;
      if (c0 + q < m && I.Ginvf) I.Ginvf[(size_t)(c0 + q) * I.ldtf + i] = (float)W[i * Q + q];
    }
    if (I.Ginv)
      for (int e = threadIdx.x; e < m * Q; e += kThr)
        if (c0 + e % Q < m) I.Ginv[(size_t)(e / Q) * m + c0 + e % Q] = W[e];
    __syncthreads();
  }
}

// What a dense instance needs of its inputs, by 32 x 32 tiles of A: the FP64 values of an FP32
// source, the FP32 copies of A and A^T of the mixed path (padding is zero already), and a test
// of every value (bound by the tile's one read of A).
__global__ void __launch_bounds__(kThr) ingest_kernel(const DenseInst* __restrict__ insts, const DenseSource* __restrict__ src,
                                                      int* __restrict__ flags) {
  __shared__ double T[32][33];
  const DenseInst& I = insts[blockIdx.y];
  const DenseSource S = src[blockIdx.y];
  const int m = I.m, n = I.n;
  const int tm = (m + 31) / 32, tiles = tm * ((n + 31) / 32);
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  double* A = const_cast<double*>(I.A);
  float* Af = const_cast<float*>(I.Af);
  float* ATf = const_cast<float*>(I.ATf);
  bool bad = false;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int i0 = (t % tm) * 32, j0 = (t / tm) * 32;
    for (int r = row; r < 32; r += kThr / 32) {
      const int i = i0 + r, j = j0 + lane;
      double v = 0.0;
      if (i < m && j < n) {
        v = S.f32 ? (double)S.f32[(size_t)i * S.ld + j] : A[(size_t)i * I.ld + j];
        bad |= !isfinite(v);
        if (S.f32) A[(size_t)i * I.ld + j] = v;
        if (Af) Af[(size_t)i * I.ldf + j] = (float)v;
      }
      T[r][lane] = v;
    }
    __syncthreads();
    if (ATf)
      for (int r = row; r < 32; r += kThr / 32)
        if (j0 + r < n && i0 + lane < m) ATf[(size_t)(j0 + r) * I.ldtf + i0 + lane] = (float)T[lane][r];
    __syncthreads();
  }
  if (bad) atomicOr(flags + blockIdx.y, 1);
  if (blockIdx.x == 0) {
    bool vec = false;
    for (int i = threadIdx.x; i < m; i += kThr) vec |= !isfinite(I.b[i]);
    for (int j = threadIdx.x; j < n; j += kThr) vec |= !isfinite(I.c[j]);
    if (vec) atomicOr(flags + blockIdx.y, 2);
  }
}

// A^T, rows padded to an even length (the padding is zero already), 32 x 32 tiles
__global__ void __launch_bounds__(kThr) transpose_tiles_kernel(const DenseInst* __restrict__ insts) {
  __shared__ double T[32][33];
  const DenseInst& I = insts[blockIdx.y];
  const int m = I.m, n = I.n, mp = m + (m & 1);
  const int tm = (m + 31) / 32, tiles = tm * ((n + 31) / 32);
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
  for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int i0 = (t % tm) * 32, j0 = (t / tm) * 32;
    for (int r = row; r < 32; r += kThr / 32)
      T[r][lane] = (i0 + r < m && j0 + lane < n) ? I.A[(size_t)(i0 + r) * I.ld + j0 + lane] : 0.0;
    __syncthreads();
    for (int r = row; r < 32; r += kThr / 32)
      if (j0 + r < n && i0 + lane < m) I.AT[(size_t)(j0 + r) * mp + i0 + lane] = T[lane][r];
    __syncthreads();
  }
}

constexpr size_t kInverseSmemMax = 200 * 1024;   // beside at most 25 KB of static shared memory
template <int Q>
cudaError_t launch_inverse(DenseInst* inst, int count, int mmax, int sms, cudaStream_t st) {
  const size_t smem = (size_t)mmax * Q * sizeof(double);
  // one limit whatever the call needs: it is the process's, and other threads set it too
  cudaError_t e = cudaFuncSetAttribute(inverse_tiles_kernel<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kInverseSmemMax);
  if (e != cudaSuccess) return e;
  for (int k0 = 0; k0 < count; k0 += 32768) {   // gridDim.y is limited to 65535
    const int cnt = std::min(32768, count - k0);
    inverse_tiles_kernel<Q><<<dim3((mmax + Q - 1) / Q, cnt), kThr, smem, st>>>(inst + k0);
  }
  return cudaGetLastError();
}

cudaError_t launch_cholesky(DenseInst* inst, int count, int mmax, int sms, cudaStream_t st) {
  const int nt = (mmax + 31) / 32, tiles = nt * (nt + 1) / 2;
  // CTAs per factorisation: a power of two up to 16 while the SMs outnumber the CTAs and a
  // CTA has more than one tile of the first trailing update, and a cluster of them fits the device
  int C = 1;
  while (C < 16 && 2 * C * count <= sms && 2 * C <= tiles) C *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThr);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (;; C /= 2) {
    at[0].val.clusterDim.x = (unsigned)C;
    cfg.gridDim = dim3((unsigned)(std::min(count, 4 * sms) * C));
    if (C == 1) break;
    cudaError_t e = cudaSuccess;
    if (C > 8) e = cudaFuncSetAttribute(chol_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    int n = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, chol_cluster_kernel, &cfg);
    if (e == cudaSuccess && n > 0) break;
    cudaGetLastError();
  }
  return cudaLaunchKernelEx(&cfg, chol_cluster_kernel, inst, count);
}

}  // namespace

cudaError_t launch_dense_factor(DenseInst* inst, int count, int mmax, int sms, cudaStream_t st) {
  const int nt = (mmax + 31) / 32, tiles = nt * (nt + 1) / 2;
  for (int k0 = 0; k0 < count; k0 += 32768) {
    const int cnt = std::min(32768, count - k0);
    // enough CTAs to fill the SMs a few times; the rest of an instance's tiles in a loop
    const int gx = std::max(1, std::min(tiles, (8 * sms + cnt - 1) / cnt));
    gram_tiles_kernel<<<dim3(gx, cnt), kThr, 0, st>>>(inst + k0);
  }
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_cholesky(inst, count, mmax, sms, st);
}

cudaError_t launch_sparse_factor(DenseInst* inst, int m, const GroupSparse& sp, int sms, cudaStream_t st) {
  gram_sparse_kernel<<<std::max(1, std::min(4 * sms, (m + 7) / 8)), kThr, 0, st>>>(inst, sp);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_cholesky(inst, 1, m, sms, st);
}

cudaError_t launch_dense_ingest(const DenseInst* inst, const DenseSource* src, int* flags, int count, int mmax, int nmax,
                                int sms, cudaStream_t st) {
  const int64_t tiles = (int64_t)((mmax + 31) / 32) * ((nmax + 31) / 32);
  for (int k0 = 0; k0 < count; k0 += 32768) {
    const int cnt = std::min(32768, count - k0);
    const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (8 * sms + cnt - 1) / cnt));
    ingest_kernel<<<dim3(gx, cnt), kThr, 0, st>>>(inst + k0, src + k0, flags + k0);
  }
  return cudaGetLastError();
}

cudaError_t launch_dense_transpose(DenseInst* inst, int count, int mmax, int nmax, int sms, cudaStream_t st) {
  const int64_t tiles = (int64_t)((mmax + 31) / 32) * ((nmax + 31) / 32);
  for (int k0 = 0; k0 < count; k0 += 32768) {
    const int cnt = std::min(32768, count - k0);
    const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (8 * sms + cnt - 1) / cnt));
    transpose_tiles_kernel<<<dim3(gx, cnt), kThr, 0, st>>>(inst + k0);
  }
  return cudaGetLastError();
}

cudaError_t launch_dense_inverse(DenseInst* inst, int count, int mmax, int sms, cudaStream_t st) {
  // Columns per CTA.  32 lanes of columns use the FP64 pipe best and serve a batch that fills
  // the SMs by itself; fewer columns spread a small one over more SMs, and keep the m x Q
  // working set inside the shared memory of a tall instance.
  const int64_t tiles32 = (int64_t)count * ((mmax + 31) / 32);
  if (tiles32 >= 2 * (int64_t)sms && (size_t)mmax * 32 * 8 <= 100 * 1024) return launch_inverse<32>(inst, count, mmax, sms, st);
  if (tiles32 * 4 >= 2 * (int64_t)sms && (size_t)mmax * 8 * 8 <= 200 * 1024) return launch_inverse<8>(inst, count, mmax, sms, st);
  return launch_inverse<4>(inst, count, mmax, sms, st);
}

}  // namespace abip
