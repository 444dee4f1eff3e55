// Dense ABIP in FP64 with a group of CTAs per LP: a thread-block cluster (1 .. 16 CTAs) per
// instance of a batch, or a cooperative grid for one large LP.
//
// What bounds it: the FP64 pipe, 2 FMA per clock and SM on this part, so an LP on one SM pays
// its 3 m n + m^2 multiply-adds per update at 1/152 of the chip; and, for a small LP, the chain
// of dependent phases.  Hence
//  * the rows of A and of the factor's inverse and the columns of A (rows of the stored A^T)
//    are dealt out to the CTAs of the group; every CTA keeps the vectors q, t, z_y, x and s
//    whole in shared memory and publishes its part of each (distributed shared memory in a
//    cluster, L2 in a grid);
//  * z_y = G^{-1} q is two products, t = L^{-1} q and z_y = L^{-T} t, with the inverse of the
//    factor formed at setup, instead of two sweeps of m / 32 serial blocks.  One product with
//    G^{-1} itself would save a barrier, but its error is larger than the sweeps' (x of a 512 x
//    1154 L1-SVM after 60 updates, relative: sweeps 5.0e-14, G^{-1} 6.1e-13, this 3.7e-14);
//  * A^T y follows from the update's linearity, y <- alpha u_y + (1 - alpha) y, whose error does
//    not grow (|1 - alpha| < 1) and which only the tests of Sec. 4.1 read: three products with
//    the entries of A per update instead of four;
//  * eight rows (or four with two vectors) per warp, their sums reduced together: 9 additions
//    for 8 sums where butterflies take 40 -- a warp-wide FP64 addition costs 16 clocks here;
//  * what a CTA reads every update (its rows of the matrices and of the vectors) is copied to
//    shared memory when it fits.
// The same kernel serves the sparse direct projection of an LP with few rows (SPARSE): the
// products with A run over its CSR rows and columns, L^{-1} stays dense.
//  * H^T z, which fixes (t1, t2), needs no z: H^T M^{-1} w = (M^{-T} H)^T w, so its sums over
//    w = (y, x + s) join the test sums and the scalars' own step runs on one warp beside the
//    products of the others; the tests are decided the same way, beside t = L^{-1} q, which is
//    dropped when the decision is not another update.
// One update has four barriers of the group: products and all sums | t | z_y | x, s.
// Measured, us per update, one CTA with triangular sweeps -> this kernel: 50 x 120 76.9 -> 9.8
// (the chain of dependent FP64 operations: about 100 clocks each, four barriers of 500),
// 512 x 1154 1564 -> 22 over the grid, the slowest of 64 LPs of m 16 .. 256 621 -> 60.
#include <algorithm>

#include <cooperative_groups.h>

#include "abip_device.cuh"
#include "abip_internal.h"
#include "barrier_refined.h"
#include "dense_device.cuh"

namespace cg = cooperative_groups;

namespace abip {
namespace {

using dense::kWarps;
using dense::sum_together;
constexpr int kThr = dense::kThreads;
constexpr int kSums = 11;   // the nine of the tests and the two of H^T z

// The order of the sums over rows and columns follows from the LP alone, whatever group solves it, so
// that its bits do not follow the batch it is in.  The LP has P parts (DenseInst::parts, the most CTAs
// that its work is worth in a cluster) of nine cells each: runs of rows and of columns.  A cell's sums
// are chains in order, a part's nine are joined by a fixed tree and the parts by another.  A CTA owns
// whole parts or, in the grid, a cell: 144 is the largest count up to the chip's 152 SMs that 16
// parts divide.  Against sums in the order of the CTAs' own elements, us per update: 50 x 120 9.9 -> 9.8,
// 512 x 1154 22.3 -> 22.1, 16 x 16 grid flow 11.5 -> 11.4; 32 x 32 and 39 x 39 on 144 CTAs instead of
// 152 21.7 -> 22.6 and 27.8 -> 30.2.
constexpr int kPerPart = 9, kMaxParts = 16;
constexpr int kGridCtas = kPerPart * kMaxParts;
// the first of `len` elements that rank r of a group of `size` owns; ranks past the parts own none
__host__ __device__ __forceinline__ int own_start(int r, int size, int parts, bool grid, int len) {
  const int C = grid ? kGridCtas : size < parts ? size : parts;
  return (int)((int64_t)(r < C ? r : C) * len / C);
}
// most elements that a CTA owns
__host__ __device__ __forceinline__ int own_room(int size, int parts, bool grid, int len) {
  const int C = grid ? kGridCtas : size < parts ? size : parts;
  return (len + C - 1) / C;
}

enum Act : int { ACT_STEP = 0, ACT_WARM = 1, ACT_STOP = 2 };

// out(which, i, sum_j M[row0 + i][j] v_which[j]) for i < rows: R rows per warp at a time, NV
// vectors; rows of M are ld (even) doubles, 16-byte aligned and zero-padded like v0, v1.
// By the warps from W0 on.
template <int R, int NV, int W0, typename F>
__device__ __forceinline__ void dots(const double* M, int64_t ld, int rows, const double* v0, const double* v1, F out) {
  constexpr int P = R * NV;
  constexpr int kShift = P == 16 ? 1 : P == 8 ? 2 : P == 4 ? 3 : P == 2 ? 4 : 5;
  const int lane = threadIdx.x & 31, wid = (int)(threadIdx.x >> 5) - W0;
  const int nq = (int)(ld >> 1);
  if (wid < 0) return;
  for (int g = wid * R; g < rows; g += (kWarps - W0) * R) {
    double a[P];
#pragma unroll
    for (int k = 0; k < P; ++k) a[k] = 0.0;
    const double2* r[R];
#pragma unroll
    for (int u = 0; u < R; ++u) r[u] = reinterpret_cast<const double2*>(M + (size_t)min(g + u, rows - 1) * ld);
#pragma unroll(R >= 4 ? 1 : 4)
    for (int t = lane; t < nq; t += 32) {
      const double2 x = reinterpret_cast<const double2*>(v0)[t];
      double2 z = x;
      if (NV == 2) z = reinterpret_cast<const double2*>(v1)[t];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const double2 w = r[u][t];
        a[u] += w.x * x.x;
        if (NV == 2) a[R + u] += w.x * z.x;
        a[u] += w.y * x.y;
        if (NV == 2) a[R + u] += w.y * z.y;
      }
    }
    const double v = sum_together<P>(a, lane);
    if ((lane & ((1 << kShift) - 1)) == 0) {
      const int k = lane >> kShift, u = k % R;
      if (g + u < rows) out(k / R, g + u, v);
    }
  }
}

// rows per warp by the rows of the CTA: all warps busy first, then more sums per reduction
template <int NV, int W0, typename F>
__device__ __forceinline__ void dots_any(const double* M, int64_t ld, int rows, const double* v0, const double* v1, F out) {
  constexpr int W = kWarps - W0;
  if (rows > 4 * W) dots<8, NV, W0>(M, ld, rows, v0, v1, out);
  else if (rows > 2 * W) dots<4, NV, W0>(M, ld, rows, v0, v1, out);
  else if (rows > W) dots<2, NV, W0>(M, ld, rows, v0, v1, out);
  else dots<1, NV, W0>(M, ld, rows, v0, v1, out);
}

// out(k, sum_j M[k][j] v[j]) for the CTA's rows k < rows of a triangular M, row k being row
// rank + size k of the matrix at M + k * stride: dealt out in turn, since the rows grow (LOWER)
// or shrink in length.  Only the triangle is read, in pairs of columns and to the longest of
// the R rows that a warp has at once (the entries beyond are stored zeros).  By all warps but
// the first, which has the scalars' work meanwhile.
template <int R, bool LOWER, typename F>
__device__ __forceinline__ void tri_dots(const double* M, int64_t stride, int rows, int rank, int size, int nq,
                                         const double* v, F out) {
  constexpr int kShift = R == 8 ? 2 : R == 4 ? 3 : R == 2 ? 4 : 5;
  const int lane = threadIdx.x & 31, wid = (int)(threadIdx.x >> 5) - 1;
  if (wid < 0) return;
  for (int g = wid * R; g < rows; g += (kWarps - 1) * R) {
    double a[R];
    const double2* r[R];
#pragma unroll
    for (int u = 0; u < R; ++u) {
      a[u] = 0.0;
      r[u] = reinterpret_cast<const double2*>(M + (size_t)min(g + u, rows - 1) * stride);
    }
    const int t0 = LOWER ? 0 : ((rank + size * g) >> 1) & ~31;   // a lane sums the same pairs in every group
    const int t1 = LOWER ? ((rank + size * min(g + R - 1, rows - 1)) >> 1) + 1 : nq;
#pragma unroll(R >= 4 ? 1 : 4)
    for (int t = t0 + lane; t < t1; t += 32) {
      const double2 x = reinterpret_cast<const double2*>(v)[t];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        const double2 w = r[u][t];
        a[u] += w.x * x.x;
        a[u] += w.y * x.y;
      }
    }
    const double d = sum_together<R>(a, lane);
    if ((lane & ((1 << kShift) - 1)) == 0) {
      const int u = lane >> kShift;
      if (g + u < rows) out(g + u, d);
    }
  }
}
template <bool LOWER, typename F>
__device__ __forceinline__ void tri_any(const double* M, int64_t stride, int rows, int rank, int size, int nq,
                                        const double* v, F out) {
  constexpr int W = kWarps - 1;
  if (rows > 4 * W) tri_dots<8, LOWER>(M, stride, rows, rank, size, nq, v, out);
  else if (rows > 2 * W) tri_dots<4, LOWER>(M, stride, rows, rank, size, nq, v, out);
  else if (rows > W) tri_dots<2, LOWER>(M, stride, rows, rank, size, nq, v, out);
  else tri_dots<1, LOWER>(M, stride, rows, rank, size, nq, v, out);
}

// The group of CTAs that solves an LP: a cluster (GRID = false) or the cooperative grid.
template <bool GRID>
struct Group {
  int rank, size;
  GridBarrier gb;
  unsigned long long target;
  __device__ Group(const GridBarrier& b) : gb(b), target(0) {
    if constexpr (GRID) {
      rank = blockIdx.x;
      size = gridDim.x;
    } else {
      cg::cluster_group cl = cg::this_cluster();
      rank = (int)cl.block_rank();
      size = (int)cl.num_blocks();
    }
  }
  // all CTAs of the group; false (everywhere) after a grid wait past its limit
  __device__ __forceinline__ bool sync() {
    if constexpr (GRID) return grid_sync(gb, target);
    cg::this_cluster().sync();
    return true;
  }
  // entry i of a shared vector, in every CTA's copy (cluster) or in the L2 copy g (grid)
  __device__ __forceinline__ void put(double* vec, double* g, int i, double v) const {
    if constexpr (GRID) {
      __stcg(g + i, v);
    } else {
      const cg::cluster_group cl = cg::this_cluster();
      for (int r = 0; r < size; ++r) *cl.map_shared_rank(vec + i, r) = v;
    }
  }
  // after a sync: the grid's copy comes into shared memory (the caller syncs the CTA)
  __device__ __forceinline__ void fetch(double* vec, const double* g, int len) const {
    if constexpr (GRID)
      for (int i = threadIdx.x; i < len; i += kThr) vec[i] = __ldcg(g + i);
  }
};

// a b + c d with the second product rounded: where two products meet, which of them a compiler
// fuses would differ between the kernels below, and with it the bits
__device__ __forceinline__ double two_products(double a, double b, double c, double d) {
  return __fma_rn(a, b, __dmul_rn(c, d));
}

// barrier_step_refined from the hardware's estimates (2^-22.9 and one unit in the last place off at
// most): half the dependent operations of the library's root and quotient, and an update's critical
// path holds this chain.
__device__ __forceinline__ void barrier_step_fast(double omega, double c, double& x, double& s) {
  barrier_step_refined(
      omega, c,
      [](float v) {
        float r;
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
        return r;
      },
      [](float v) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
        return r;
      },
      x, s);
}

struct GroupArgs {
  DenseInst* insts;
  int count;
  DenseParams P;
  int* queue;
  const int* order;
  int cache_vec, cache_mat;       // copies in shared memory: the CTA's vectors, its matrix rows
  GroupSparse sp;                 // SPARSE: A by rows and by columns
  // grid mode: published vectors (q, t, z_y: even(m) each; x, s: even(n) each), partial sums, barrier
  double* gvec;
  double* gpart;                  // kSums * grid
  unsigned long long* bar;
  int* err;
  unsigned long long bar_limit_ns;
};

struct Scal {
  double tau, kappa, theta, mu, t1, t2, itau, cmu, gk;
  int action, status, outer, ok;
  int64_t total;
  double a[kSums];   // the sums
};

// the sum of a part's nine cells
__device__ __forceinline__ double part_tree(const double (&v)[kPerPart]) {
  return (((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]))) + v[8];
}

// The CTA's part sums, from its cells' (cs: [sum][cell], `cells` of them), into the slots of every CTA
// of the cluster, [part][sum]; in a grid the CTA's one cell into the L2, [part / 2][cell][sum][part % 2].
template <bool GRID>
__device__ __forceinline__ void publish_sums(const Group<GRID>& G, const double* cs, int cells, double* slots, double* gslots) {
  if constexpr (GRID) {
    const int p = G.rank / kPerPart, i = G.rank % kPerPart, k = threadIdx.x;
    if (k < kSums) __stcg(gslots + ((p >> 1) * kPerPart + i) * 2 * kSums + 2 * k + (p & 1), cs[k]);
  } else {
    const int parts = cells / kPerPart, t = threadIdx.x;
    if (t >= parts * kSums) return;
    const int k = t % kSums, pl = t / kSums;
    double v[kPerPart];
#pragma unroll
    for (int i = 0; i < kPerPart; ++i) v[i] = cs[k * cells + pl * kPerPart + i];
    const double sum = part_tree(v);
    double* at = slots + (G.rank * parts + pl) * kSums + k;
    const cg::cluster_group cl = cg::this_cluster();
    for (int r = 0; r < G.size; ++r) *cl.map_shared_rank(at, r) = sum;
  }
}

// After the barrier: the totals into out (shared), by warp 0, in the same order in every CTA.
template <bool GRID>
__device__ __forceinline__ void total_sums(const double* slots, const double* gslots, int parts, double* out) {
  const int lane = threadIdx.x & 31, k = lane >> 1, h = lane & 1;
  double p[kMaxParts / 2];   // parts h, h + 2, ..., 0 beyond the last
  if constexpr (GRID) {
#pragma unroll
    for (int q0 = 0; q0 < kMaxParts / 2; q0 += 4) {   // 36 loads in flight
      double v[4][kPerPart];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < kPerPart; ++i) v[q][i] = k < kSums ? __ldcg(gslots + ((q0 + q) * kPerPart + i) * 2 * kSums + lane) : 0.0;
#pragma unroll
      for (int q = 0; q < 4; ++q) p[q0 + q] = part_tree(v[q]);
    }
  } else {
#pragma unroll
    for (int q = 0; q < kMaxParts / 2; ++q) p[q] = k < kSums && 2 * q + h < parts ? slots[(2 * q + h) * kSums + k] : 0.0;
  }
  double v = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  if (h == 0 && k < kSums) out[k] = v;
  __syncwarp();
}

__device__ __forceinline__ int even(int k) { return (k + 1) & ~1; }

// rp, ci, va: CSR rows (of the CTA).  out(which, i, sum_j A_ij v_which[j]) for i < rows, eight
// lanes per row (the sums of the rows of a grid flow LP's incidence matrix are 4 to 8 long).
template <typename F>
__device__ __forceinline__ void sparse_rows2(const int32_t* rp, const int32_t* ci, const double* va, int rows,
                                             const double* v0, const double* v1, F out) {
  const int sub = threadIdx.x & 7;
  const int per = kThr / 8, n8 = (rows + per - 1) / per * per;   // whole warps enter the shuffles
  for (int i = threadIdx.x >> 3; i < n8; i += per) {
    double a0 = 0.0, a1 = 0.0;
    if (i < rows)
      for (int e = rp[i] + sub; e < rp[i + 1]; e += 8) {
        const double a = va[e];
        const int j = ci[e];
        a0 += a * v0[j];
        a1 += a * v1[j];
      }
    // the two sums together: lanes 0-3 carry a0, 4-7 a1
    const double send = sub < 4 ? a1 : a0, keep = sub < 4 ? a0 : a1;
    double v = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    if (i < rows && (sub & 3) == 0) out(sub >> 2, i, v);
  }
}
// out(j, sum_i A_ij v[i]) for the CTA's columns, a thread per column, by the warps from W0 on
template <int W0, typename F>
__device__ __forceinline__ void sparse_cols(const int32_t* cp, const int32_t* ri, const double* cv, int cols,
                                            const double* v, F out) {
  if (threadIdx.x < 32 * W0) return;
  for (int j = threadIdx.x - 32 * W0; j < cols; j += kThr - 32 * W0) {
    double a = 0.0;
    for (int e = cp[j]; e < cp[j + 1]; ++e) a += cv[e] * v[ri[e]];
    out(j, a);
  }
}

// Algorithm 2 (with the relaxation of Sec. 4.2) for one instance by the group.
template <bool GRID, bool SPARSE>
__device__ void solve_one(DenseInst& I, const GroupArgs& Q, Group<GRID>& G, double* sm, Scal& S) {
  const DenseParams& P = Q.P;
  const int m = I.m, n = I.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int mp = even(m), np = even(n);
  const int parts = I.parts;
  const int mc = own_room(G.size, parts, GRID, m), nc_ = own_room(G.size, parts, GRID, n);
  const int i0 = own_start(G.rank, G.size, parts, GRID, m), mr = own_start(G.rank + 1, G.size, parts, GRID, m) - i0;   // its rows
  const int j0 = own_start(G.rank, G.size, parts, GRID, n), nr = own_start(G.rank + 1, G.size, parts, GRID, n) - j0;   // columns
  const int most = GRID ? 1 : kPerPart * (parts / min(G.size, parts));   // cells of a CTA that owns any
  const int cells = GRID || G.rank < parts ? most : 0;
  double* q = sm;
  double* tv = q + mp;
  double* zy = tv + mp;
  double* x = zy + mp;
  double* s = x + np;
  double* rslot = s + np;                               // the parts' sums (a grid's lie in the L2)
  double* cs = rslot + (GRID ? 0 : kSums * kMaxParts);  // the cells' sums
  int* ct = reinterpret_cast<int*>(cs + kSums * most);
  int* rt = ct + most + 1;
  double* y = cs + (kSums + 1) * most + 1;              // own rows
  double* Ax = y + mc;
  double* As = Ax + mc;
  double* k1y = As + mc;                                // M^{-T} h1, M^{-T} h2
  double* k2y = k1y + mc;
  double* aty = k2y + mc;                               // own columns
  double* v = aty + nc_;
  double* rx = v + nc_;                                 // factors of the sums; of w = x + s in v, of the
  double* dr = rx + nc_;                                // rows in the idle t and z_y
  double* as = dr + nc_;
  double* k1x = as + nc_;
  double* k2x = k1x + nc_;
  double* top = k2x + nc_;
  double* gq = Q.gvec;
  double* gtv = gq + mp;
  double* gzy = gtv + mp;
  double* gx = gzy + mp;
  double* gs = gx + np;
  double* grs = Q.gpart;
  const double* b = I.b + i0;
  const double* bbar = I.bbar + i0;
  const double* g1y = I.g1 + i0;
  const double* g2y = I.g2 + i0;
  const double* c = I.c + j0;
  const double* cbar = I.cbar + j0;
  const double* g1x = I.g1 + m + j0;
  const double* g2x = I.g2 + m + j0;
  const double* Ar = SPARSE ? nullptr : I.A + (size_t)i0 * I.ld;
  const double* ATr = SPARSE ? nullptr : I.AT + (size_t)j0 * mp;
  const int32_t* rp = SPARSE ? Q.sp.rp + i0 : nullptr;   // entries [rp[i], rp[i + 1]) of ci, va
  const int32_t* cp = SPARSE ? Q.sp.cp + j0 : nullptr;
  const int32_t *ci = Q.sp.ci, *ri = Q.sp.ri;
  const double *va = Q.sp.va, *cv = Q.sp.cv;
  // L^{-1} and L^{-T}: rows rank, rank + size, ...
  const int tr = G.rank < m ? (m - G.rank + G.size - 1) / G.size : 0;
  int64_t tstride = (int64_t)G.size * mp;
  const double* Lr = I.Li + (size_t)min(G.rank, m - 1) * mp;
  const double* Ur = I.LiT + (size_t)min(G.rank, m - 1) * mp;
  if (Q.cache_vec) {
    double* d = top;
    auto copy = [&](const double*& src, int len, int room) {
      for (int i = threadIdx.x; i < len; i += kThr) d[i] = src[i];
      src = d;
      d += room;
    };
    copy(b, mr, mc); copy(bbar, mr, mc); copy(g1y, mr, mc); copy(g2y, mr, mc);
    copy(c, nr, nc_); copy(cbar, nr, nc_); copy(g1x, nr, nc_); copy(g2x, nr, nc_);
    top = sm + even((int)(d - sm));
  }
  if (Q.cache_mat) {
    double* d = top;
    auto copy = [&](const double*& src, int rows, int ld, int64_t stride, int room) {
      for (int e = threadIdx.x; e < rows * ld; e += kThr) d[e] = src[(int64_t)(e / ld) * stride + e % ld];
      src = d;
      d += room * ld;
    };
    if constexpr (!SPARSE) { copy(Ar, mr, np, np, mc); copy(ATr, nr, mp, mp, nc_); }
    copy(Lr, tr, mp, tstride, mc);
    copy(Ur, tr, mp, tstride, mc);
    tstride = mp;
    if constexpr (SPARSE) {
      // the CTA's entries, offsets shifted to the copies
      auto entries = [&](const int32_t*& ptr, const int32_t*& idx, const double*& val, int rows, int room, int prow) {
        const int e0 = ptr[0], len = ptr[rows] - e0;
        int32_t* di = reinterpret_cast<int32_t*>(d + room);
        int32_t* dp = di + room;
        for (int e = threadIdx.x; e < len; e += kThr) { d[e] = val[e0 + e]; di[e] = idx[e0 + e]; }
        for (int r = threadIdx.x; r <= rows; r += kThr) dp[r] = ptr[r] - e0;
        val = d; idx = di; ptr = dp;
        d += room + (room + prow + 1 + 1) / 2;
      };
      entries(rp, ci, va, mr, Q.sp.room_a, mc);
      entries(cp, ri, cv, nr, Q.sp.room_at, nc_);
    }
  }
  const double alpha = P.alpha, eps = P.eps, a1 = 1.0 - alpha;
  const double zbar = I.zbar, xi = -(double)n - 1.0, nb = I.nb, nc = I.nc;
  const double Ki0 = I.Kinv[0], Ki1 = I.Kinv[1], Ki2 = I.Kinv[2], Ki3 = I.Kinv[3];
  // screens of the Sec. 4.1 tests without square roots and divisions; a sum that passes is
  // tested as written
  const double tp = eps * (1.0 + nb) * (1.0 + 1e-12), td = eps * (1.0 + nc) * (1.0 + 1e-12);
  const double tp2 = tp * tp, td2 = td * td, nb2 = nb * nb, nc2 = nc * nc;
  const bool resume = I.resume != 0;
  for (int i = threadIdx.x; i < mp; i += kThr) {
    q[i] = 0.0;
    tv[i] = 0.0;
    zy[i] = 0.0;
  }
  for (int j = n + threadIdx.x; j < np; j += kThr) {   // the padding
    x[j] = 0.0;
    s[j] = 0.0;
  }
  for (int i = threadIdx.x; i < mr; i += kThr) y[i] = resume ? I.y[i0 + i] : 0.0;
  for (int j = threadIdx.x; j < nr; j += kThr) aty[j] = 0.0;
  if (threadIdx.x == 0) {
    S.tau = resume ? I.r_tau : 1.0;
    S.kappa = resume ? I.r_kappa : 1.0;
    S.theta = resume ? I.r_theta : 1.0;
    S.mu = resume ? I.r_mu : P.beta;
    S.total = resume ? I.r_iters : 0;
    S.outer = resume ? I.r_outer : 0;
    S.itau = 1.0 / S.tau;
    S.status = 0;
    S.ok = 1;
  }
  __syncthreads();
  // rows of A times two vectors, and columns of A times one, over the CTA's share
  auto rows_A = [&](const double* v0, const double* v1, auto out) {
    if constexpr (SPARSE) sparse_rows2(rp, ci, va, mr, v0, v1, out);
    else dots_any<2, 0>(Ar, np, mr, v0, v1, out);
  };
  // z_y = L^{-T} L^{-1} q of the published q, published; two barriers.  The first warp has
  // `beside` and `beside2` to do meanwhile.
  auto solve_G = [&](auto beside, auto beside2) -> bool {
    if (wid == 0) beside();
    tri_any<true>(Lr, tstride, tr, G.rank, G.size, mp >> 1, q, [&](int k, double d) { G.put(tv, gtv, G.rank + G.size * k, d); });
    if (!G.sync()) return false;
    if (S.action != ACT_STEP) return true;
    G.fetch(tv, gtv, m);
    if constexpr (GRID) __syncthreads();
    if (wid == 0) beside2();
    tri_any<false>(Ur, tstride, tr, G.rank, G.size, mp >> 1, tv, [&](int k, double d) { G.put(zy, gzy, G.rank + G.size * k, d); });
    if (!G.sync()) return false;
    G.fetch(zy, gzy, m);
    if constexpr (GRID) __syncthreads();
    return true;
  };
  const int rows0 = (nr + 31) & ~31;   // the CTA's rows start at a warp of their own
  const int items = rows0 + mr;
  // where each cell of this CTA begins among its columns (ct) and rows, and after the last its end
  for (int k = threadIdx.x; k <= cells; k += kThr) {
    const int64_t at = GRID ? G.rank + k : kPerPart * (G.rank * (parts / min(G.size, parts))) + k;
    ct[k] = (int)(at * n / (kPerPart * parts)) - j0;
    rt[k] = (int)(at * m / (kPerPart * parts)) - i0;
  }
  const int inv_cells = (1 << 20) / max(cells, 1) + 1;   // t / cells = t inv_cells >> 20 for t < kSums cells <= 1584
  if (!G.sync()) return;   // nobody publishes into a CTA that is still filling its copies
  // M^{-T} h = J M^{-1} J h, J = diag(I, -I): for h = [a; d], G g = a + A d and
  // M^{-T} h = [g; d - A^T g].  The columns d of h1 and h2 stand in x and s meanwhile.
  if (threadIdx.x == 0) S.action = ACT_STEP;
  for (int j = threadIdx.x; j < n; j += kThr) { x[j] = I.c[j]; s[j] = -I.cbar[j]; }
  __syncthreads();
  rows_A(x, s, [&](int w, int i, double d) { (w == 0 ? Ax : As)[i] = d; });
  __syncthreads();
  for (int col = 0; col < 2; ++col) {
    for (int i = threadIdx.x; i < mr; i += kThr) G.put(q, gq, i0 + i, col == 0 ? Ax[i] - b[i] : As[i] + bbar[i]);
    if (!G.sync()) return;
    G.fetch(q, gq, m);
    __syncthreads();
    if (!solve_G([] {}, [] {})) return;
    double* ky = col == 0 ? k1y : k2y;
    double* kx = col == 0 ? k1x : k2x;
    const double* d = col == 0 ? x : s;
    for (int i = threadIdx.x; i < mr; i += kThr) ky[i] = zy[i0 + i];
    auto put_k = [&](int j, double t) { kx[j] = d[j0 + j] - t; };
    if constexpr (SPARSE) sparse_cols<0>(cp, ri, cv, nr, zy, put_k);
    else dots_any<1, 0>(ATr, mp, nr, zy, zy, [&](int, int j, double t) { put_k(j, t); });
    if (!G.sync()) return;   // z_y has been read
  }
  // start of Algorithm 2, or a state loaded by abip_set_state
  for (int j = threadIdx.x; j < n; j += kThr) {
    x[j] = resume ? I.x[j] : 1.0;
    s[j] = resume ? I.s[j] : 1.0;
  }
  if (resume) {   // A^T y of the loaded state, once (z_y's buffer holds y)
    for (int i = threadIdx.x; i < m; i += kThr) zy[i] = I.y[i];
    __syncthreads();
    if constexpr (SPARSE) sparse_cols<0>(cp, ri, cv, nr, zy, [&](int j, double d) { aty[j] = d; });
    else dots_any<1, 0>(ATr, mp, nr, zy, zy, [&](int, int j, double d) { aty[j] = d; });
  }
  bool first = true;   // the sums of a start or of a warm start: no test, no count
  if (!G.sync()) return;
  for (;;) {
    // ---- the sums over the columns, the products A x, A s, the sums over the rows, and q
    {
      const double ta = S.tau, th = S.theta, it = S.itau;
      double *ry = tv, *pr = zy;
      for (int e = threadIdx.x; e < nr; e += kThr) {
        const double at = aty[e], sj = s[j0 + e], cj = c[e];
        const double a = at + sj;
        rx[e] = two_products(cj, ta, -cbar[e], th) - a;
        dr[e] = a * it - cj;
        as[e] = a;
        v[e] = x[j0 + e] + sj;
      }
      rows_A(x, s, [&](int w, int i, double d) { (w == 0 ? Ax : As)[i] = d; });
      __syncthreads();
      for (int i = threadIdx.x; i < mr; i += kThr) {
        const double ax = Ax[i], bi = b[i];
        G.put(q, gq, i0 + i, y[i] - (ax + As[i]));
        ry[i] = ax - bi * ta + bbar[i] * th;
        pr[i] = ax * it - bi;
      }
      __syncthreads();
      for (int t = threadIdx.x; t < kSums * cells; t += kThr) {   // a chain: sum k over a cell's columns, then its rows
        const int k = t * inv_cells >> 20, cell = t - k * cells;
        const double *pc = nullptr, *qc = nullptr, *p = nullptr, *pq = nullptr;
        switch (k) {
          case 0: pc = qc = rx; p = pq = ry; break;
          case 1: p = pq = pr; break;
          case 2: pc = qc = dr; break;
          case 3: p = pq = Ax; break;
          case 4: pc = qc = as; break;
          case 5: p = b; pq = y; break;
          case 6: p = bbar; pq = y; break;
          case 7: pc = c; qc = x + j0; break;
          case 8: pc = cbar; qc = x + j0; break;
          case 9: pc = k1x; qc = v; p = k1y; pq = y; break;
          default: pc = k2x; qc = v; p = k2y; pq = y; break;
        }
        double acc = 0.0;
        if (pc)
          for (int e = ct[cell]; e < ct[cell + 1]; ++e) acc += pc[e] * qc[e];
        if (p)
          for (int i = rt[cell]; i < rt[cell + 1]; ++i) acc += p[i] * pq[i];
        cs[t] = acc;
      }
      __syncthreads();
      publish_sums<GRID>(G, cs, cells, rslot, grs);
    }
    if (!G.sync()) return;
    G.fetch(q, gq, m);
    if constexpr (GRID) __syncthreads();
    // ---- projection: z_y = G^{-1} (y - A (x + s)), beside it the decision on the sums and
    // t = K^{-1} (w_{tau,theta} + H^T z)
    auto decide = [&] {
      total_sums<GRID>(rslot, grs, parts, S.a);
      if (lane != 0) return;
      const double* a = S.a;
      const double tau = S.tau;
      const double rt = a[5] - a[7] + zbar * S.theta - S.kappa;
      const double rth = -a[6] + a[8] - zbar * tau - xi;
      const double inner2 = a[0] + rt * rt + rth * rth;
      int st = 0, action = ACT_STEP;
      if (!isfinite(inner2)) {
        S.ok = 0;
        action = ACT_STOP;
      } else {
        if (!first) {
          S.total += 1;
          if (P.stop_rule == 0) {
            if (a[1] <= tp2 && a[2] <= td2) {
              const double ps = sqrt(a[1]) / (1.0 + nb), ds = sqrt(a[2]) / (1.0 + nc);
              const double gp = fabs(a[7] / tau - a[5] / tau) / (1.0 + fabs(a[7] / tau) + fabs(a[5] / tau));
              if (ps <= eps && ds <= eps && gp <= eps) st = ABIP_OPTIMAL;
            }
            const double pe = eps * a[5], de = eps * a[7];
            if (st == 0 && a[5] > 0 && a[4] * nb2 <= pe * pe * (1.0 + 1e-11) && sqrt(a[4]) <= pe / nb)
              st = ABIP_PRIMAL_INFEASIBLE;
            if (st == 0 && a[7] < 0 && a[3] * nc2 <= de * de * (1.0 + 1e-11) && sqrt(a[3]) <= -de / nc)
              st = ABIP_DUAL_INFEASIBLE;
          }
          if (st == 0 && S.total >= P.max_admm) st = ABIP_MAX_ITER;
        }
        if (st == 0 && inner2 <= S.mu) {
          double rho = 0.0;
          if (P.gamma_max > 0.0)
            rho = fmax(sqrt(a[1]) / (1.0 + nb),
                       fmax(sqrt(a[2]) / (1.0 + nc),
                            fabs(a[7] / tau - a[5] / tau) / (1.0 + fabs(a[7] / tau) + fabs(a[5] / tau))));
          S.gk = adaptive_gamma(P.gamma, P.gamma_max, eps, rho);
          S.mu *= S.gk;
          S.outer += 1;
          action = ACT_WARM;
          if (P.stop_rule == 1 && S.mu < eps) st = ABIP_OPTIMAL;
          else if (S.outer >= kMaxOuter) st = ABIP_MAX_ITER;   // mu has underflowed
        }
        if (st != 0) {
          S.status = st;
          action = ACT_STOP;
        }
      }
      S.action = action;
    };
    auto scalars = [&] {
      if (lane != 0) return;
      const double v1 = S.tau + S.kappa + S.a[9], v2 = S.theta + xi + S.a[10];
      S.t1 = two_products(Ki0, v1, Ki1, v2);
      S.t2 = two_products(Ki2, v1, Ki3, v2);
      S.cmu = S.mu / P.beta;
    };
    if (!solve_G(decide, scalars)) return;
    if (S.action == ACT_STOP) break;
    if (S.action == ACT_WARM) {
      const double gk = S.gk, sg = sqrt(gk);
      for (int j = threadIdx.x; j < n; j += kThr) {   // every CTA its own copies of x and s
        if (P.warmstart == 1) { x[j] *= sg; s[j] *= sg; }
        else if (x[j] >= s[j]) s[j] *= gk;
        else x[j] *= gk;
      }
      for (int i = threadIdx.x; i < mr; i += kThr) y[i] *= sg;
      for (int j = threadIdx.x; j < nr; j += kThr) aty[j] *= sg;
      if (threadIdx.x == 0) {
        if (P.warmstart == 1) { S.tau *= sg; S.kappa *= sg; }
        else if (S.tau >= S.kappa) S.kappa *= gk;
        else S.tau *= gk;
        S.theta *= sg;
        S.itau = 1.0 / S.tau;
      }
      first = true;
      // no CTA publishes q, t or its sums before all have read the last ones
      if (!G.sync()) return;
      continue;
    }
    first = false;
    // ---- A^T z_y, relaxation, barrier and dual steps (Eqs. Simple-Update:*), A^T y by
    // linearity; the step of tau, kappa and theta on the first warp
    const double t1 = S.t1, t2 = S.t2, cmu = S.cmu;
    if (threadIdx.x == 0) {
      const double th = two_products(alpha, t1, a1, S.tau);
      double tn, kn;
      barrier_step_fast(th - S.kappa, cmu, tn, kn);
      S.tau = tn;
      S.kappa = kn;
      S.theta = two_products(alpha, t2, a1, S.theta);
      S.itau = 1.0 / tn;
    }
    if constexpr (SPARSE) sparse_cols<1>(cp, ri, cv, nr, zy, [&](int j, double d) { v[j] = d; });
    else dots_any<1, 1>(ATr, mp, nr, zy, zy, [&](int, int j, double d) { v[j] = d; });
    __syncthreads();
    for (int e = threadIdx.x; e < items; e += kThr) {
      if (e < nr) {
        const int j = j0 + e;
        const double x0 = x[j], s0 = s[j], vj = v[e];
        const double gx1 = g1x[e], gx2 = g2x[e];
        // A^T g1y = g1x - c and A^T g2y = g2x + cbar (M g = h)
        aty[e] = two_products(alpha, vj - (gx1 - c[e]) * t1 - (gx2 + cbar[e]) * t2, a1, aty[e]);
        const double ux = x0 + s0 + vj - gx1 * t1 - gx2 * t2;
        double xn, sn;
        barrier_step_fast(two_products(alpha, ux, a1, x0) - s0, cmu, xn, sn);
        G.put(x, gx, j, xn);
        G.put(s, gs, j, sn);
      } else if (e >= rows0) {
        const int i = e - rows0;
        const double uy = zy[i0 + i] - g1y[i] * t1 - g2y[i] * t2;
        y[i] = two_products(alpha, uy, a1, y[i]);
      }
    }
    if (!G.sync()) return;
    G.fetch(x, gx, n);
    G.fetch(s, gs, n);
    if constexpr (GRID) __syncthreads();
  }
  // outputs: raw state and the scaled candidate or certificate (Sec. 4.1)
  const double bty = S.a[5], ctx = S.a[7], tau = S.tau;
  const int status = S.status;
  double sx = 1.0 / tau, sy = 1.0 / tau;
  if (status == ABIP_PRIMAL_INFEASIBLE) { sx = 1.0; sy = 1.0 / bty; }
  if (status == ABIP_DUAL_INFEASIBLE) { sx = -1.0 / ctx; sy = 1.0; }
  for (int i = threadIdx.x; i < mr; i += kThr) {
    I.y[i0 + i] = y[i];
    if (I.out_y) I.out_y[i0 + i] = y[i] * sy;
  }
  for (int e = threadIdx.x; e < nr; e += kThr) {
    const int j = j0 + e;
    I.x[j] = x[j];
    I.s[j] = s[j];
    if (I.out_x) I.out_x[j] = x[j] * sx;
    if (I.out_s) I.out_s[j] = s[j] * sy;
  }
  // the descriptor is read by every CTA until here
  if (!G.sync()) return;
  if (G.rank == 0 && threadIdx.x == 0) {
    const double* a = S.a;
    I.tau = tau; I.kappa = S.kappa; I.theta = S.theta; I.mu = S.mu;
    I.resume = 0;
    I.pres = sqrt(a[1]) / (1.0 + nb);
    I.dres = sqrt(a[2]) / (1.0 + nc);
    I.dgap = fabs(ctx / tau - bty / tau) / (1.0 + fabs(ctx / tau) + fabs(bty / tau));
    I.ctx = ctx; I.bty = bty; I.obj = ctx / tau;
    I.admm_iters = S.total; I.outer_iters = S.outer; I.status = status;
    I.beta_last = P.beta;
    if (!S.ok) I.err = DEV_ERR_NONFINITE;
  }
}

template <int MINB, bool SPARSE>
__global__ void __launch_bounds__(kThr, MINB) dense_cluster_kernel(GroupArgs Q) {
  extern __shared__ __align__(16) double sm[];
  __shared__ Scal S;
  __shared__ int s_id;
  cg::cluster_group cl = cg::this_cluster();
  Group<false> G(GridBarrier{});
  cl.sync();   // no CTA writes to a peer (s_id below) that may not have started
  for (;;) {
    if (G.rank == 0 && threadIdx.x == 0) {
      const int k = atomicAdd(Q.queue, 1);
      const int id = k < Q.count ? (Q.order ? Q.order[k] : k) : -1;
      for (int r = 0; r < G.size; ++r) *cl.map_shared_rank(&s_id, r) = id;
    }
    cl.sync();
    const int id = s_id;
    if (id < 0) return;   // the same in every CTA, after which none writes to another
    DenseInst& I = Q.insts[id];
    if (I.err == 0) solve_one<false, SPARSE>(I, Q, G, sm, S);
    cl.sync();            // every CTA has read s_id and its copies
  }
}

template <bool SPARSE>
__global__ void __launch_bounds__(kThr, 1) dense_grid_kernel(GroupArgs Q) {
  extern __shared__ __align__(16) double sm[];
  __shared__ Scal S;
  Group<true> G(GridBarrier{Q.bar, Q.err, Q.bar_limit_ns});
  if (Q.insts[0].err == 0) solve_one<true, SPARSE>(Q.insts[0], Q, G, sm, S);
}

using ClusterFn = void (*)(GroupArgs);
ClusterFn cluster_fn(int variant, bool sparse) {
  if (sparse) return dense_cluster_kernel<1, true>;
  // a batch plans two CTAs per SM, so that is the default (one LP takes variant 1: 6 % faster)
  return variant == 2 ? dense_cluster_kernel<3, false> : variant == 1 ? dense_cluster_kernel<1, false>
                                                                      : dense_cluster_kernel<2, false>;
}
ClusterFn grid_fn(bool sparse) { return sparse ? dense_grid_kernel<true> : dense_grid_kernel<false>; }

struct SmemPlan {
  size_t bytes;
  int cache_vec, cache_mat;
};

size_t base_doubles(int m, int n, int C, int parts, bool grid) {
  const size_t mp = (m + 1) / 2 * 2, np = (n + 1) / 2 * 2, mc = own_room(C, parts, grid, m), nc = own_room(C, parts, grid, n);
  const size_t cells = grid ? 1 : kPerPart * (parts / std::min(C, parts));
  const size_t sums = (grid ? 0 : kSums * kMaxParts) + (kSums + 1) * cells + 1;
  return 3 * mp + 2 * np + sums + 5 * mc + 7 * nc;
}
size_t vec_doubles(size_t mc, size_t nc) { return 4 * mc + 4 * nc + 2; }
size_t mat_doubles(int m, int n, size_t mc, size_t nc) {
  const size_t mp = (m + 1) / 2 * 2, np = (n + 1) / 2 * 2;
  return mc * (np + 2 * mp) + nc * mp + 2;
}

size_t sparse_doubles(int m, size_t mc, size_t nc, int room_a, int room_at) {
  const size_t mp = (m + 1) / 2 * 2;
  return 2 * mc * mp + 2 + room_a + (room_a + mc + 2) / 2 + room_at + (room_at + nc + 2) / 2;
}

// the shared memory of a launch for the given sizes: the copies that fit the budget
SmemPlan plan_smem(const int* m, const int* n, int count, int C, bool grid, size_t budget,
                   const GroupSparse* sp = nullptr, int sp_parts = 0) {
  size_t base = 0, vec = 0, mat = 0;
  for (int k = 0; k < count; ++k) {
    const int parts = sp ? sp_parts : dense_parts(m[k], n[k]);
    const size_t mc = own_room(C, parts, grid, m[k]), nc = own_room(C, parts, grid, n[k]);
    const size_t b = base_doubles(m[k], n[k], C, parts, grid), v = b + vec_doubles(mc, nc);
    base = std::max(base, b);
    vec = std::max(vec, v);
    mat = std::max(mat, v + (sp ? sparse_doubles(m[k], mc, nc, sp->room_a, sp->room_at) : mat_doubles(m[k], n[k], mc, nc)));
  }
  SmemPlan p{base * 8 + 16, 0, 0};
  if (vec * 8 <= budget) { p.bytes = vec * 8 + 16; p.cache_vec = 1; }
  if (p.cache_vec && mat * 8 <= budget) { p.bytes = mat * 8 + 16; p.cache_mat = 1; }
  return p;
}

constexpr size_t kSmemMax = 224 * 1024;

cudaError_t cluster_config(ClusterFn f, int C, size_t smem, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at) {
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  // one split of the SM's memory for every launch, so that buckets of different shared memory
  // run side by side on an SM (a mixed batch of 128 LPs, 200 updates: 17.9 -> 11.7 ms)
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cfg.blockDim = dim3(kThr);
  cfg.gridDim = dim3((unsigned)C);
  cfg.dynamicSmemBytes = smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return e;
}

}  // namespace

int plan_dense_grid(int m, int n, int sms, DenseGroupPlan& plan) {
  if (sms < kGridCtas) return 0;
  const SmemPlan s = plan_smem(&m, &n, 1, kGridCtas, true, kSmemMax - 16);
  plan = DenseGroupPlan{kGridCtas, 1, s.cache_vec, s.cache_mat, s.bytes, 0};
  return s.bytes <= kSmemMax;
}

namespace {
// A cluster plan from C CTAs: more, up to 8, where `at` (the plan of a size) does not fit the shared
// memory, then fewer where the device holds no cluster of that size.  16 CTAs need an SM each of one
// GPC, which a partitioned device may not have.
template <typename F>
int settle_cluster(int C, ClusterFn f, DenseGroupPlan& plan, F at) {
  for (; plan = at(C), plan.smem > kSmemMax; C *= 2)
    if (C >= 8) return 0;
  for (; C >= 1; C /= 2) {
    plan = at(C);
    if (plan.smem > kSmemMax) return 0;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    int n = 0;
    if (cluster_config(f, C, plan.smem, cfg, attr) == cudaSuccess && cudaOccupancyMaxActiveClusters(&n, f, &cfg) == cudaSuccess && n > 0)
      return 1;
    cudaGetLastError();
  }
  return 0;
}
}  // namespace

int plan_dense_cluster(const int* m, const int* n, int count, int C, size_t budget, DenseGroupPlan& plan) {
  return settle_cluster(C, cluster_fn(count == 1 ? 1 : 0, false), plan, [&](int c) {
    const SmemPlan s = plan_smem(m, n, count, c, false, budget);
    return DenseGroupPlan{c, 0, s.cache_vec, s.cache_mat, s.bytes, 0};
  });
}

namespace {
// most entries a CTA's rows hold: ptr (len + 1), C CTAs
int share_room(const int32_t* ptr, int len, int C, int parts, bool grid) {
  int most = 0;
  for (int r = 0; r < C; ++r)
    most = std::max(most, ptr[own_start(r + 1, C, parts, grid, len)] - ptr[own_start(r, C, parts, grid, len)]);
  return most;
}
}  // namespace

int dense_parts(int m, int n) { return cluster_ctas(dense_work(m, n), kClusterWork); }

int plan_sparse_group(int m, int n, const int32_t* rp, const int32_t* cp, int sms, GroupSparse& sp, DenseGroupPlan& plan,
                      int& parts) {
  if (m > kDirectMaxRows) return 0;
  const double w = 3.0 * rp[m] + (double)m * m + 80.0 * (m + n);
  parts = cluster_ctas(w, kClusterWork);
  const bool grid = w > kGridWork && sms >= kGridCtas;   // as for a dense LP
  auto at = [&](int C) {
    sp.room_a = share_room(rp, m, C, parts, grid);
    sp.room_at = share_room(cp, n, C, parts, grid);
    const SmemPlan s = plan_smem(&m, &n, 1, C, grid, kSmemMax - 16, &sp, parts);
    return DenseGroupPlan{C, grid, s.cache_vec, s.cache_mat, s.bytes, 1};
  };
  if (!grid) return settle_cluster(parts, cluster_fn(1, true), plan, at);
  plan = at(kGridCtas);
  return plan.smem <= kSmemMax;
}

size_t dense_group_scratch(int m, int n) {
  const size_t mp = (m + 1) / 2 * 2, np = (n + 1) / 2 * 2;
  return 3 * mp + 2 * np + (size_t)kSums * kGridCtas + 4;
}

cudaError_t launch_dense_group(DenseInst* inst, int count, const DenseParams& prm, int* queue, const int* order,
                               const DenseGroupPlan& plan, const GroupSparse& sp, int variant, double* scratch,
                               size_t scratch_len, unsigned long long limit_ns, cudaStream_t st) {
  GroupArgs Q{inst, count, prm, queue, order, plan.cache_vec, plan.cache_mat, sp, nullptr, nullptr, nullptr, nullptr, limit_ns};
  if (plan.grid_mode) {
    // barrier counter and error word at the end of the scratch, zeroed by the caller
    Q.bar = reinterpret_cast<unsigned long long*>(scratch + scratch_len - 2);
    Q.err = reinterpret_cast<int*>(scratch + scratch_len - 1);
    Q.gpart = scratch;
    Q.gvec = scratch + (size_t)kSums * kGridCtas;   // even
    const ClusterFn f = grid_fn(plan.sparse != 0);
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
    void* args[] = {&Q};
    return cudaLaunchCooperativeKernel((const void*)f, dim3(plan.ctas), dim3(kThr), args, plan.smem, st);
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  ClusterFn f = cluster_fn(count == 1 ? 1 : variant, plan.sparse != 0);
  cudaError_t e = cluster_config(f, plan.ctas, plan.smem, cfg, at);
  if (e != cudaSuccess) return e;
  int ncl = 0;
  e = cudaOccupancyMaxActiveClusters(&ncl, f, &cfg);
  if (e != cudaSuccess) return e;
  if (ncl < 1) return cudaErrorInvalidConfiguration;
  cfg.gridDim = dim3((unsigned)(std::min(count, ncl) * plan.ctas));
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, f, Q);
}

int dense_group_ctas_per_sm(const DenseGroupPlan& plan, int variant) {
  int per = 0;
  if (plan.grid_mode) {
    cudaFuncSetAttribute(grid_fn(false), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, grid_fn(false), kThr, plan.smem);
    return per;
  }
  ClusterFn f = cluster_fn(variant, false);
  cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, f, kThr, plan.smem);
  return per;
}

}  // namespace abip
