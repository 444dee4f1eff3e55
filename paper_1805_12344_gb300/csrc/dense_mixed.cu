// Dense ABIP in mixed precision (FP64 state, FP32 products of changes; the scheme stands in
// dense_solver.cu) with a thread-block cluster of C = 1 .. 16 CTAs per LP.
//
// What bounds one LP on one CTA: the FP64 pipe of its SM (2 operations per clock: about 90 per
// column and update for the steps and sums) and the stream of 16 m n + 4 m^2 bytes of FP32
// matrices from L2 per update.  A cluster divides both.
//
// Every number is formed by the operations of the one-CTA form in its order: a row's FP32
// product by one warp, and each of the test sums by 256 chains, chain t over the elements t, t +
// 256, ... (one thread each there), joined by the same butterflies.  CTA r of C therefore owns
// the elements (rows and columns) with index mod 256 in [256 r / C, 256 (r + 1) / C), and with
// them whole chains.  The results are the same bits for every C: a last-bit difference would
// change the FP32 rounding of later changes, and those differences grow to 1e-6 of the result.
//
// Measured: one L1-SVM 512 x 1154 203 -> 24 us per update (16 CTAs; 2.6 us of it the exact
// recomputation every 100 updates, whose triangular solves stay serial); 200 updates of 8 / 64 /
// 200 LPs of m 16 .. 256 24.2 -> 4.6, 25.2 -> 6.9, 34.3 -> 19.5 ms.
// Barriers of the cluster per update: G^{-1} dq | H^T z | changes of the state | test sums and
// the next dq.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "abip_device.cuh"
#include "abip_internal.h"
#include "dense_device.cuh"

namespace cg = cooperative_groups;

namespace abip {
namespace {

using dense::kWarps;
using dense::sum_together;
using dense::trsv_lower;
using dense::trsv_lower_t;
constexpr int kThr = dense::kThreads;
constexpr int kRefresh = 100;   // updates between exact FP64 recomputations of the products
constexpr int kHz = 9;          // slots of the two sums of H^T z, after the nine of the tests

// The elements of a CTA: local e <-> index 256 (e / V) + r V + e % V, V = 256 / C.
struct Own {
  int V, base;
  __device__ __forceinline__ int at(int e) const { return 256 * (e / V) + base + e % V; }
  __host__ __device__ static int count(int len, int V, int base) {
    const int rem = len % 256 - base;
    return len / 256 * V + (rem < 0 ? 0 : rem < V ? rem : V);
  }
};

// o0[e] += (row own.at(e) of M) . v0 (and o1 with v1) for e < rows: a warp per row, four rows in
// flight, float4 loads, FP32 accumulation.  M rows start at M + stride * row, nq float4 long.
// f(e, sum) runs on the lane that holds the first sum.
template <bool TWO, typename F>
__device__ __forceinline__ void rows_f32(const float* M, int64_t stride, int nq, int rows, bool packed, const Own& own,
                                         const float* v0, const float* v1, double* o0, double* o1, F f) {
  constexpr int R = 4, P = TWO ? 8 : 4, kShift = TWO ? 2 : 3;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const float4* p0 = reinterpret_cast<const float4*>(v0);
  const float4* p1 = reinterpret_cast<const float4*>(v1);
  for (int g = wid * R; g < rows; g += kWarps * R) {
    float a[P];
    const float4* r[R];
#pragma unroll
    for (int q = 0; q < P; ++q) a[q] = 0.f;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int e = min(g + q, rows - 1);
      r[q] = reinterpret_cast<const float4*>(M + (size_t)(packed ? e : own.at(e)) * stride);
    }
#pragma unroll 2
    for (int t = lane; t < nq; t += 32) {
      const float4 x = p0[t];
      float4 z = x;
      if (TWO) z = p1[t];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const float4 w = r[q][t];
        a[q] += w.x * x.x + w.y * x.y + w.z * x.z + w.w * x.w;
        if (TWO) a[R + q] += w.x * z.x + w.y * z.y + w.z * z.z + w.w * z.w;
      }
    }
    const float s = sum_together<P>(a, lane);
    if ((lane & ((1 << kShift) - 1)) == 0) {
      const int k = lane >> kShift, e = g + k % R;
      if (e < rows) {
        if (k < R) {
          o0[e] += (double)s;
          f(e, s);
        } else {
          o1[e] += (double)s;
        }
      }
    }
  }
}

struct MixArgs {
  DenseInst* insts;
  int count;
  DenseParams P;
  int* queue;
  const int* order;
  int cache_at;   // the CTA's rows of A^T in shared memory
};

enum Act : int { ACT_STEP = 0, ACT_WARM = 1, ACT_STOP = 2, ACT_CONFIRM = 3 };

// The scalars of the iteration, the same in every CTA of the cluster: one thread forms them (a
// warp-wide FP64 operation costs 16 clocks, so 256 threads each forming them would show).
struct MixScal {
  double tau, kappa, theta, mu, itau, cmu, t1, t2, gk, inner2;
  double a[9];                     // the test sums
  int64_t total, next_confirm;
  int action, status, outer, ok;
};

// doubles of shared memory of a CTA but for the A^T copy, floats counted as halves
__host__ __device__ inline size_t mix_doubles(int m, int n, int C) {
  const size_t mp = (m + 3) / 4 * 4, np = (n + 3) / 4 * 4;
  const size_t mc = Own::count(m, 256 / C, 0), nc = Own::count(n, 256 / C, 0);
  return (3 * mp + 2 * np) / 2 + 2 * (size_t)m + 11 * mc + 11 * nc + 11 * 256 + 2;
}

__device__ void delta_group(DenseInst& I, const MixArgs& Q, unsigned char* smraw, double* wsum, double* hz, MixScal& S) {
  const DenseParams& P = Q.P;
  const cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int m = I.m, n = I.n, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t ld = I.ld;
  const int mp = I.ldtf, np = I.ldf;
  Own own;
  own.V = 256 / C;
  own.base = rank * own.V;
  const int V = own.V;
  const int mr = Own::count(m, V, own.base), nr = Own::count(n, V, own.base);
  const int mc = Own::count(m, V, 0), nc_ = Own::count(n, V, 0);   // rank 0 owns the most
  float* dq = reinterpret_cast<float*>(smraw);
  float* dz = dq + mp;
  float* dy = dz + mp;
  float* dx = dy + mp;
  float* ds = dx + np;
  double* full = reinterpret_cast<double*>(ds + np);   // 2 m: y and z_y of a refresh
  double* y = full + 2 * m;                            // own rows
  double* Ax = y + mc;
  double* As = Ax + mc;
  double* zy = As + mc;
  double* qp = zy + mc;
  double* ry = qp + mc;
  double* pr = ry + mc;
  double* b = pr + mc;
  double* bbar = b + mc;
  double* g1y = bbar + mc;
  double* g2y = g1y + mc;
  double* x = g2y + mc;                                // own columns
  double* s = x + nc_;
  double* ATy = s + nc_;
  double* ATz = ATy + nc_;
  double* rx = ATz + nc_;                              // also z_x
  double* dr = rx + nc_;
  double* as = dr + nc_;
  double* c = as + nc_;
  double* cbar = c + nc_;
  double* g1x = cbar + nc_;
  double* g2x = g1x + nc_;
  double* slots = g2x + nc_;                           // 11 x 256: the chains' sums
  const float* AT = I.ATf;
  bool at_packed = false;
  if (Q.cache_at) {
    float* d = reinterpret_cast<float*>((reinterpret_cast<size_t>(slots + 11 * 256) + 15) & ~(size_t)15);
    for (int e = threadIdx.x; e < nr * mp; e += kThr) d[e] = I.ATf[(size_t)own.at(e / mp) * mp + e % mp];
    AT = d;
    at_packed = true;
  }
  const double alpha = P.alpha, beta = P.beta, gamma = P.gamma, eps = P.eps;
  const double zbar = I.zbar, xi = -(double)n - 1.0, nb = I.nb, nc = I.nc;
  const double Ki0 = I.Kinv[0], Ki1 = I.Kinv[1], Ki2 = I.Kinv[2], Ki3 = I.Kinv[3];
  const bool resume = I.resume != 0;
  if (threadIdx.x == 0) {
    S.tau = resume ? I.r_tau : 1.0;
    S.kappa = resume ? I.r_kappa : 1.0;
    S.theta = resume ? I.r_theta : 1.0;
    S.mu = resume ? I.r_mu : beta;
    S.itau = 1.0 / S.tau;
    S.total = resume ? I.r_iters : 0;
    S.outer = resume ? I.r_outer : 0;
    S.next_confirm = 0;
    S.status = 0;
    S.ok = 1;
  }
  for (int e = threadIdx.x; e < mr; e += kThr) {
    const int i = own.at(e);
    y[e] = resume ? I.y[i] : 0.0;
    b[e] = I.b[i]; bbar[e] = I.bbar[i]; g1y[e] = I.g1[i]; g2y[e] = I.g2[i];
  }
  for (int e = threadIdx.x; e < nr; e += kThr) {
    const int j = own.at(e);
    x[e] = resume ? I.x[j] : 1.0;
    s[e] = resume ? I.s[j] : 1.0;
    c[e] = I.c[j]; cbar[e] = I.cbar[j]; g1x[e] = I.g1[m + j]; g2x[e] = I.g2[m + j];
  }
  // the padding of the FP32 vectors meets zero padding of the FP32 matrices
  for (int i = threadIdx.x; i < 3 * mp + 2 * np; i += kThr) dq[i] = 0.f;
  cl.sync();
  int since_refresh = 0;

  // element i of a vector of changes, in every CTA's copy
  auto put = [&](float* vec, int i, float v) {
    for (int r = 0; r < C; ++r) *cl.map_shared_rank(vec + i, r) = v;
  };
  auto put_slot = [&](int k, int u, double v) {
    double* at = slots + k * 256 + own.base + u;
    for (int r = 0; r < C; ++r) *cl.map_shared_rank(at, r) = v;
  };
  // the block sums of NS slots from k0 on, as block_allsum forms them, by warp 0 into out; then
  // f() on thread 0, after which every thread may read what it wrote
  auto totals = [&](auto ns, int k0, double* out, auto f) {
    constexpr int NS = decltype(ns)::value, PP = NS > 2 ? 16 : 2, kShift = NS > 2 ? 1 : 4;
    double v[PP];
#pragma unroll
    for (int k = 0; k < PP; ++k) v[k] = k < NS ? slots[(k0 + k) * 256 + threadIdx.x] : 0.0;
    const double t = sum_together<PP>(v, lane);
    const int k = lane >> kShift;
    if ((lane & ((1 << kShift) - 1)) == 0 && k < NS) wsum[k * kWarps + wid] = t;
    __syncthreads();
    if (wid == 0) {
      if (lane < NS) {   // the butterfly over the eight warps
        const double* w = wsum + lane * kWarps;
        out[lane] = ((w[0] + w[4]) + (w[2] + w[6])) + ((w[1] + w[5]) + (w[3] + w[7]));
      }
      __syncwarp();
      if (lane == 0) f();
    }
    __syncthreads();
  };

  // exact FP64 products of the current state.  The vectors go through the instance's arrays in
  // L2 (x, s, y; out_y carries q and then z_y); the triangular solves run on the first CTA.
  auto refresh = [&]() {
    for (int e = threadIdx.x; e < nr; e += kThr) { const int j = own.at(e); __stcg(I.x + j, x[e]); __stcg(I.s + j, s[e]); }
    for (int e = threadIdx.x; e < mr; e += kThr) __stcg(I.y + own.at(e), y[e]);
    cl.sync();
    for (int e = wid; e < mr; e += kWarps) {
      const double* row = I.A + (size_t)own.at(e) * ld;
      double a0 = 0.0, a1 = 0.0;
      for (int j = lane; j < n; j += 32) {
        const double a = row[j];
        a0 += a * __ldcg(I.x + j);
        a1 += a * __ldcg(I.s + j);
      }
      a0 = warp_sum(a0);
      a1 = warp_sum(a1);
      if (lane == 0) { Ax[e] = a0; As[e] = a1; }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < mr; e += kThr) {
      const double q = y[e] - (Ax[e] + As[e]);
      qp[e] = q;
      __stcg(I.out_y + own.at(e), q);
    }
    cl.sync();
    if (rank == 0) {
      for (int i = threadIdx.x; i < m; i += kThr) full[m + i] = __ldcg(I.out_y + i);
      __syncthreads();
      trsv_lower<double>(I.L, m, full + m);
      trsv_lower_t<double>(I.L, m, full + m);
      for (int i = threadIdx.x; i < m; i += kThr) __stcg(I.out_y + i, full[m + i]);
    }
    cl.sync();
    for (int i = threadIdx.x; i < m; i += kThr) { full[i] = __ldcg(I.y + i); full[m + i] = __ldcg(I.out_y + i); }
    __syncthreads();
    for (int e = threadIdx.x; e < mr; e += kThr) zy[e] = full[m + own.at(e)];
    for (int e = threadIdx.x; e < nr; e += kThr) {
      const double* col = I.A + own.at(e);
      double a0 = 0.0, a1 = 0.0;
#pragma unroll 4
      for (int i = 0; i < m; ++i) {
        const double aij = col[(size_t)i * ld];
        a0 += aij * full[i];
        a1 += aij * full[m + i];
      }
      ATy[e] = a0;
      ATz[e] = a1;
    }
    __syncthreads();
    since_refresh = 0;
  };
  // The Sec. 4.1 tests on the sums; 0 = none passes.
  auto tests = [&](double margin) -> int {
    const double* a = S.a;
    const double tau = S.tau;
    const double ps = sqrt(a[1]) / (1.0 + nb), dsn = sqrt(a[2]) / (1.0 + nc);
    const double gp = fabs(a[7] / tau - a[5] / tau) / (1.0 + fabs(a[7] / tau) + fabs(a[5] / tau));
    if (ps <= margin * eps && dsn <= margin * eps && gp <= margin * eps) return ABIP_OPTIMAL;
    if (a[5] > 0 && sqrt(a[4]) <= margin * eps * a[5] / nb) return ABIP_PRIMAL_INFEASIBLE;
    if (a[7] < 0 && sqrt(a[3]) <= margin * eps * (-a[7]) / nc) return ABIP_DUAL_INFEASIBLE;
    return 0;
  };
  // the test with margin 4 as products first, so that an update pays no root and no quotient;
  // sums near a bound are tested as written
  auto screen = [&]() -> bool {
    const double* a = S.a;
    const double m4 = 4.0 * eps * (1.0 + 1e-11), tp = m4 * (1.0 + nb), td = m4 * (1.0 + nc);
    const double pe = m4 * a[5], de = m4 * a[7];
    return ((a[1] <= tp * tp && a[2] <= td * td) || (a[5] > 0 && a[4] * (nb * nb) <= pe * pe) ||
            (a[7] < 0 && a[3] * (nc * nc) <= de * de)) &&
           tests(4.0) != 0;
  };
  // what happens next, from the sums: `counted` after an update, `exact` on recomputed products
  auto decide = [&](bool counted, bool exact) {
    const double* a = S.a;
    const double rt = a[5] - a[7] + zbar * S.theta - S.kappa;
    const double rth = -a[6] + a[8] - zbar * S.tau - xi;
    S.inner2 = a[0] + rt * rt + rth * rth;
    S.action = ACT_STOP;
    if (!isfinite(S.inner2)) { S.ok = 0; return; }
    if (counted) {
      if (!exact) S.total += 1;
      if (P.stop_rule == 0) {
        if (exact) {
          S.status = tests(1.0);
          S.next_confirm = S.total + P.check_every;
        } else if (S.total >= S.next_confirm && screen()) {
          S.action = ACT_CONFIRM;
          return;
        }
      }
      if (S.status == 0 && S.total >= P.max_admm) S.status = ABIP_MAX_ITER;
      if (S.status != 0) return;
    }
    S.action = ACT_STEP;
    if (S.inner2 <= S.mu) {
      double rho = 0.0;
      if (P.gamma_max > 0.0)
        rho = fmax(sqrt(a[1]) / (1.0 + nb),
                   fmax(sqrt(a[2]) / (1.0 + nc),
                        fabs(a[7] / S.tau - a[5] / S.tau) / (1.0 + fabs(a[7] / S.tau) + fabs(a[5] / S.tau))));
      S.gk = adaptive_gamma(gamma, P.gamma_max, eps, rho);
      S.mu *= S.gk;
      S.outer += 1;
      S.action = ACT_WARM;
      if (P.stop_rule == 1 && S.mu < eps) S.status = ABIP_OPTIMAL;
      else if (S.outer >= kMaxOuter) S.status = ABIP_MAX_ITER;
      if (S.status != 0) S.action = ACT_STOP;
    }
  };
  // the nine sums of the tests from the maintained products, the change of q, and the decision
  auto evaluate = [&](bool counted, bool exact) {
    const double tau = S.tau, theta = S.theta, itau = S.itau;
    for (int e = threadIdx.x; e < mr; e += kThr) {
      const double ax = Ax[e], bi = b[e], bb = bbar[e];
      ry[e] = ax - bi * tau + bb * theta;
      pr[e] = ax * itau - bi;
      const double q = y[e] - (ax + As[e]);
      put(dq, own.at(e), (float)(q - qp[e]));
    }
    for (int e = threadIdx.x; e < nr; e += kThr) {
      const double aty = ATy[e], sj = s[e], cj = c[e], cb = cbar[e];
      rx[e] = -aty + cj * tau - cb * theta - sj;
      dr[e] = (aty + sj) * itau - cj;
      as[e] = aty + sj;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < 9 * V; t += kThr) {   // chain u of sum k: its rows, then its columns
      const int k = t / V, u = t % V;
      const double *p = nullptr, *q = nullptr, *pc = nullptr, *qc = nullptr;
      switch (k) {
        case 0: p = q = ry; pc = qc = rx; break;
        case 1: p = q = pr; break;
        case 2: pc = qc = dr; break;
        case 3: p = q = Ax; break;
        case 4: pc = qc = as; break;
        case 5: p = b; q = y; break;
        case 6: p = bbar; q = y; break;
        case 7: pc = c; qc = x; break;
        default: pc = cbar; qc = x; break;
      }
      double acc = 0.0;
      if (p)
        for (int e = u; e < mr; e += V) acc += p[e] * q[e];
      if (pc)
        for (int e = u; e < nr; e += V) acc += pc[e] * qc[e];
      put_slot(k, u, acc);
    }
    cl.sync();
    totals(std::integral_constant<int, 9>{}, 0, S.a, [&] { decide(counted, exact); });
  };
  auto nothing = [](int, float) {};
  // maintained products after a change (dy, dx, ds) of the iterate
  auto maintain = [&]() {
    rows_f32<true>(I.Af, np, np / 4, mr, false, own, dx, ds, Ax, As, nothing);
    rows_f32<false>(AT, mp, mp / 4, nr, at_packed, own, dy, dy, ATy, ATy, nothing);
    __syncthreads();
  };

  refresh();
  evaluate(false, false);
  while (S.action != ACT_STOP) {
    if (S.action == ACT_CONFIRM) {
      refresh();
      evaluate(true, true);
      continue;
    }
    if (S.action == ACT_WARM) {
      const double gk = S.gk, sg = sqrt(gk);
      for (int e = threadIdx.x; e < nr; e += kThr) {
        const double x0 = x[e], s0 = s[e];
        if (P.warmstart == 1) { x[e] = x0 * sg; s[e] = s0 * sg; }
        else if (x0 >= s0) s[e] = s0 * gk;
        else x[e] = x0 * gk;
        const int j = own.at(e);
        put(dx, j, (float)(x[e] - x0));
        put(ds, j, (float)(s[e] - s0));
      }
      for (int e = threadIdx.x; e < mr; e += kThr) {
        const double y0 = y[e];
        y[e] = y0 * sg;
        put(dy, own.at(e), (float)(y[e] - y0));
      }
      if (threadIdx.x == 0) {
        if (P.warmstart == 1) { S.tau *= sg; S.kappa *= sg; }
        else if (S.tau >= S.kappa) S.kappa *= gk;
        else S.tau *= gk;
        S.theta *= sg;
        S.itau = 1.0 / S.tau;
      }
      cl.sync();
      maintain();
      evaluate(false, false);
      continue;
    }
    // projection on the change of q = y - A(x + s), which the sums published:
    // zy += G^{-1} dq (dz the FP32 change), A^T zy += A^T dz
    for (int e = threadIdx.x; e < mr; e += kThr) qp[e] = y[e] - (Ax[e] + As[e]);
    rows_f32<false>(I.Ginvf, mp, mp / 4, mr, false, own, dq, dq, zy, zy, [&](int e, float v) { put(dz, own.at(e), v); });
    cl.sync();
    rows_f32<false>(AT, mp, mp / 4, nr, at_packed, own, dz, dz, ATz, ATz, nothing);
    __syncthreads();
    for (int e = threadIdx.x; e < nr; e += kThr) rx[e] = x[e] + s[e] + ATz[e];
    __syncthreads();
    for (int t = threadIdx.x; t < 2 * V; t += kThr) {
      const int k = t / V, u = t % V;
      double acc = 0.0;
      if (k == 0) {
        for (int e = u; e < nr; e += V) acc += c[e] * rx[e];
        for (int e = u; e < mr; e += V) acc -= b[e] * zy[e];
      } else {
        for (int e = u; e < nr; e += V) acc -= cbar[e] * rx[e];
        for (int e = u; e < mr; e += V) acc += bbar[e] * zy[e];
      }
      put_slot(kHz + k, u, acc);
    }
    cl.sync();
    totals(std::integral_constant<int, 2>{}, kHz, hz, [&] {
      const double v1 = S.tau + S.kappa + hz[0], v2 = S.theta + xi + hz[1];
      S.t1 = Ki0 * v1 + Ki1 * v2;
      S.t2 = Ki2 * v1 + Ki3 * v2;
      S.cmu = S.mu / beta;
    });
    const double t1 = S.t1, t2 = S.t2, cmu = S.cmu;
    for (int e = threadIdx.x; e < mr; e += kThr) {
      const double uy = zy[e] - g1y[e] * t1 - g2y[e] * t2;
      const double y0 = y[e];
      y[e] = alpha * uy + (1.0 - alpha) * y0;
      put(dy, own.at(e), (float)(y[e] - y0));
    }
    for (int e = threadIdx.x; e < nr; e += kThr) {
      const double ux = rx[e] - g1x[e] * t1 - g2x[e] * t2;
      const double x0 = x[e], s0 = s[e];
      const double xh = alpha * ux + (1.0 - alpha) * x0;
      double xn, sn;
      barrier_step_newton(xh - s0, cmu, xn, sn);   // few FP64 operations (the FP64 pipe binds here)
      x[e] = xn;
      s[e] = sn;
      const int j = own.at(e);
      put(dx, j, (float)(xn - x0));
      put(ds, j, (float)(sn - s0));
    }
    if (threadIdx.x == kThr - 1) {
      // the multiply-adds as the one-CTA form's compiler contracted them (kept bit for bit)
      const double a1 = 1.0 - alpha;
      const double omega = __fma_rn(a1, S.tau, __dmul_rn(alpha, t1)) - S.kappa;
      const double c4 = S.mu / beta;
      const double D = sqrt(__fma_rn(4.0, c4, __dmul_rn(omega, omega)));
      const double tn = omega >= 0.0 ? 0.5 * (omega + D) : (2.0 * c4) / (D - omega);
      const double kn = omega >= 0.0 ? (2.0 * c4) / (omega + D) : 0.5 * (D - omega);
      S.tau = tn;
      S.kappa = kn;
      S.theta = __fma_rn(a1, S.theta, __dmul_rn(alpha, t2));
      S.itau = 1.0 / tn;
    }
    cl.sync();
    maintain();
    if (++since_refresh >= kRefresh) refresh();
    evaluate(true, false);
  }
  // outputs: raw state and the scaled candidate or certificate (Sec. 4.1)
  const double tau = S.tau, bty = S.a[5], ctx = S.a[7];
  const int status = S.status;
  double sx = 1.0 / tau, sy = 1.0 / tau;
  if (status == ABIP_PRIMAL_INFEASIBLE) { sx = 1.0; sy = 1.0 / bty; }
  if (status == ABIP_DUAL_INFEASIBLE) { sx = -1.0 / ctx; sy = 1.0; }
  for (int e = threadIdx.x; e < mr; e += kThr) {
    const int i = own.at(e);
    I.y[i] = y[e];
    I.out_y[i] = y[e] * sy;
  }
  for (int e = threadIdx.x; e < nr; e += kThr) {
    const int j = own.at(e);
    I.x[j] = x[e];
    I.s[j] = s[e];
    if (I.out_x) I.out_x[j] = x[e] * sx;
    if (I.out_s) I.out_s[j] = s[e] * sy;
  }
  cl.sync();   // the descriptor is read by every CTA until here
  if (rank == 0 && threadIdx.x == 0) {
    const double* a = S.a;
    const int64_t total = S.total;
    I.tau = tau; I.kappa = S.kappa; I.theta = S.theta; I.mu = S.mu;
    I.resume = 0;
    I.pres = sqrt(a[1]) / (1.0 + nb);
    I.dres = sqrt(a[2]) / (1.0 + nc);
    I.dgap = fabs(ctx / tau - bty / tau) / (1.0 + fabs(ctx / tau) + fabs(bty / tau));
    I.ctx = ctx; I.bty = bty; I.obj = ctx / tau;
    I.admm_iters = total; I.outer_iters = S.outer; I.status = status;
    I.fp32_iters_lo = (int32_t)(total & 0x7fffffff);
    I.fp32_iters_hi = (int32_t)(total >> 31);
    if (!S.ok) I.err = DEV_ERR_NONFINITE;
  }
}

template <int MINB>
__global__ void __launch_bounds__(kThr, MINB) dense_mixed_kernel(MixArgs Q) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double wsum[9 * kWarps], hz[2];
  __shared__ MixScal S;
  __shared__ int s_id;
  const cg::cluster_group cl = cg::this_cluster();
  cl.sync();   // no CTA writes to a peer (s_id below) that may not have started
  for (;;) {
    if (cl.block_rank() == 0 && threadIdx.x == 0) {
      const int k = atomicAdd(Q.queue, 1);
      const int id = k < Q.count ? (Q.order ? Q.order[k] : k) : -1;
      for (int r = 0; r < (int)cl.num_blocks(); ++r) *cl.map_shared_rank(&s_id, r) = id;
    }
    cl.sync();
    const int id = s_id;
    if (id < 0) return;   // the same in every CTA, after which none writes to another
    DenseInst& I = Q.insts[id];
    if (I.err == 0) delta_group(I, Q, smraw, wsum, hz, S);
    cl.sync();            // every CTA has read s_id and its copies
  }
}

using MixFn = void (*)(MixArgs);
MixFn mix_fn(int variant) {
  return variant == 2 ? dense_mixed_kernel<4> : variant == 1 ? dense_mixed_kernel<3> : dense_mixed_kernel<2>;
}

constexpr size_t kSmemMax = 224 * 1024;

}  // namespace

static cudaError_t mixed_config(const DenseGroupPlan& plan, int variant, cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at) {
  const MixFn f = mix_fn(variant);
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  // one split of the SM's memory for every launch, so that buckets of different shared memory
  // run side by side on an SM (a mixed batch of 128 LPs, 200 updates: 17.9 -> 11.7 ms)
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && plan.ctas > 8) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cfg.blockDim = dim3(kThr);
  cfg.gridDim = dim3((unsigned)plan.ctas);
  cfg.dynamicSmemBytes = plan.smem;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)plan.ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return e;
}

int plan_dense_mixed(const int* m, const int* n, int count, int C, size_t budget, DenseGroupPlan& plan) {
  auto at = [&](int c) {
    size_t base = 0, copy = 0;
    for (int k = 0; k < count; ++k) {
      const size_t d = mix_doubles(m[k], n[k], c) * 8, mp = (m[k] + 3) / 4 * 4;
      base = std::max(base, d);
      copy = std::max(copy, d + 16 + (size_t)Own::count(n[k], 256 / c, 0) * mp * 4);
    }
    plan = DenseGroupPlan{};
    plan.ctas = c;
    plan.smem = copy <= budget ? copy : base;
    plan.cache_mat = copy <= budget;
    return plan.smem <= kSmemMax;
  };
  for (; !at(C); C *= 2)
    if (C >= 16) return 0;
  // fewer CTAs where the device holds no cluster of that size (16 need an SM each of one GPC)
  for (; C >= 1 && at(C); C /= 2) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    int n_active = 0;
    if (mixed_config(plan, 0, cfg, attr) == cudaSuccess && cudaOccupancyMaxActiveClusters(&n_active, mix_fn(0), &cfg) == cudaSuccess &&
        n_active > 0)
      return 1;
    cudaGetLastError();
  }
  return 0;
}

cudaError_t launch_dense_mixed(DenseInst* inst, int count, const DenseParams& prm, int* queue, const int* order,
                               const DenseGroupPlan& plan, int variant, cudaStream_t st) {
  MixArgs Q{inst, count, prm, queue, order, plan.cache_mat};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cudaError_t e = mixed_config(plan, variant, cfg, at);
  if (e != cudaSuccess) return e;
  int ncl = 0;
  e = cudaOccupancyMaxActiveClusters(&ncl, mix_fn(variant), &cfg);
  if (e != cudaSuccess) return e;
  if (ncl < 1) return cudaErrorInvalidConfiguration;
  cfg.gridDim = dim3((unsigned)(std::min(count, ncl) * plan.ctas));
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, mix_fn(variant), Q);
}

int dense_mixed_ctas_per_sm(const DenseGroupPlan& plan, int variant) {
  int per = 0;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  if (mixed_config(plan, variant, cfg, at) != cudaSuccess) return 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, mix_fn(variant), kThr, plan.smem);
  return per;
}

}  // namespace abip
