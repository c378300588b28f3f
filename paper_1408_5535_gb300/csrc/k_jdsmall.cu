// The inner solve of the Jacobi-Davidson correction equation (k_inner.cu) for
// short vectors: all MINRES steps of a block in one launch of one cluster.
//
// A step of the general form is 20 small launches, 66 us at n = 4096 for four
// systems, of which the arithmetic is a few: the rest is the chain of launches
// and their ramps.  Here a cluster of 16 CTAs (or 8) keeps the systems to itself:
// the phases of a step are separated by hardware cluster barriers, the vectors
// stay in L2, each row belongs to one thread for the whole solve, and the
// reductions go through distributed shared memory, in a fixed order.  Every CTA
// carries the scalars of the recurrences, alike.
//   1. u = D^-1/2 v (scaled form), g = Q^T u
//   2. u <- u - Q g, row-major copy for the product
//   3. z = A u
//   4. y = A^T z (own rows), Q^T y, u^T y, u^T u, x^T y
//   5. the projected, shifted operator and the Lanczos recurrence, ||y||^2
//   6. Givens step, w, s, v (no barrier: own rows)
// One cluster has the bandwidth of 16 SMs, about 0.35 TB/s of L2, and a step has 4
// barriers, in the scaled form 5 (after xrm, z and each reduction), at 4 to 6 us with the
// work between them (29 us at n = 4096).  Time of stage 1 per step, general
// form and this one (four systems, scaled form, weighted grid gradients):
//   n = 4096 FP32 (3 MB moved)      71 and 29 us    n = 10,000 FP64 (15 MB) 112 and 83 us
//   n = 16,384 FP64 (24 MB)        114 and 94 us    n = 32,400 FP32 (24 MB)  84 and 68 us
//   n = 50,176 FP32 (38 MB)         83 and 82 us    n = 65,536 FP32 (48 MB)  88 and 94 us
//   n = 32,400 FP64 (47 MB)        118 and 156 us
// FP32 meets the general form near 38 MB, FP64 near 30 MB; JD_SMALL_BYTES lies
// below both.  A whole solve (10 smallest values, n = 4096) takes 82 ms,
// with the general form 167 ms.
#include <cooperative_groups.h>

#include "cluster.cuh"
#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace ph {

namespace {

constexpr int JT = 512, JW = JT / 32;     // threads and warps per CTA
constexpr int JMAXC = 16;                 // CTAs at most
constexpr int JV = 64 * 8 + 24;           // values of a reduction at most: Q^T y and three dots per system

template <typename T>
struct JdSmem {
  double slot[2][JMAXC][JV];              // partial sums of every CTA, by parity of the reduction
  double sum[JV];
  T sumt[JV];                             // the same in T, for the row loops (a conversion holds the FP64 pipe)
  T wsum[JW][JV];                         // warp sums
  T cf[9][8];                             // the scalars of the row loops in T
  double beta1[8], beta[8], oldb[8], dbar[8], epsln[8], phibar[8], cs[8], sn[8], phi[8], gamma[8], delta[8], oldeps[8],
      alfa[8], act[8], theta[8];
};

struct JdArgs {
  int n, m, q, nq, scaled, steps, nc;     // nc: CTAs
  int la, lat;                            // lanes per row of A, of A^T
  const int *rp, *ci, *cp, *ri;
  const void *va, *cv;
  const void *Xq, *X, *ds;
  void *v, *u, *r1, *r2, *w1, *w2, *sol, *cvec, *xrm, *z;
  const double* theta;
  double* sc;
  int* done;                              // steps taken
  double tol;
};

// FP32 -> FP64 on the integer pipe (finite values; the sums of a solve that has
// broken down may be anything)
__device__ __forceinline__ double wide(float f) {
  const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
  if (m < 0x00800000u) return 0.0;
  if (m >= 0x7f800000u) return __hiloint2double(0x7ff80000, 0);
  return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double wide(double f) { return f; }

template <typename T, int Q>
__global__ void __launch_bounds__(JT, 1) k_jd_cluster(JdArgs g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  JdSmem<T>& sm = *reinterpret_cast<JdSmem<T>*>(smem_raw);
  cg::cluster_group cl = cg::this_cluster();
  const int cr = (int)cl.block_rank(), nc = g.nc, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = g.n, q = g.q, nq = g.nq;
  const int per = (n + nc - 1) / nc, i0 = min(n, cr * per), i1 = min(n, i0 + per);
  const int mper = (g.m + nc - 1) / nc, m0 = min(g.m, cr * mper), m1 = min(g.m, m0 + mper);
  const T* Xq = static_cast<const T*>(g.Xq);
  const T* X = static_cast<const T*>(g.X);
  const T* ds = static_cast<const T*>(g.ds);
  T *v = static_cast<T*>(g.v), *u = static_cast<T*>(g.u), *r1 = static_cast<T*>(g.r1), *r2 = static_cast<T*>(g.r2);
  T *w1 = static_cast<T*>(g.w1), *w2 = static_cast<T*>(g.w2), *sol = static_cast<T*>(g.sol);
  T *cv = static_cast<T*>(g.cvec), *xrm = static_cast<T*>(g.xrm), *z = static_cast<T*>(g.z);
  if (tid < 8) {
    const int c = tid;
    sm.beta1[c] = g.sc[0 * 8 + c];
    sm.beta[c] = g.sc[1 * 8 + c];
    sm.oldb[c] = g.sc[2 * 8 + c];
    sm.dbar[c] = g.sc[3 * 8 + c];
    sm.epsln[c] = g.sc[4 * 8 + c];
    sm.phibar[c] = g.sc[5 * 8 + c];
    sm.cs[c] = g.sc[6 * 8 + c];
    sm.sn[c] = g.sc[7 * 8 + c];
    sm.act[c] = g.sc[JD_FIELD_ACT * 8 + c];
    sm.theta[c] = c < q ? g.theta[c] : 0.0;
    sm.cf[0][c] = (T)sm.theta[c];
    sm.cf[8][c] = sm.act[c] != 0.0 ? T(1) : T(0);
  }
  const bool long_a = long_rows<JT>(g.rp, m0, m1, g.la), long_t = long_rows<JT>(g.cp, i0, i1, g.lat);
  cl.sync();                                       // every CTA has started, and its scalars are set
  int par = 0;                                     // parity of the reductions
  // sm.sum / sm.sumt[0 .. cnt) = the sums over the CTAs of sm.wsum
  auto reduce = [&](int cnt) {
    __syncthreads();
    for (int o = tid; o < cnt; o += JT) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < JW; ++w) t += wide(sm.wsum[w][o]);
      for (int r = 0; r < nc; ++r) cl.map_shared_rank(&sm, r)->slot[par][cr][o] = t;
    }
    cl.sync();
    for (int o = tid; o < cnt; o += JT) {
      double t = 0.0;
#pragma unroll 8
      for (int r = 0; r < nc; ++r) t += sm.slot[par][r][o];
      sm.sum[o] = t;
      sm.sumt[o] = (T)t;
    }
    par ^= 1;                                      // (the next one must not overwrite what a slow CTA still reads)
    __syncthreads();
  };
  // the warp's sums of 32 values per thread into wsum[off .. off + cnt), cnt <= 32
  auto warp_sums = [&](T (&v)[32], int off, int cnt) {
    reduce_scatter<T, 32>(v, lane);
    if (lane < cnt) sm.wsum[warp][off + lane] = v[0];
  };
  // wsum[off + l * Q + c] = sums over this CTA's rows of Xq(i, l) y(i, c)
  auto project = [&](const T* y, int off) {
    constexpr int GL = 32 / Q;                     // basis vectors per group of 32 sums
    for (int l0 = 0; l0 < nq; l0 += GL) {
      T s[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) s[k] = T(0);
      for (int i = i0 + tid; i < i1; i += JT) {
        T yr[Q];
#pragma unroll
        for (int c = 0; c < Q; ++c) yr[c] = c < q ? y[(size_t)c * n + i] : T(0);
#pragma unroll
        for (int l = 0; l < GL; ++l) {
          const T x = l0 + l < nq ? Xq[(size_t)(l0 + l) * n + i] : T(0);
#pragma unroll
          for (int c = 0; c < Q; ++c) s[l * Q + c] = fma(x, yr[c], s[l * Q + c]);
        }
      }
      warp_sums(s, off + l0 * Q, min(GL, nq - l0) * Q);
    }
  };
  int step = 0;
  for (; step < g.steps; ++step) {
    bool any = false;
    for (int c = 0; c < q; ++c) any = any || sm.cf[8][c] != T(0);
    if (!any) break;                               // the same in every CTA
    // ---- 1, 2: the operator's input u, row-major for the product
    if (g.scaled) {
      for (int i = i0 + tid; i < i1; i += JT) {
        const T d = ds[i];
        for (int c = 0; c < q; ++c) u[(size_t)c * n + i] = d * v[(size_t)c * n + i];
      }
      if (nq) {
        project(u, 0);
        reduce(nq * Q);
      }
    }
    const bool sub = g.scaled && nq;
    for (int i = i0 + tid; i < i1; i += JT) {
      T y[Q];
#pragma unroll
      for (int c = 0; c < Q; ++c) y[c] = c < q ? u[(size_t)c * n + i] : T(0);
      if (sub) {
#pragma unroll 4
        for (int l = 0; l < nq; ++l) {
          const T x = Xq[(size_t)l * n + i];
#pragma unroll
          for (int c = 0; c < Q; ++c) y[c] = fma(-x, sm.sumt[l * Q + c], y[c]);
        }
        for (int c = 0; c < Q; ++c)
          if (c < q) u[(size_t)c * n + i] = y[c];
      }
      store_row<T, Q>(xrm + (size_t)i * Q, y);
    }
    cl.sync();
    // ---- 3: z = A u
    spmm_rows<T, Q, JT>(g.rp, g.ci, static_cast<const T*>(g.va), xrm, m0, m1, g.la, long_a,
                    [&](int i, const T (&acc)[Q]) { store_row<T, Q>(z + (size_t)i * Q, acc); });
    cl.sync();
    // ---- 4: y = A^T z on the own rows, and its projections
    spmm_rows<T, Q, JT>(g.cp, g.ri, static_cast<const T*>(g.cv), z, i0, i1, g.lat, long_t, [&](int i, const T (&acc)[Q]) {
#pragma unroll
      for (int c = 0; c < Q; ++c)
        if (c < q) cv[(size_t)c * n + i] = acc[c];
    });
    __syncthreads();
    {
      T s[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) s[k] = T(0);
      for (int i = i0 + tid; i < i1; i += JT)
#pragma unroll
        for (int c = 0; c < Q; ++c)
          if (c < q) {
            const T a = u[(size_t)c * n + i], y = cv[(size_t)c * n + i];
            s[c] = fma(a, y, s[c]);
            s[8 + c] = fma(a, a, s[8 + c]);
            if (X) s[16 + c] = fma(X[(size_t)c * n + i], y, s[16 + c]);
          }
      warp_sums(s, 0, 24);
      project(cv, 24);
      reduce(24 + nq * Q);
    }
    if (tid < q && sm.act[tid] != 0.0) {
      const int c = tid;
      const double alfa = sm.sum[c] - sm.theta[c] * sm.sum[8 + c];
      sm.alfa[c] = alfa;
      sm.cf[1][c] = (T)((step > 0 && sm.oldb[c] > 0.0) ? sm.beta[c] / sm.oldb[c] : 0.0);
      sm.cf[2][c] = (T)(alfa / sm.beta[c]);
    }
    __syncthreads();
    // ---- 5: y = C u - theta u - Q (Q^T C u) - x (x^T C u), scaled, minus the Lanczos
    // terms; r1 <- r2, r2 <- y
    {
      T s[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) s[k] = T(0);
      T th[Q], ex[Q], k1[Q], k2[Q];
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        th[c] = sm.cf[0][c];
        ex[c] = sm.sumt[16 + c];
        k1[c] = sm.cf[1][c];
        k2[c] = sm.cf[2][c];
      }
      for (int i = i0 + tid; i < i1; i += JT) {
        T y[Q];
#pragma unroll
        for (int c = 0; c < Q; ++c) {
          y[c] = T(0);
          if (c < q) {
            const size_t k = (size_t)c * n + i;
            y[c] = fma(-th[c], u[k], cv[k]);
            if (X) y[c] = fma(-ex[c], X[k], y[c]);
          }
        }
#pragma unroll 4
        for (int l = 0; l < nq; ++l) {
          const T x = Xq[(size_t)l * n + i];
#pragma unroll
          for (int c = 0; c < Q; ++c) y[c] = fma(-x, sm.sumt[24 + l * Q + c], y[c]);
        }
        const T d = g.scaled ? ds[i] : T(1);
#pragma unroll
        for (int c = 0; c < Q; ++c)
          if (c < q && sm.cf[8][c] != T(0)) {
            const size_t k = (size_t)c * n + i;
            const T a1 = r1[k], a2 = r2[k];
            const T t = fma(-k2[c], a2, fma(-k1[c], a1, g.scaled ? y[c] * d : y[c]));
            s[c] = fma(t, t, s[c]);
            r1[k] = a2;
            r2[k] = t;
          }
      }
      warp_sums(s, 0, 8);
      reduce(8);
    }
    // ---- 6: the Givens step (MINRES), then w, s and the next v
    if (tid < q) {
      const int c = tid;
      if (sm.act[c] == 0.0) {
        sm.phi[c] = 0.0;
      } else {
        const double alfa = sm.alfa[c], oldb = sm.beta[c], beta = sqrt(fmax(sm.sum[c], 0.0));
        const double cs = sm.cs[c], sn = sm.sn[c], dbar = sm.dbar[c], oldeps = sm.epsln[c];
        const double gbar = sn * dbar - cs * alfa;
        const double gamma = fmax(sqrt(gbar * gbar + beta * beta), 1e-300);
        const double cs2 = gbar / gamma, sn2 = beta / gamma, phibar = sm.phibar[c];
        sm.oldb[c] = oldb;
        sm.beta[c] = beta;
        sm.oldeps[c] = oldeps;
        sm.delta[c] = cs * dbar + sn * alfa;
        sm.epsln[c] = sn * beta;
        sm.dbar[c] = -cs * beta;
        sm.gamma[c] = gamma;
        sm.cs[c] = cs2;
        sm.sn[c] = sn2;
        sm.phi[c] = cs2 * phibar;
        sm.phibar[c] = sn2 * phibar;
        const double b1 = sm.beta1[c];
        if (!(sn2 * fabs(phibar) > g.tol * b1) || !(beta > 1e-30 * b1)) sm.act[c] = -1.0;   // stops after this update
      }
      sm.cf[3][c] = (T)sm.oldeps[c];
      sm.cf[4][c] = (T)sm.delta[c];
      sm.cf[5][c] = (T)(1.0 / sm.gamma[c]);
      sm.cf[6][c] = (T)sm.phi[c];
      sm.cf[7][c] = (sm.act[c] > 0.0 && sm.beta[c] > 0.0) ? (T)(1.0 / sm.beta[c]) : T(0);
      sm.cf[8][c] = sm.act[c] != 0.0 ? T(1) : T(0);
    }
    __syncthreads();
    {
      T ce[Q], cd[Q], cg_[Q], cp_[Q], cb[Q];
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        ce[c] = sm.cf[3][c];
        cd[c] = sm.cf[4][c];
        cg_[c] = sm.cf[5][c];
        cp_[c] = sm.cf[6][c];
        cb[c] = sm.cf[7][c];
      }
      for (int i = i0 + tid; i < i1; i += JT)
#pragma unroll
        for (int c = 0; c < Q; ++c)
          if (c < q && sm.cf[8][c] != T(0)) {
            const size_t k = (size_t)c * n + i;
            const T a1 = w1[k], a2 = w2[k];
            const T w = (v[k] - ce[c] * a1 - cd[c] * a2) * cg_[c];
            w1[k] = a2;
            w2[k] = w;
            sol[k] = fma(cp_[c], w, sol[k]);
            v[k] = r2[k] * cb[c];
          }
    }
    __syncthreads();
    if (tid < q) {
      if (sm.act[tid] < 0.0) sm.act[tid] = 0.0;
      sm.cf[8][tid] = sm.act[tid] != 0.0 ? T(1) : T(0);
    }
    __syncthreads();
  }
  if (cr == 0 && tid == 0) *g.done = step;
  cl.sync();                                       // no CTA leaves while a peer may still reach it
}

template <typename T, int Q>
int cluster_ctas() {
  static std::atomic<int> known[64];
  return cluster_size(k_jd_cluster<T, Q>, JT, sizeof(JdSmem<T>), sizeof(JdSmem<T>), known);
}

template <typename T, int Q>
bool go(cudaStream_t s, JdArgs g) {
  // (a barrier of 8 costs less than short vectors gain from 16)
  g.nc = std::min(cluster_ctas<T, Q>(), g.n <= 4 * JT ? 8 : 16);
  return g.nc && launch_cluster(k_jd_cluster<T, Q>, g.nc, JT, sizeof(JdSmem<T>), s, g);
}

}  // namespace

template <typename T>
bool jd_solve_small(cudaStream_t s, const SparseView<T>& A, const SparseView<T>& At, int q, int nq, bool scaled,
                    const T* Xq, const T* X, const T* ds, const double* theta, T* v, T* u, T* r1, T* r2, T* w1, T* w2,
                    T* sol, T* cv, T* xrm, T* z, double* sc, int steps, double tol, int* done) {
  const int n = At.nrows, Q = q >= 5 ? 8 : q >= 3 ? 4 : q;
  // bytes a step moves through the cluster's L2 ports: Q (scaled form twice more),
  // the vectors, the gathers (of the CTA with the most entries, times the CTAs)
  const double bytes =
      sizeof(T) * ((double)n * (nq * (scaled ? 4 : 2) + 20.0 * q) + (A.skew + At.skew) * A.nnz * (Q + 2));
  if (bytes > JD_SMALL_BYTES || nq > 64) return false;
  ProfScope ps(s, sizeof(T) == 4 ? PROF_F32 + PROF_SMALL : PROF_SMALL);
  JdArgs g{};
  g.n = n;
  g.m = A.nrows;
  g.q = q;
  g.nq = nq;
  g.scaled = scaled;
  g.steps = steps;
  g.la = cluster_lanes(A.avg_row());
  g.lat = cluster_lanes(At.avg_row());
  g.rp = A.ptr;
  g.ci = A.idx;
  g.va = A.val;
  g.cp = At.ptr;
  g.ri = At.idx;
  g.cv = At.val;
  g.Xq = Xq;
  g.X = X;
  g.ds = ds;
  g.v = v;
  g.u = u;
  g.r1 = r1;
  g.r2 = r2;
  g.w1 = w1;
  g.w2 = w2;
  g.sol = sol;
  g.cvec = cv;
  g.xrm = xrm;
  g.z = z;
  g.theta = theta;
  g.sc = sc;
  g.done = done;
  g.tol = tol;
  switch (Q) {
    case 1: return go<T, 1>(s, g);
    case 2: return go<T, 2>(s, g);
    case 4: return go<T, 4>(s, g);
    default: return go<T, 8>(s, g);
  }
}
template bool jd_solve_small<float>(cudaStream_t, const SparseView<float>&, const SparseView<float>&, int, int, bool,
                                    const float*, const float*, const float*, const double*, float*, float*, float*,
                                    float*, float*, float*, float*, float*, float*, float*, double*, int, double, int*);
template bool jd_solve_small<double>(cudaStream_t, const SparseView<double>&, const SparseView<double>&, int, int, bool,
                                     const double*, const double*, const double*, const double*, double*, double*,
                                     double*, double*, double*, double*, double*, double*, double*, double*, double*,
                                     int, double, int*);

}  // namespace ph
