// One block of stage 1 joins the basis, for short vectors, in one launch of one
// cluster: orthogonalisation against [Xl | V] (classical Gram-Schmidt twice, then
// CholQR twice), W = C V of the new columns and the new rows of the projected matrix.
//
// The general form is 25 to 30 graph nodes (norms, three Gram-Schmidt passes with
// their sums, two Cholesky factors, two products, transposes, the new Gram columns,
// and a memset before each sum) and one host read in between: 90 us at n = 1000
// for one column, of which 15 are arithmetic.  Here
// each row belongs to one CTA of the cluster, the block's rows stay in shared
// memory, V's in L1/L2; the phases meet at 5 to 7 cluster barriers, sums go through
// distributed shared memory in a fixed order, and every CTA factorises alike.
//   warps x 4 columns    G = P^T T: lanes over the rows, butterflies in T, CTAs in FP64
//   rows x LG lanes      T -= P G: LG lanes share the columns of a row
// Sums are as accurate as the general form's, which adds two terms per lane and a warp's
// lanes in T, and FP64 from there.  A lane has up to 63 terms here: in FP32 it adds four at
// a time, and these, as the lanes, with the rounding error carried along (two_sum), FP64
// across CTAs; in FP64 plainly.
//
// Time per iteration of stage 1 with the general form and with this one (2n x n, 8 entries
// per row, 35 basis vectors at most, blocks of 1, 4, 8); a dash: this one not taken (forced, it
// was the slower one there):
//   FP64 n =   300   212 144   406 304   641 469 us
//        n =  1000   210 144   360 272   507 387
//        n =  2000   207 151   356 309   521 455
//        n =  8000   225 175   365 350   553  -
//        n = 16000   232 223   380  -    566  -
//   FP32 n =   300   200 129   337 218   521 348
//        n =  1000   207 133   335 218   461 313
//        n =  8000   219 156   339 248   487 370
//        n = 16000   230 186   366 290   541 451
//        n = 32000   227  -    375  -    568  -
// In FP64 the 16 SMs' arithmetic decides (n p b), in FP32 their reads of the basis
// (n p).  A 2000 x 1000 solve with the defaults: 174 ms -> 122 to 140 ms (its iterations vary
// with the autotuned product).
#include <algorithm>

#include <cooperative_groups.h>

#include "cluster.cuh"
#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace ph {

namespace {

constexpr int XT = 512, XW = XT / 32;
constexpr int XC = 4;                     // columns of P per warp and round
constexpr int XMAXC = 16;

struct ExSmem {
  double G[64], N[8], L[64], M[64];
  int bad;
};

struct ExArgs {
  int n, m, nb, nlock, j, nc, rows, cap, la, lat, nsp, ldh;
  const int *rp, *ci, *cp, *ri;
  const void *va, *cv;
  const void* Xl;
  void *V, *W, *Tb, *xrm, *z;
  double *Ht, *S, *sprev;
  int *flags, *bad;
};

// Cholesky of the q x q Gram matrix P by one warp, M = L^{-T}; returns whether a
// column lost all but drop of its norm (ref: squared norms before, or null), with
// its flag in fl[c].
__device__ bool warp_chol(int q, const double* P, const double* ref, double drop, double* L, double* M, int* fl,
                          int lane) {
  int bad = 0;
  for (int c = 0; c < q; ++c) {
    double d = P[c + c * q];
    for (int k = 0; k < c; ++k) d -= L[c + k * 8] * L[c + k * 8];
    const double r0 = ref ? ref[c] : P[c + c * q];
    int f = 0;
    if (!(d > drop * drop * r0) || !(d > 0.0)) {
      f = 1;
      d = 1.0;                                     // keep the factor finite; the caller replaces the column
    }
    if (fl && lane == 0) fl[c] = f;
    bad |= f;
    const double lcc = sqrt(d);
    if (lane == c) L[c + c * 8] = lcc;
    if (lane > c && lane < q) {
      double v = P[lane + c * q];
      for (int k = 0; k < c; ++k) v -= L[lane + k * 8] * L[c + k * 8];
      L[lane + c * 8] = f ? 0.0 : v / lcc;
    }
    __syncwarp();
  }
  if (lane < q)                                    // L^T M = I, a column per lane
    for (int r = q - 1; r >= 0; --r) {
      double v = r == lane ? 1.0 : 0.0;
      for (int k = r + 1; k < q; ++k) v -= L[k + r * 8] * M[k + lane * 8];
      M[r + lane * 8] = v / L[r + r * 8];
    }
  if (fl && lane == 0) fl[q] = bad;
  __syncwarp();
  return bad;
}

// hi + lo = the sum so far plus v, to twice FP32 (Knuth's TwoSum: exact for hi + v).
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v) {
  const float s = __fadd_rn(hi, v), z = __fadd_rn(s, -hi);
  lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(hi, -__fadd_rn(s, -z)), __fadd_rn(v, -z)));
  hi = s;
}
// As reduce_scatter, of sums hi + lo.
template <int N, int O, int CUR>
__device__ __forceinline__ void reduce_scatter2(float (&hi)[N], float (&lo)[N], int lane) {
  if constexpr (O > 0) {
    constexpr int H = CUR > 1 ? CUR / 2 : 1;
    const bool up = CUR > 1 && (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      float a = hi[i], b = lo[i], sa = a, sb = b;  // what the lane keeps and what it sends
      if constexpr (CUR > 1) {
        if (up) {
          a = hi[i + H];
          b = lo[i + H];
        } else {
          sa = hi[i + H];
          sb = lo[i + H];
        }
      }
      const float ra = __shfl_xor_sync(0xffffffffu, sa, O), rb = __shfl_xor_sync(0xffffffffu, sb, O);
      two_sum(a, b, ra);
      hi[i] = a;
      lo[i] = __fadd_rn(b, rb);
    }
    reduce_scatter2<N, O / 2, H>(hi, lo, lane);
  }
}

template <typename T, int Q>
__global__ void __launch_bounds__(XT, 1) k_expand_cluster(ExArgs g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ ExSmem sm;
  cg::cluster_group cl = cg::this_cluster();
  const int cr = (int)cl.block_rank(), nc = g.nc, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* slot = reinterpret_cast<double*>(smem_raw);            // [2][nc][cap]
  double* sum = slot + (size_t)2 * nc * g.cap;                   // [cap]
  T* sumt = reinterpret_cast<T*>(sum + g.cap);                   // [cap]
  T* ts = sumt + g.cap;                                          // [Q][rows]
  const int n = g.n, q = g.nb, j = g.j, nlock = g.nlock, p = nlock + j, R = g.rows;
  const int i0 = min(n, cr * R), nr = min(n, i0 + R) - i0;       // own rows
  const int mper = (g.m + nc - 1) / nc, m0 = min(g.m, cr * mper), m1 = min(g.m, m0 + mper);
  const T* Xl = static_cast<const T*>(g.Xl) + i0;
  T *V = static_cast<T*>(g.V) + i0, *W = static_cast<T*>(g.W), *Tb = static_cast<T*>(g.Tb) + i0;
  T *xrm = static_cast<T*>(g.xrm), *z = static_cast<T*>(g.z);
  for (int e = tid; e < Q * R; e += XT) {
    const int c = e / R, i = e - c * R;
    ts[e] = c < q && i < nr ? Tb[(size_t)c * n + i] : T(0);
  }
  const bool long_a = long_rows<XT>(g.rp, m0, m1, g.la), long_t = long_rows<XT>(g.cp, i0, i0 + nr, g.lat);
  cl.sync();                                       // (every CTA has started: its shared memory can be written)
  int par = 0;
  // sum[l * Q + r] = sum over all rows of (column l) . T(:, r): the columns of Xl
  // (c1), of V (c2), then T's own
  auto dots = [&](int c1, int c2, bool own) {
    const int L = c1 + c2 + (own ? Q : 0);
    __syncthreads();
    for (int l0 = warp * XC; l0 < L; l0 += XW * XC) {
      const T* pc[XC];
#pragma unroll
      for (int a = 0; a < XC; ++a) {
        const int l = l0 + a;
        pc[a] = l < c1 ? Xl + (size_t)l * n : l < c1 + c2 ? V + (size_t)(l - c1) * n : l < L ? ts + (l - c1 - c2) * R
                                                                                            : ts;
      }
      T s[XC * Q];
#pragma unroll
      for (int k = 0; k < XC * Q; ++k) s[k] = T(0);
      double total;
      if constexpr (sizeof(T) == 4) {
        constexpr int U = 4;                       // rows whose products are added plainly
        T lo[XC * Q];
#pragma unroll
        for (int k = 0; k < XC * Q; ++k) lo[k] = T(0);
        for (int i = lane; i < nr; i += 32 * U) {
          T x[U][XC];
#pragma unroll
          for (int u = 0; u < U; ++u)
#pragma unroll
            for (int a = 0; a < XC; ++a) x[u][a] = i + 32 * u < nr ? pc[a][i + 32 * u] : T(0);
#pragma unroll
          for (int r = 0; r < Q; ++r) {
            T t[U];
#pragma unroll
            for (int u = 0; u < U; ++u) t[u] = i + 32 * u < nr ? ts[r * R + i + 32 * u] : T(0);
#pragma unroll
            for (int a = 0; a < XC; ++a) {
              T v = x[0][a] * t[0];
#pragma unroll
              for (int u = 1; u < U; ++u) v = fma(x[u][a], t[u], v);
              two_sum(s[a * Q + r], lo[a * Q + r], v);
            }
          }
        }
        reduce_scatter2<XC * Q, 16, XC * Q>(s, lo, lane);
        total = (double)s[0] + (double)lo[0];
      } else {
#pragma unroll 2
        for (int i = lane; i < nr; i += 32) {
          T x[XC];
#pragma unroll
          for (int a = 0; a < XC; ++a) x[a] = pc[a][i];
#pragma unroll
          for (int r = 0; r < Q; ++r) {
            const T t = ts[r * R + i];
#pragma unroll
            for (int a = 0; a < XC; ++a) s[a * Q + r] = fma(x[a], t, s[a * Q + r]);
          }
        }
        reduce_scatter<T, XC * Q>(s, lane);
        total = s[0];
      }
      constexpr int REP = 32 / (XC * Q);           // lanes that hold the same sum
      const int o = l0 * Q + lane / REP;
      if (o < L * Q)
        for (int r = lane % REP; r < nc; r += REP)
          *cl.map_shared_rank(slot + ((size_t)par * nc + cr) * g.cap + o, r) = total;
    }
    cl.sync();
    for (int o = tid; o < L * Q; o += XT) {
      double t = 0.0;
#pragma unroll 8
      for (int r = 0; r < nc; ++r) t += slot[((size_t)par * nc + r) * g.cap + o];
      sum[o] = t;
      sumt[o] = (T)t;
    }
    par ^= 1;                                      // (the next must not overwrite what a slow CTA still reads)
    __syncthreads();
  };
  // T -= P sum, LG lanes per row
  auto subtract = [&](int LG) {
    const int RL = 32 / LG, rl = lane % RL, lg = lane / RL;
    for (int base = warp * RL; base < nr; base += XW * RL) {
      const int i = base + rl;
      T acc[Q];
#pragma unroll
      for (int r = 0; r < Q; ++r) acc[r] = T(0);
      if (i < nr) {
#pragma unroll 4
        for (int l = lg; l < p; l += LG) {
          const T x = (l < nlock ? Xl + (size_t)l * n : V + (size_t)(l - nlock) * n)[i];
#pragma unroll
          for (int r = 0; r < Q; ++r) acc[r] = fma(x, sumt[l * Q + r], acc[r]);
        }
      }
      for (int o = RL; o < 32; o <<= 1)
#pragma unroll
        for (int r = 0; r < Q; ++r) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], o);
      if (lg == 0 && i < nr)
#pragma unroll
        for (int r = 0; r < Q; ++r) ts[r * R + i] -= acc[r];
    }
  };
  // the q x q Gram matrix of T among the sums from row l on
  auto gram = [&](int l) {
    if (tid < q * q) sm.G[tid] = sum[(l + tid % q) * Q + tid / q];
    __syncthreads();
  };
  // T <- T M; the last one also into V and, row-major, for the product
  auto scale = [&](bool last) {
    for (int i = tid; i < nr; i += XT) {
      T t[Q], o[Q];
#pragma unroll
      for (int r = 0; r < Q; ++r) t[r] = ts[r * R + i];
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        o[c] = T(0);
        if (c < q)
          for (int r = 0; r < q; ++r) o[c] = fma(t[r], (T)sm.M[r + c * 8], o[c]);
      }
#pragma unroll
      for (int c = 0; c < Q; ++c) {
        ts[c * R + i] = o[c];
        if (last && c < q) V[(size_t)(j + c) * n + i] = o[c];
      }
      if (last) store_row<T, Q>(xrm + (size_t)(i0 + i) * Q, o);
    }
  };
  const int LG = R <= 64 ? 8 : R <= 128 ? 4 : R <= 256 ? 2 : 1;
  dots(nlock, j, true);
  if (tid < q) sm.N[tid] = sum[(p + tid) * Q + tid];             // squared norms on entry
  subtract(LG);
  if (p) {
    dots(nlock, j, false);
    subtract(LG);
  }
  dots(0, 0, true);
  gram(0);
  if (warp == 0) {
    const bool bad = warp_chol(q, sm.G, sm.N, 1e-10, sm.L, sm.M, cr == 0 ? g.flags : nullptr, lane);
    if (lane == 0) sm.bad = bad;
    if (lane == 0 && cr == 0) *g.bad = bad;
  }
  __syncthreads();
  if (sm.bad) {                                    // in every CTA alike: the block goes back, reduced against P
    for (int e = tid; e < q * R; e += XT) {
      const int c = e / R, i = e - c * R;
      if (i < nr) Tb[(size_t)c * n + i] = ts[e];
    }
    cl.sync();
    return;
  }
  if (q > 1) {
    scale(false);
    dots(0, 0, true);
    gram(0);
    if (warp == 0) warp_chol(q, sm.G, nullptr, 0.0, sm.L, sm.M, nullptr, lane);
    __syncthreads();
  }
  scale(true);
  cl.sync();
  spmm_rows<T, Q, XT>(g.rp, g.ci, static_cast<const T*>(g.va), xrm, m0, m1, g.la, long_a,
                      [&](int i, const T (&acc)[Q]) { store_row<T, Q>(z + (size_t)i * Q, acc); });
  cl.sync();
  spmm_rows<T, Q, XT>(g.cp, g.ri, static_cast<const T*>(g.cv), z, i0, i0 + nr, g.lat, long_t,
                      [&](int i, const T (&acc)[Q]) {
#pragma unroll
    for (int c = 0; c < Q; ++c) {
      ts[c * R + i - i0] = acc[c];
      if (c < q) W[(size_t)(j + c) * n + i] = acc[c];
    }
  });
  dots(0, j + q, false);                           // V^T W of the new columns
  if (cr == 0) {
    const int jn = j + q;
    for (int e = tid; e < jn * q; e += XT) {
      const int r = e % jn, c = e / jn;
      double v = sum[r * Q + c];
      if (r >= j) v = 0.5 * (v + sum[(j + c) * Q + (r - j)]);
      g.Ht[r + (size_t)(j + c) * g.ldh] = v;
      g.Ht[(j + c) + (size_t)r * g.ldh] = v;
      g.S[r + (size_t)(j + c) * g.ldh] = r == j + c ? 1.0 : 0.0;
      if (r < j) g.S[(j + c) + (size_t)r * g.ldh] = 0.0;
    }
    for (int e = tid; e < g.nsp * q; e += XT) g.sprev[(j + e % q) + (size_t)(e / q) * g.ldh] = 0.0;
  }
  cl.sync();                                       // no CTA leaves while a peer may still reach it
}

size_t expand_smem(int nc, int cap, int Q, int rows, size_t el) {
  return (size_t)(2 * nc + 1) * cap * 8 + (size_t)cap * el + (size_t)Q * rows * el;
}

template <typename T, int Q>
bool go(cudaStream_t s, ExArgs g) {
  static std::atomic<int> known[64];
  constexpr size_t SMEM_MAX = 200 * 1024;
  g.cap = ((std::max(g.nlock + g.j, g.j + g.nb) + Q) * Q + 1) & ~1;
  g.nc = cluster_size(k_expand_cluster<T, Q>, XT, SMEM_MAX, SMEM_MAX, known);
  if (g.nc == 0) return false;
  // 8 leave half of the SMs to the other solves of a batch, and take as long for one vector (per
  // iteration at n = 300, 500, 1000: 144, 148, 144 us with either; blocks of 8 at n = 2000: 455,
  // with 16 440)
  if (g.n <= 2048) g.nc = 8;
  g.rows = ((g.n + g.nc - 1) / g.nc + 1) & ~1;
  const size_t smem = expand_smem(g.nc, g.cap, Q, g.rows, sizeof(T));
  if (smem > SMEM_MAX) return false;
  return launch_cluster(k_expand_cluster<T, Q>, g.nc, XT, smem, s, g);
}

}  // namespace

template <typename T>
bool expand_small(cudaStream_t s, const SparseView<T>& A, const SparseView<T>& At, int nb, int nlock, int j, int nsp,
                  const T* Xl, T* V, T* W, T* Tb, T* xrm, T* z, double* Ht, double* S, double* sprev, int ldh,
                  int* flags, int* bad) {
  const int n = At.nrows, Q = nb > 4 ? 8 : nb > 2 ? 4 : nb;
  // the line (above): in FP64 the cluster's arithmetic, in FP32 its reads of the
  // basis, and the product's gathers on 16 SMs against what the launches cost
  const double np = (double)n * (nlock + j + 8);
  const double bytes = (A.skew + At.skew) * A.nnz * (Q + 2) * sizeof(T);
  if ((sizeof(T) == 8 ? np * (Q + 1) / 2e6 : np / 1e6) + bytes / (26e6 + 4e6 * Q) > 1.0) return false;
  ProfScope ps(s, sizeof(T) == 4 ? PROF_F32 + PROF_GRAM : PROF_GRAM);
  ExArgs g{};
  g.n = n;
  g.m = A.nrows;
  g.nb = nb;
  g.nlock = nlock;
  g.j = j;
  g.la = cluster_lanes(A.avg_row());
  g.lat = cluster_lanes(At.avg_row());
  g.nsp = nsp;
  g.ldh = ldh;
  g.rp = A.ptr;
  g.ci = A.idx;
  g.va = A.val;
  g.cp = At.ptr;
  g.ri = At.idx;
  g.cv = At.val;
  g.Xl = Xl;
  g.V = V;
  g.W = W;
  g.Tb = Tb;
  g.xrm = xrm;
  g.z = z;
  g.Ht = Ht;
  g.S = S;
  g.sprev = sprev;
  g.flags = flags;
  g.bad = bad;
  bool ok;
  switch (Q) {
    case 1: ok = go<T, 1>(s, g); break;
    case 2: ok = go<T, 2>(s, g); break;
    case 4: ok = go<T, 4>(s, g); break;
    default: ok = go<T, 8>(s, g); break;
  }
  if (!ok) return false;
  const double p = nlock + j, q = nb;
  count_work(sizeof(T) == 4 ? PROF_F32 + PROF_GRAM : PROF_GRAM, 2.0 * n * q * (4.0 * p + j + q) + 4.0 * n * q * (q + 1),
             (double)sizeof(T) * n * (4.0 * p + j + 6.0 * q));
  count_work(sizeof(T) == 4 ? PROF_F32 + PROF_CSPMM : PROF_CSPMM, 4.0 * (double)A.nnz * nb,
             (double)A.nnz * (sizeof(T) + 4) * 2.0 + (double)sizeof(T) * nb * (2.0 * n + 2.0 * A.nrows));
  return true;
}
template bool expand_small<float>(cudaStream_t, const SparseView<float>&, const SparseView<float>&, int, int, int, int,
                                  const float*, float*, float*, float*, float*, float*, double*, double*, double*, int,
                                  int*, int*);
template bool expand_small<double>(cudaStream_t, const SparseView<double>&, const SparseView<double>&, int, int, int,
                                   int, const double*, double*, double*, double*, double*, double*, double*, double*,
                                   double*, int, int*, int*);

}  // namespace ph
