// The projected eigenproblem of a stage-1 iteration (Algorithm 1: the Ritz pairs
// of H = V^T C V) in one launch: an FP32 Jacobi pass, then FP64 refinement.
//
// H is j x j with j <= 64, so there is nothing to move: the time is the serial
// chain.  As separate launches (FP32 frame, one-CTA Jacobi, four products for
// two Newton-Schulz steps, the FP64 frame, a Jacobi clean-up of the targets,
// ordering, gather: 19 of them) it took more than half of a small solve.  Here:
//  * a cluster of 8 CTAs works in its own shared memories.  The FP32 Jacobi pass
//    runs in every CTA alike (same data, same order, same result), so that its
//    rounds exchange nothing; of the rotation it accumulates, each CTA keeps an
//    eighth of the rows;
//  * a Jacobi round costs one barrier: every warp computes all rotations of
//    the round itself (lane = pair) and passes them around by shuffles, and the
//    matrix is read from one buffer and written to another.  8 warps: with 16,
//    issuing the rotations 16 times over took longer than the updates;
//  * FP64 accuracy comes from the quadratically convergent refinement of
//    Ogita and Aishima ("Iterative refinement for symmetric eigenvalue
//    decomposition", Jpn. J. Ind. Appl. Math. 35, 2018), which orthonormalises
//    and diagonalises at once: from X with G = X^T X and B = X^T H X,
//      lambda_i = B_ii / G_ii,  X <- X + X E,
//      E_ij = m_ij / (lambda_j - lambda_i) - G_ij / 2,  E_ii = (1 - G_ii) / 2,
//      m_ij = B_ij - (lambda_i + lambda_j) G_ij / 2,
//    by columns, each CTA its own (the products are independent of one another,
//    where FP64 Jacobi rounds depend on the one before).  Two or three steps
//    take the FP32 vectors to FP64;
//  * where a target's m_ij is not small against its gap, the targets and all that is
//    coupled to them in this way, directly or through others, are rotated first: X
//    is made orthonormal (to first order, so that the matrix of the m_ij is X^T H X),
//    then classical Jacobi until every m_ij of these rows is below E_ROT of its gap.
//    Rotating X^T H X of an X that is orthonormal to FP32 only, or the targets alone,
//    ends with the couplings of a cluster as they were: lambda G_ij outweighs its
//    gaps, and the first-order steps go through the pairs left out.  Other such pairs
//    only span the restart space and are left as they are.
// FP64 instructions hold an SM's pipe for 16 clocks a warp, so what is not a
// product (maxima, ranks, angles) runs on integers or in FP32.
// Measured: 75 us at j = 28 (of 145,000 clocks 74,000 in 108 Jacobi rounds, 54,000
// in three refinement steps), where the kernels it replaces took 326 us beside
// their launches; a 2000 x 1000 solve with the defaults, 850 iterations: 500 ms
// -> 183 ms.
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"

namespace cg = cooperative_groups;

namespace ph {

namespace {

constexpr int EC = 8;                  // CTAs
constexpr int ET = 256;                // threads per CTA
constexpr int EW = ET / 32;
constexpr int EJ = 64, EL = EJ + 1;    // largest order, leading dimension in shared memory
constexpr int EMAT = EJ * EL;
// leading dimension of the FP32 pass: its pairs are (r + k, r - k), so an even
// one puts the entries a_pq of a round in different banks, and 14 more than 64
// the blocks of neighbouring pairs
constexpr int FL = EJ + 14, FMAT = EJ * FL;
constexpr int E_STEPS = 8;             // refinement steps at most (two or three are usual)
constexpr double E_SMALL = 0.02;       // m_ij / gap up to which a pair is refined; above, rotated
// ... down to this: in a cluster the second-order terms add up over its members and the ratios
// of its gaps (emulated, 14 values within 1e-4 and the couplings that FP32 leaves: from 0.02
// the steps run out in a quarter of the cases, from here in none; 93 rotations, and 4 steps for 7)
constexpr double E_ROT = 3e-4;
constexpr int E_MOST = 8 * EJ;         // rotations at most
// Largest |E_ij| after which the update has reached FP64: it leaves X^T X = I + O(j
// E^2), and a basis transformed by less orthogonal coefficients drifts over the
// restarts.
constexpr float E_DONE = 2e-10f;
constexpr float E_ANGLE = 1e-8f;       // the largest rotation whose square is below eps
constexpr float J_TOL = 1e-6f;         // FP32 threshold, relative to max |h_ij|
constexpr int J_SWEEPS = 30;

struct EigSmem {
  double H[EMAT], X[2][EMAT], B[EMAT];
  double W[EC][EJ], Bc[EC][EJ], Gc[EC][EJ], Ec[EC][EJ];   // this CTA's columns
  double lam[EJ];
  long long key[EJ];
  double rot[2];
  float A[2][FMAT], S[FMAT];   // S: this CTA's rows of the accumulated rotation, then all
  float wmax[EC], red[EW];
  unsigned redu[EW];
  int rank[EJ];
  int sel;
  double wbest[EW];
  int wat[EW];
  unsigned char tgt[EJ];
};

__device__ inline double dot_col(const double* a, int stride, const double* x, int n) {
  double v = 0.0;
#pragma unroll 4
  for (int k = 0; k < n; ++k) v = fma(a[k * stride], x[k], v);
  return v;
}

__device__ __forceinline__ float rsqrt_fast(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_fast(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Work items of a round (below), and the most of them (j = 64).
__host__ __device__ constexpr int j_items(int jj, int rows) {
  return ((jj / 2 * (jj / 2 + 1) / 2 + 31) / 32 * 32) + rows * (jj / 2);
}
constexpr int J_MOST = (j_items(EJ, EJ / EC) + ET - 1) / ET;

// FP32 cyclic Jacobi of the jj x jj (even) matrix A[0] (|a_ij| <= 1, upper triangle),
// and S <- S J on the rows cr, cr + EC, ... of S.  Every thread of the CTA calls.
// A round is one chain (entries -> angles -> shuffles -> update -> barrier), so the
// entries to update are fetched along with those of the angles, and the pairs
// are carried from round to round: pair k of round r, round robin, is
// (r + k, r - k) mod m among m + 1 indices, and (r, m) for k = 0.  NI: items per
// thread.
template <int NI>
__device__ void jacobi32(EigSmem& sm, int jj, int cr, float thr, int& sweeps, int& rots) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int np = jj / 2, m = jj - 1;
  const int nrow = cr < jj ? (jj - cr + EC - 1) / EC : 0;
  const int nblk = np * (np + 1) / 2, first = (nblk + 31) & ~31, nitems = first + nrow * np;
  // this thread's items of every round: block (k <= l) of the matrix, or (row l,
  // pair k) of S, in warps of their own
  int kind[NI], ik[NI], il[NI];
#pragma unroll
  for (int u = 0; u < NI; ++u) {
    const int it = u * ET + tid;
    kind[u] = ik[u] = il[u] = 0;
    if (it < nblk) {
      int l = (int)((sqrtf(8.f * it + 1.f) - 1.f) * 0.5f);
      while (l * (l + 1) / 2 > it) --l;
      while ((l + 1) * (l + 2) / 2 <= it) ++l;
      kind[u] = 1;
      il[u] = l;
      ik[u] = it - l * (l + 1) / 2;
    } else if (it >= first && it < nitems) {
      const int i = (it - first) / np;
      kind[u] = 2;
      il[u] = cr + i * EC;
      ik[u] = it - first - i * np;
    }
  }
  auto up = [m](int v) { return v == m - 1 ? 0 : v + 1; };
  auto at = [](int x, int y) { return min(x, y) + max(x, y) * FL; };   // the upper triangle is kept
  int cur = 0, sweep = 0, nrot = 0;
  for (; sweep < J_SWEEPS; ++sweep) {
    const float* a = sm.A[cur];
    bool any = false;
#pragma unroll 8
    for (int c = 0; c < jj; ++c) {
      if (lane < c) any = any || fabsf(a[lane + c * FL]) > thr;
      if (lane + 32 < c) any = any || fabsf(a[lane + 32 + c * FL]) > thr;
    }
    if (!__any_sync(0xffffffffu, any)) break;
    // round 0: pair k = (k, m - k), pair 0 = (0, m); then both go up by one mod m
    int x = lane, y = m - lane;
    int xk[NI], yk[NI], xl[NI], yl[NI];
#pragma unroll
    for (int u = 0; u < NI; ++u) {
      xk[u] = ik[u];
      yk[u] = m - ik[u];
      xl[u] = il[u];
      yl[u] = m - il[u];
    }
    for (int r = 0; r < m; ++r) {
      const float* A = sm.A[cur];
      float b00[NI], b01[NI], b10[NI], b11[NI];
      int o00[NI], o01[NI], o10[NI], o11[NI];
#pragma unroll
      for (int u = 0; u < NI; ++u) {
        if (kind[u] == 1) {
          o00[u] = at(xk[u], xl[u]);
          o01[u] = at(xk[u], yl[u]);
          o10[u] = at(yk[u], xl[u]);
          o11[u] = at(yk[u], yl[u]);
          b00[u] = A[o00[u]];
          b01[u] = A[o01[u]];
          b10[u] = A[o10[u]];
          b11[u] = A[o11[u]];
        } else if (kind[u] == 2) {
          o00[u] = il[u] + xk[u] * FL;
          o01[u] = il[u] + yk[u] * FL;
          b00[u] = sm.S[o00[u]];
          b01[u] = sm.S[o01[u]];
        }
      }
      // lane k: the rotation of pair k
      float c = 1.f, s = 0.f;
      bool rot = false;
      if (lane < np) {
        const float axy = A[at(x, y)], d = A[y + y * FL] - A[x + x * FL];
        rot = fabsf(axy) > thr;
        // t = h sign(d) / (|d| + sqrt(d^2 + h^2)), h = 2 a_xy, c = 1 / sqrt(1 + t^2)
        const float h = 2.f * axy, e = fmaf(d, d, h * h);
        const float t = copysignf(h, __int_as_float(__float_as_int(h) ^ __float_as_int(d))) *
                        rcp_fast(fabsf(d) + e * rsqrt_fast(e));
        const float cc = rsqrt_fast(fmaf(t, t, 1.f));
        c = rot ? cc : 1.f;
        s = rot ? t * cc : 0.f;
      }
      const unsigned mask = __ballot_sync(0xffffffffu, rot);
      x = up(x);
      y = lane == 0 ? m : up(y);
#pragma unroll
      for (int u = 0; u < NI; ++u) {
        xk[u] = up(xk[u]);
        yk[u] = ik[u] == 0 ? m : up(yk[u]);
        xl[u] = up(xl[u]);
        yl[u] = il[u] == 0 ? m : up(yl[u]);
      }
      if (mask == 0u) continue;                    // the same in every warp
      nrot += __popc(mask);
      float* N = sm.A[cur ^ 1];
#pragma unroll
      for (int u = 0; u < NI; ++u) {
        const float ck = __shfl_sync(0xffffffffu, c, ik[u]), sk = __shfl_sync(0xffffffffu, s, ik[u]);
        const float cl = __shfl_sync(0xffffffffu, c, il[u]), sl = __shfl_sync(0xffffffffu, s, il[u]);
        if (kind[u] == 1) {
          const float r00 = ck * b00[u] - sk * b10[u], r01 = ck * b01[u] - sk * b11[u];
          const float r10 = sk * b00[u] + ck * b10[u], r11 = sk * b01[u] + ck * b11[u];
          N[o00[u]] = cl * r00 - sl * r01;
          N[o10[u]] = cl * r10 - sl * r11;         // (a diagonal block keeps one of the two)
          N[o01[u]] = sl * r00 + cl * r01;
          N[o11[u]] = sl * r10 + cl * r11;
        } else if (kind[u] == 2) {
          sm.S[o00[u]] = ck * b00[u] - sk * b01[u];
          sm.S[o01[u]] = sk * b00[u] + ck * b01[u];
        }
      }
      cur ^= 1;
      __syncthreads();
    }
  }
  sweeps = sweep;
  rots = nrot;
}

struct EigArgs {
  int j, ident, ntarget, tmode, nt, ld;
  const double* H;
  double *S, *theta;
  int* order;
  double *Scols, *thcols, *norms;
  int* counters;
  const int* skip;
};

__global__ void __cluster_dims__(EC, 1, 1) __launch_bounds__(ET, 1) k_eig_step(EigArgs g) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  EigSmem& sm = *reinterpret_cast<EigSmem*>(smem_raw);
  cg::cluster_group cl = cg::this_cluster();
  const int cr = (int)cl.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j = g.j, jj = j + (j & 1), ld = g.ld;
  if (cr == 0 && tid < g.nt) g.norms[tid] = 0.0;
  if (*g.skip) return;                             // the same in every CTA, before any barrier
  EigSmem* peer[EC];
#pragma unroll
  for (int r = 0; r < EC; ++r) peer[r] = cl.map_shared_rank(&sm, r);
  const int ncol = cr < j ? (j - cr + EC - 1) / EC : 0;   // this CTA's columns cr, cr + EC, ...
  // ---- H, the previous rotation in FP32, and a power of two that brings H below 1
  unsigned mh = 0;
#pragma unroll 8
  for (int q = tid; q < j * EJ; q += ET) {
    const int r = q % EJ, c = q / EJ;
    if (r < j) {
      const double v = g.H[r + (size_t)c * ld];
      const double w = g.ident ? (r == c ? 1.0 : 0.0) : g.S[r + (size_t)c * ld];
      sm.H[r + c * EL] = v;
      sm.S[r + c * FL] = (float)w;
      mh = max(mh, (unsigned)__double2hiint(v) & 0x7fffffffu);
    }
  }
  mh = __reduce_max_sync(0xffffffffu, mh);
  if (lane == 0) sm.redu[warp] = mh;
  __syncthreads();
  mh = __reduce_max_sync(0xffffffffu, lane < EW ? sm.redu[lane] : 0u);
  const double mx = __hiloint2double((int)mh, 0);                   // max |h_ij|, cut to 20 bits
  const int ex = min(max((int)(mh >> 20) - 1022, -1000), 1000);
  const double down = __hiloint2double((1023 - ex) << 20, 0);       // 2^-ex
  // ---- the FP32 frame A[0] = S^T H S (S in FP32: the refinement starts from what
  // the Jacobi pass makes of it)
  for (int c = warp; c < jj; c += EW)
    for (int r = lane; r < jj; r += 32) {
      const bool in = r < j && c < j;
      if (!in) {
        sm.A[0][r + c * FL] = 0.f;
        sm.S[r + c * FL] = r == c ? 1.f : 0.f;
      } else {
        (g.ident ? sm.A[0] : sm.A[1])[r + c * FL] = (float)(sm.H[r + c * EL] * down);
      }
    }
  if (!g.ident) {
    // by columns, each CTA its own: H S, then S^T (H S)
    float* T = reinterpret_cast<float*>(sm.B);
    __syncthreads();
    for (int i = warp; i < ncol; i += EW)
      for (int r = lane; r < j; r += 32) {
        const float* x = sm.S + (cr + i * EC) * FL;
        float v = 0.f;
#pragma unroll 8
        for (int k = 0; k < j; ++k) v = fmaf(sm.A[1][r + k * FL], x[k], v);
        T[r + i * FL] = v;
      }
    cl.sync();                                     // (and every CTA has started)
    for (int i = warp; i < ncol; i += EW)
      for (int r = lane; r < j; r += 32) {
        float v = 0.f;
#pragma unroll 8
        for (int k = 0; k < j; ++k) v = fmaf(sm.S[k + r * FL], T[k + i * FL], v);
#pragma unroll
        for (int k = 0; k < EC; ++k) peer[k]->A[0][r + (cr + i * EC) * FL] = v;
      }
    cl.sync();
    for (int c = warp; c < jj; c += EW)
      for (int r = lane; r < c; r += 32) {
        const float v = 0.5f * (sm.A[0][r + c * FL] + sm.A[0][c + r * FL]);
        sm.A[0][r + c * FL] = v;
        sm.A[0][c + r * FL] = v;
      }
  }
  __syncthreads();
  float big = 0.f;
  for (int c = warp; c < jj; c += EW)
    for (int r = lane; r < jj; r += 32) big = fmaxf(big, fabsf(sm.A[0][r + c * FL]));
  // (the bits of a non-negative float order as integers)
  const unsigned ub = __reduce_max_sync(0xffffffffu, __float_as_uint(big));
  if (lane == 0) sm.redu[warp] = ub;
  __syncthreads();
  big = __uint_as_float(__reduce_max_sync(0xffffffffu, lane < EW ? sm.redu[lane] : 0u));
  int sweeps = 0, rots = 0;
  const float thr = J_TOL * big;
  const int items = j_items(jj, (jj + EC - 1) / EC);
  if (items <= ET)
    jacobi32<1>(sm, jj, cr, thr, sweeps, rots);
  else if (items <= 2 * ET)
    jacobi32<2>(sm, jj, cr, thr, sweeps, rots);
  else
    jacobi32<J_MOST>(sm, jj, cr, thr, sweeps, rots);
  // ---- X = S J: each CTA's rows to everybody
  if (g.ident) cl.sync();                          // every CTA has started
  __syncthreads();
  for (int r = cr + EC * warp; r < j; r += EC * EW)
    for (int c = lane; c < j; c += 32) {
      const double v = (double)sm.S[r + c * FL];
#pragma unroll
      for (int k = 0; k < EC; ++k) peer[k]->X[0][r + c * EL] = v;
    }
  cl.sync();
  int xb = 0;                                      // the current X
  // ---- refinement
  // What rounding leaves in m.  Between nearly equal eigenvalues it gives angles
  // m / gap of any size that do not shrink from step to step, and each costs its
  // square of the orthogonality: such a pair is left as it is.
  const double noise = 4.0 * 2.220446049250313e-16 * mx;
  bool last = false;                               // this step only makes X orthonormal
  bool stuck = false;                              // the steps ran out
  int step = 0, turned = 0;
  float before = INFINITY;
  while (true) {
    ++step;
    double* X = sm.X[xb];
    // W = H X and G = X^T X, then B = X^T W and lambda, on this CTA's columns
    for (int q = tid; q < 2 * ncol * j; q += ET) {
      const int i2 = q / j, r = q - i2 * j;
      const bool gram = i2 >= ncol;
      const int i = gram ? i2 - ncol : i2;
      // (H is symmetric: its columns serve as its rows)
      const double v = dot_col(gram ? X + r * EL : sm.H + r * EL, 1, X + (cr + i * EC) * EL, j);
      (gram ? sm.Gc : sm.W)[i][r] = v;
    }
    __syncthreads();
    for (int q = tid; q < ncol * j; q += ET) {
      const int i = q / j, r = q - i * j;
      sm.Bc[i][r] = dot_col(X + r * EL, 1, sm.W[i], j);
    }
    __syncthreads();
    if (tid < ncol) {
      const int c = cr + tid * EC;
      const double l = sm.Bc[tid][c] / sm.Gc[tid][c];
#pragma unroll
      for (int k = 0; k < EC; ++k) peer[k]->lam[c] = l;
    }
    cl.sync();
    // the ranking and the targets: the ntarget smallest (tmode 0) or largest (1)
    // lambda, a NaN last; doubles ordered as integers
    if (tid < j) {
      const double l = sm.lam[tid];
      long long k = __double_as_longlong(g.tmode == 0 ? l : -l);
      k ^= (k >> 63) & 0x7fffffffffffffffll;
      if ((__double2hiint(l) & 0x7fffffff) >= 0x7ff00000) k = 0x7fffffffffffffffll;
      sm.key[tid] = k;
    }
    __syncthreads();
    if (tid < j) {
      const long long ki = sm.key[tid];
      int rank = 0;
      for (int t = 0; t < j; ++t) {
        const long long kt = sm.key[t];
        rank += kt < ki || (kt == ki && t < tid);
      }
      sm.rank[tid] = rank;
      sm.tgt[tid] = rank < g.ntarget;
    }
    __syncthreads();
    // E, its largest entry, and whether a target pair has to be rotated.  The
    // owner of column c makes the entries of the pairs (r, c), r < c, and sends
    // E_cr to the owner of column r: m_rc and m_cr differ by rounding, and a
    // rotation part that is not exactly antisymmetric costs X eps ||H|| / gap of
    // its orthogonality (4e-15 at j = 28; basis drift over the restarts)
    float emax = 0.f;
    bool flag = false;
    for (int q = tid; q < ncol * j; q += ET) {
      const int i = q / j, r = q - i * j, c = cr + i * EC;
      if (r > c) continue;
      const double gr = sm.Gc[i][r];
      if (r == c) {
        const double e = 0.5 * (1.0 - gr);
        sm.Ec[i][r] = e;
        emax = fmaxf(emax, fabsf((float)e));
        continue;
      }
      const double lr = sm.lam[r], lc = sm.lam[c];
      const double m = fma(-0.5 * (lr + lc), gr, sm.Bc[i][r]), gap = lc - lr;
      double k = 0.0;
      if (last) {
      } else if (fabs(m) <= E_SMALL * fabs(gap)) {
        if (m != 0.0) {
          // 1 / gap by one Newton step from FP32 (the quotient only has to be
          // good to a share of itself), where FP32 holds the gap and its reciprocal
          const double gs = gap * down;
          if (fabs(gs) > 1e-37) {
            const double y = (double)__frcp_rn((float)gs);
            k = m * down * (y * fma(-gs, y, 2.0));
          } else {
            k = m / gap;
          }
          if (fabs(k) > E_ANGLE && fabs(m) <= noise) k = 0.0;
        }
      } else if ((sm.tgt[r] || sm.tgt[c]) && fabs(m) > noise) {
        flag = true;
      }
      sm.Ec[i][r] = fma(-0.5, gr, k);
      cl.map_shared_rank(&sm, r % EC)->Ec[r / EC][c] = fma(-0.5, gr, -k);
      emax = fmaxf(emax, fmaxf(fabsf((float)k), fabsf((float)gr)));
    }
    emax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(emax)));
    flag = __any_sync(0xffffffffu, flag);
    if (lane == 0) sm.red[warp] = flag ? INFINITY : emax;
    __syncthreads();
    if (tid < EC) {
      float e = 0.f;
      for (int w = 0; w < EW; ++w) e = fmaxf(e, sm.red[w]);
      cl.map_shared_rank(&sm, tid)->wmax[cr] = e;
    }
    cl.sync();                                     // every CTA's columns of E are complete
    // X + X E of this CTA's columns, into everybody's other buffer (not used when
    // a rotation comes first)
    for (int q = tid; q < ncol * j; q += ET) {
      const int i = q / j, r = q - i * j, at = r + (cr + i * EC) * EL;
      const double v = X[at] + dot_col(X + r, EL, sm.Ec[i], j);
#pragma unroll
      for (int k = 0; k < EC; ++k) peer[k]->X[xb ^ 1][at] = v;
    }
    cl.sync();
    float e = 0.f;
#pragma unroll
    for (int k = 0; k < EC; ++k) e = fmaxf(e, sm.wmax[k]);
    if (isinf(e) && turned < 4 && step < E_STEPS) {
      // ---- rotate, the largest |m_ij| first, in every CTA alike
      ++turned;
      for (int q = tid; q < ncol * j; q += ET) {
        const int i = q / j, r = q - i * j, c = cr + i * EC;
        const double gr = sm.Gc[i][r], lr = sm.lam[r], lc = sm.lam[c];
        const double m = r == c ? lc : fma(-0.5 * (lr + lc), gr, sm.Bc[i][r]);
        sm.Ec[i][r] = r == c ? 0.5 * (1.0 - gr) : -0.5 * gr;
#pragma unroll
        for (int k = 0; k < EC; ++k) peer[k]->B[r + c * EL] = m;
      }
      __syncthreads();
      for (int q = tid; q < ncol * j; q += ET) {
        const int i = q / j, r = q - i * j, at = r + (cr + i * EC) * EL;
        const double v = X[at] + dot_col(X + r, EL, sm.Ec[i], j);
#pragma unroll
        for (int k = 0; k < EC; ++k) peer[k]->X[xb ^ 1][at] = v;
      }
      cl.sync();
      xb ^= 1;
      X = sm.X[xb];
      auto coupled = [&](int r, int t, double b, double tau) {
        return b > noise && b > tau * fabs(sm.B[t + t * EL] - sm.B[r + r * EL]);
      };
      // what is coupled to the targets joins them
      while (true) {
        unsigned hits = 0u;                        // bit i: column warp + i EW is coupled to one of them
        for (int t = warp, i = 0; t < j; t += EW, ++i) {
          bool hit = false;
          for (int r = lane; r < j && !sm.tgt[t]; r += 32)
            hit = hit || (sm.tgt[r] && coupled(r, t, fabs(sm.B[r + t * EL]), E_SMALL));
          if (__any_sync(0xffffffffu, hit)) hits |= 1u << i;
        }
        if (!__syncthreads_or(hits != 0u)) break;
        if (lane == 0)
          for (int i = 0; i < EJ / EW; ++i)
            if ((hits >> i) & 1u) sm.tgt[warp + i * EW] = 1;
        __syncthreads();
      }
      for (int n = 0; n < E_MOST; ++n) {
        double best = 0.0;
        int at = -1;
        for (int t = warp; t < j; t += EW) {
          if (!sm.tgt[t]) continue;
          for (int r = lane; r < j; r += 32) {
            const double b = fabs(sm.B[r + t * EL]);
            if (r != t && b > best && coupled(r, t, b, E_ROT)) {
              best = b;
              at = r + t * 64;
            }
          }
        }
        auto larger = [&](double ob, int oa) {
          if (ob > best || (ob == best && oa > at)) {
            best = ob;
            at = oa;
          }
        };
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double ob = __shfl_xor_sync(0xffffffffu, best, o);
          larger(ob, __shfl_xor_sync(0xffffffffu, at, o));
        }
        if (lane == 0) {
          sm.wbest[warp] = best;
          sm.wat[warp] = at;
        }
        __syncthreads();
        if (warp == 0) {
          for (int w = 1; w < EW; ++w) larger(sm.wbest[w], sm.wat[w]);
          if (at >= 0) {
            // the angle in FP32 (what it leaves is refined), c and s orthonormal
            // in FP64: c = x^(-1/2), x = 1 + t^2, by a Halley step
            const int p = min(at & 63, at >> 6), q = max(at & 63, at >> 6);
            const double un = 1.0 / best;
            const float d = (float)fmax(fmin((sm.B[q + q * EL] - sm.B[p + p * EL]) * un, 1e9), -1e9);
            const float h = 2.f * (float)(sm.B[p + q * EL] * un);
            const double t = (double)(copysignf(1.f, d) * h / (fabsf(d) + sqrtf(fmaf(d, d, h * h))));
            const double x = fma(t, t, 1.0), y = (double)rsqrtf((float)x), z = x * (y * y);
            const double c = y * 0.125 * fma(z, fma(z, 3.0, -10.0), 15.0);
            if (lane == 0) {
              sm.rot[0] = c;
              sm.rot[1] = t * c;
            }
          }
          if (lane == 0) sm.sel = at;
        }
        __syncthreads();
        at = sm.sel;
        if (at < 0) break;
        const int p = min(at & 63, at >> 6), q = max(at & 63, at >> 6);
        const double c = sm.rot[0], s = sm.rot[1];
        if (tid < j) {                             // rows p, q of B
          const double x = sm.B[p + tid * EL], y = sm.B[q + tid * EL];
          sm.B[p + tid * EL] = c * x - s * y;
          sm.B[q + tid * EL] = s * x + c * y;
        } else if (tid >= 64 && tid < 64 + j) {    // columns p, q of X
          const int r = tid - 64;
          const double x = X[r + p * EL], y = X[r + q * EL];
          X[r + p * EL] = c * x - s * y;
          X[r + q * EL] = s * x + c * y;
        }
        __syncthreads();
        if (tid < j) {                             // columns p, q of B
          const double x = sm.B[tid + p * EL], y = sm.B[tid + q * EL];
          sm.B[tid + p * EL] = c * x - s * y;
          sm.B[tid + q * EL] = s * x + c * y;
        }
        __syncthreads();
        if (tid == 0) {
          sm.B[p + q * EL] = 0.0;
          sm.B[q + p * EL] = 0.0;
          ++rots;
        }
        __syncthreads();
      }
      cl.sync();
      continue;
    }
    xb ^= 1;
    // done, or on the rounding floor of a pair that is nearly one; what a last large
    // rotation has cost X is mended by one more step
    if (last) break;
    const bool done = !(e > E_DONE) || (e < 1e-7f && e > 0.1f * before);
    if (done || step >= E_STEPS) {
      stuck = !done;
      if (!(e > E_ANGLE)) break;
      last = true;
    }
    before = e;
  }
  // ---- results
  for (int i = warp; i < ncol; i += EW)
    for (int r = lane; r < j; r += 32) g.S[r + (size_t)(cr + i * EC) * ld] = sm.X[xb][r + (cr + i * EC) * EL];
  if (cr == 0) {
    if (tid < j) {
      g.theta[tid] = sm.lam[tid];
      g.order[sm.rank[tid]] = tid;
    }
    for (int c = warp; c < j; c += EW) {
      const int to = sm.rank[c];
      if (to >= g.nt) continue;
      for (int r = lane; r < j; r += 32) g.Scols[r + (size_t)to * ld] = sm.X[xb][r + c * EL];
      if (lane == 0) g.thcols[to] = sm.lam[c];
    }
    if (tid == 0) {
      g.counters[0] = sweeps;
      g.counters[1] = rots;
      g.counters[2] = step;
      g.counters[3] = turned;
      g.counters[4] = stuck;
    }
  }
}

}  // namespace

void eig_step(cudaStream_t s, int j, const double* H, double* S, int ld, bool ident, int ntarget, int tmode, int nt,
              double* theta, int* order, double* Scols, double* thcols, double* norms,
              int* counters, const int* skip) {
  ProfScope ps(s, PROF_JACOBI);
  static std::atomic<uint64_t> done{0};
  once_per_device(done, [&] {
    cudaFuncSetAttribute(k_eig_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(EigSmem));
  });
  EigArgs g{j, ident ? 1 : 0, ntarget, tmode, nt, ld, H, S, theta, order, Scols, thcols, norms, counters, skip};
  k_eig_step<<<EC, ET, sizeof(EigSmem), s>>>(g);
  count_launch();
}

}  // namespace ph
