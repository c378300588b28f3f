// FP64 tall-skinny products on the FP16 tensor cores, by exact splitting.
//
// GB300's FP64 pipe takes a warp instruction every 16 clocks per SM (1.25
// TFLOP/s in all), so P^T T and P Y with tall P are bound by it at 5% of the
// memory bandwidth.  Here each operand is scaled by powers of two (per row or
// column of a tile), taken to a 62-bit integer and cut into 8 signed digits of
// 8 bits (Ozaki, Ogita, Oishi, Rump, "Error-free transformations of matrix
// multiplication", Numer. Algorithms 59, 2012; the digits are integers, as in
// the INT8 variants of that scheme, but held in FP16).  The products of two
// digits are exact in FP16 x FP16 -> FP32, and so are their sums: over at most
// 64 terms an accumulator stays within 2^22 (acc_of), and every accumulator
// starts at 1.5 * 2^23, where FP32 counts in ones, so that its bits are the
// integer sum.  Digit pairs (s, t) with s + t <= 7 are kept (36 of 64); the sums
// of all orders are put together as one 64-bit integer and rounded to FP64 once.
//
// Accuracy.  What is cut off is relative to (row maximum) x (column maximum): with
// integers M, N below 2^62, each of K terms loses at most 2 * 2^62 by the cuts of M
// and N and 7.1 * 2^62 by the dropped pairs, the sum 2^67 by its last place, K * 2^65.2
// + 2^67 in all.  A chain of FP64 multiply-adds is relative to the sum of the moduli,
// S = sum |M N|, which may lie far below: P(i,:) = (1e25, 1, 1, ..) times (0, 1, 1, ..).
// The entry points keep to that (ST): one more product per step adds up the moduli of the leading digits (FP16
// accumulators, saturating).  |M| >= 0.498 * 2^56 |leading digit|, so a sum of
// 2^8 proves S >= 2^118 and the error below (K + 4) 2^-52 S; an output that does not
// reach it is computed in FP64 from the tile in shared memory (redo).  What is kept is in
// fact better than the chain: random values with p = 8 to 64: at most 0.5 eps S, mean
// 0.04, against 2.5 and 0.18; with identity-like coefficients, a quarter computed anew,
// at most 1.0 and mean 0.20 against 6.5 and 0.79.
// The solver's own products go without (ST = false): its bases are orthonormal and
// its tolerances are norms, for which (row maximum) x (column maximum) is as good; on the
// localised vectors of a heavy-tailed matrix most outputs would be computed anew (1,000,000 x
// 500,000, 20 largest, FP64: 146 ms and 188 ms).
//
// Why mma.sync: a tile's contraction is 16 x 8 x 64 per digit pair and its
// operands are made in registers by the warp that uses them, so a warp-level
// instruction takes them where they are; staging 8 digit planes of every tile
// in shared memory or TMEM for tcgen05 would cost more than the products.  The
// kernels are bound by the integer pipe that cuts the digits (64 lanes a clock)
// and by the tensor pipe (2.15 clocks per m16n8k16) about equally, at half of
// either's rate: the two take turns within a warp, and 16 warps fit an SM.
//
// Measured on the FP64 pipe and here: Gram-Schmidt pass, 500,000 x 55 against 8,
// subtract and project, 796 us -> 225 us; V Y, 500,000 x 35 to 21, 694 us -> 173 us; to
// 8, 265 us -> 81 us (without the sums of moduli 218, 173 and 74 us).  Where outputs are
// computed anew it takes longer: the pass on log-normal(2) elements 542 us, on elements over 10
// decades 705 us; V Y of such up to 850 us.
//
// A tile with an Inf, a NaN or values below 2^-950 is computed in plain FP64.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace ph {

namespace {

constexpr int NS = 8;                  // digits
constexpr int NACC = 11;               // accumulators of a 16 x 8 tile
constexpr unsigned MAGIC = 0x4B400000u;   // bits of 1.5 * 2^23
constexpr int E_MIN = 64;              // smallest usable scale (zeros must shift out)

__device__ __forceinline__ unsigned shr_clamp(unsigned v, int sh) {
  unsigned r;
  asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(sh));
  return r;
}

// The 62-bit integer x * 2^(1084 - base) (base >= the biased exponent of x),
// plus 0x80 in every byte: byte k minus 128 is then the signed digit of 2^(8k).
__device__ __forceinline__ void fix62(double x, int base, unsigned& wl, unsigned& wh) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int sh = base - (int)((hi >> 20) & 0x7ffu);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned Mh = __funnelshift_l(lo, mh, 9), Ml = lo << 9;
  unsigned l = shr_clamp(__funnelshift_rc(Ml, Mh, sh), max(sh - 32, 0));
  unsigned h = shr_clamp(Mh, sh);
  const unsigned s = (unsigned)((int)hi >> 31);
  l ^= s;
  h ^= s;
  asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, 0x80808080;"
      : "=r"(wl), "=r"(wh)
      : "r"(l), "r"(h), "r"(0x80808080u - s));
}

// FP16 digit pairs of two such integers: d[s] = (digit s of the first, digit s
// of the second), s = 0 the most significant.  0x64 over a byte u is the FP16
// number 1024 + u; 1152 less is the digit.
__device__ __forceinline__ unsigned dig(unsigned v) {
  unsigned r;
  asm("sub.f16x2 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(0x64806480u));
  return r;
}
__device__ __forceinline__ void pack_digits(unsigned l0, unsigned h0, unsigned l1, unsigned h1, unsigned (&d)[NS]) {
  const unsigned c = 0x64646464u;
  const unsigned a = __byte_perm(h0, h1, 0x6273), b = __byte_perm(h0, h1, 0x4051);
  const unsigned e = __byte_perm(l0, l1, 0x6273), f = __byte_perm(l0, l1, 0x4051);
  d[0] = dig(__byte_perm(a, c, 0x4140));
  d[1] = dig(__byte_perm(a, c, 0x4342));
  d[2] = dig(__byte_perm(b, c, 0x4140));
  d[3] = dig(__byte_perm(b, c, 0x4342));
  d[4] = dig(__byte_perm(e, c, 0x4140));
  d[5] = dig(__byte_perm(e, c, 0x4342));
  d[6] = dig(__byte_perm(f, c, 0x4140));
  d[7] = dig(__byte_perm(f, c, 0x4342));
}
__device__ __forceinline__ void digits2(double x0, int base0, double x1, int base1, unsigned (&d)[NS]) {
  unsigned l0, h0, l1, h1;
  fix62(x0, base0, l0, h0);
  fix62(x1, base1, l1, h1);
  pack_digits(l0, h0, l1, h1, d);
}

// The accumulator of the digit pair (s, t): orders s + t = 0..4 have one
// each, 5, 6 and 7 two each.  The leading digit of a 62-bit integer is at most 64 in
// modulus, the others 128: four pairs of these, or five with two leading digits among
// them (order 4), over 64 terms are at most 2^22.
__host__ __device__ constexpr int acc_of(int s, int t) {
  return s + t <= 4 ? s + t : s + t == 5 ? (s < 3 ? 5 : 6) : s + t == 6 ? (s < 4 ? 7 : 8) : (s < 4 ? 9 : 10);
}
constexpr bool acc_fits() {
  for (int k = 0; k < NACC; ++k) {
    int most = 0;
    for (int a = 0; a < NS; ++a)
      for (int b = 0; a + b < NS; ++b)
        if (acc_of(a, b) == k) most += 64 * (a ? 128 : 64) * (b ? 128 : 64);
    if (most > 1 << 22) return false;
  }
  return true;
}
static_assert(acc_fits(), "an accumulator would leave the binade in which FP32 counts in ones");

__device__ __forceinline__ void mma16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct Acc {
  float c[NACC][4];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < NACC; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i) c[k][i] = __uint_as_float(MAGIC);
  }
  // the sum of output i, in units of 2^67 of the integer products: order o
  // has the weight 2^(45 - 8 o), so |sum| < 2^63 for 64 terms
  __device__ __forceinline__ long long sum(int i) const {
    auto bits = [&](int k) { return (int)__float_as_uint(c[k][i]); };
    auto two = [&](int k) { return (unsigned)bits(k) + (unsigned)bits(k + 1) - 2u * MAGIC; };
    const int s5 = (int)two(5), s6 = (int)(two(7) + 4u), s7 = (int)(two(9) + 1024u);
    const int low = (s5 << 5) + (s6 >> 3) + (s7 >> 11);
    // the accumulators' offset, once for all orders (64-bit integers wrap)
    constexpr unsigned long long off = (unsigned long long)MAGIC * ((1ull << 13) + (1ull << 21) + (1ull << 29)) +
                                       (((unsigned long long)(MAGIC * 32u + MAGIC * 8192u)) << 32);
    long long v = (long long)low - (long long)off;
    v += (long long)bits(4) * (1 << 13);
    v += (long long)bits(3) * (1 << 21);
    v += (long long)bits(2) * (1 << 29);
    const unsigned top = (unsigned)bits(1) * 32u + (unsigned)bits(0) * 8192u;
    v += (long long)((unsigned long long)top << 32);
    return v;
  }
};

// k * 2^D in FP64 (one rounding; scalbn's where the result is subnormal or overflows)
__device__ __forceinline__ double times_pow2(long long k, int D) {
  const double v = __ll2double_rn(k);
  const int hi = __double2hiint(v);
  const int ne = ((hi >> 20) & 0x7ff) + D;
  if (k == 0) return 0.0;
  if ((unsigned)(ne - 1) < 2046u) return __hiloint2double(hi + (int)((unsigned)D << 20), __double2loint(v));
  return scalbn(v, D);
}
constexpr int E_OUT = 2101;            // value = sum * 2^(base_a + base_b - E_OUT)

// Sums of the moduli of the leading digits, beside the products (16 x 8, FP16).
struct Mag {
  unsigned c[2];
  __device__ __forceinline__ void clear() { c[0] = c[1] = 0u; }
  __device__ __forceinline__ void add(unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
    constexpr unsigned ABS = 0x7fff7fffu;
    asm("mma.sync.aligned.m16n8k16.row.col.f16.f16.f16.f16 {%0,%1}, {%2,%3,%4,%5}, {%6,%7}, {%0,%1};"
        : "+r"(c[0]), "+r"(c[1])
        : "r"(a0 & ABS), "r"(a1 & ABS), "r"(a2 & ABS), "r"(a3 & ABS), "r"(b0 & ABS), "r"(b1 & ABS));
  }
  // biased exponents of the sums of outputs 2 h and 2 h + 1 (k + 15 for 2^k, 0 for no sum), in halves
  __device__ __forceinline__ unsigned levels(int h) const { return (c[h] >> 10) & 0x001f001fu; }
};
constexpr unsigned MAG_MIN = (8 + 15) * 0x10001u;   // sums of 2^8 and more
// bits 0, 1: a half of v is below that of w
__device__ __forceinline__ unsigned less2(unsigned v, unsigned w) {
  return ((v & 0xffffu) < (w & 0xffffu) ? 1u : 0u) | ((v >> 16) < (w >> 16) ? 2u : 0u);
}
// whether either half of any of the warp's v is below that of its w
__device__ __forceinline__ bool any_less2(unsigned v, unsigned w) {
  return __any_sync(0xffffffffu, __vmaxu2(v, w) != v);
}

// out[i] = sum over k < len of x(a, k) y(b, k) in FP64 for the outputs i of the lane's
// bits in need, a = g + 8 (i / 2), b = 2 t + i % 2 (strides xa, xk, yb, yk).  The warp
// shares the work: as many lanes per output as there are outputs for.  A multiply-add
// holds the SM's FP64 pipe for 16 clocks whatever the lanes in use, so a few outputs take
// a tenth of the tile's FP64 time.  list: 128 bytes of the warp.  Returns how many there are.
__device__ __noinline__ int redo_list(unsigned need, const double* x, int xa, int xk, const double* y, int yb, int yk,
                                      int len, unsigned char* list, double* fix) {
  const int lane = threadIdx.x & 31;
  int at[4], total = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool mine = (need >> i) & 1u;
    const unsigned m = __ballot_sync(0xffffffffu, mine);
    at[i] = total + __popc(m & ((1u << lane) - 1u));
    if (mine) list[at[i]] = (unsigned char)(i * 32 + lane);
    total += __popc(m);
  }
  __syncwarp();
  int sh = 0;                                    // 2^sh lanes per output
  while (sh < 5 && (total << (sh + 1)) <= 32) ++sh;
  for (int base = 0; base < total; base += 32 >> sh) {
    const int j = base + (lane >> sh);
    double v = 0.0;
    if (j < total) {
      const int i = list[j] >> 5, l = list[j] & 31;
      const double* xp = x + ((l >> 2) + 8 * (i >> 1)) * (ptrdiff_t)xa;
      const double* yp = y + (2 * (l & 3) + (i & 1)) * (ptrdiff_t)yb;
#pragma unroll 8
      for (int k = lane & ((1 << sh) - 1); k < len; k += 1 << sh)
        v = fma(xp[k * (ptrdiff_t)xk], yp[k * (ptrdiff_t)yk], v);
    }
    for (int o = (1 << sh) >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k = at[i] - base;
      const double w = __shfl_sync(0xffffffffu, v, (k << sh) & 31);
      if (((need >> i) & 1u) && k >= 0 && k < (32 >> sh)) fix[i] = w;
    }
  }
  __syncwarp();
  return total;
}
__device__ __forceinline__ void redo(unsigned need, const double* x, int xa, int xk, const double* y, int yb, int yk,
                                     int len, unsigned char* list, double (&out)[4]) {
  double fix[4];
  redo_list(need, x, xa, xk, y, yb, yk, len, list, fix);
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if ((need >> i) & 1u) out[i] = fix[i];
}
// V Y where nearly all outputs of 16 x 8 are weak: the digits are wasted, and a warp takes
// its next tiles in plain FP64 before it tries again (elements over 10 decades, 35 columns to
// 21: 803 us, and 998 us without this; with 80 for 112, log-normal(2) elements took 780 for 706).
constexpr int WEAK_MANY = 112, WEAK_SKIP = 7;

__device__ inline int expo(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

__device__ inline void cp16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ inline void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ inline void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Rows [row0, row0 + ROWS) of the cnt columns at src into dst (column stride
// LDS_), zeros past n, by NT threads.
template <int ROWS, int LDS_, int NT>
__device__ inline void load_cols(const double* __restrict__ src, int ld, int cnt, int n, int row0, bool vec,
                                 double* dst, int id) {
  constexpr int SEG = ROWS / 2;
  if (vec && row0 + ROWS <= n) {
    for (int e = id; e < cnt * SEG; e += NT) {
      const int c = e / SEG, sg = e % SEG;
      cp16(dst + c * LDS_ + 2 * sg, src + (size_t)c * ld + row0 + 2 * sg);
    }
  } else {
    for (int e = id; e < cnt * ROWS; e += NT) {
      const int c = e / ROWS, rr = e % ROWS;
      dst[c * LDS_ + rr] = row0 + rr < n ? src[(size_t)c * ld + row0 + rr] : 0.0;
    }
  }
}

// Scales of the basis columns, as exponents relative to the largest (<= 0).
// Set 0 is flat: an element's digits then count from the largest of its row,
// which is 9 bits finer than FP64 where the columns are of one size, but coarse
// for a column far below the others.  Set 1 scales each column by its largest
// element in the CTA's first tiles (in shared memory, so no row that another
// CTA may be writing is read).  That is a guess: a tile whose rows it would
// cost more than SCALE_LOSS bits takes set 0.  Set 1 is not made when the
// columns are within a factor of 4.
constexpr int SCALE_LOSS = 6;
struct Scales {
  int b[2][64];          // exponent of each column
  int F[2][64];          // largest exponent of each column of the coefficients, scaled
  int seen[64];
  int bmin, slack, bad, two;
  int peak[64], peaks;   // V Y: the one coefficient of a column that is kept out of the digits, or -1
  double ypeak[64];
};

// seen[c] = largest exponent of column c among 16 rows of a tile, by a warp
template <int LDS_>
__device__ inline void see_columns(const double* tile, int p, Scales& sc, int lane) {
  for (int c = lane >> 4; c < p + (p & 1); c += 2) {
    int e = c < p ? expo(tile[c * LDS_ + (lane & 15)]) : 0;
    if (e == 0x7ff) e = 0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    if ((lane & 15) == 0 && e > 0) atomicMax(&sc.seen[c], e);
  }
}
__device__ inline void set_scales(int p, Scales& sc, int warp, int lane) {
  if (warp == 0) {
    int mx = 0;
    for (int c = lane; c < p; c += 32) mx = max(mx, sc.seen[c]);
    mx = __reduce_max_sync(0xffffffffu, mx);
    int mn = 0;
    for (int c = lane; c < 64; c += 32) {
      int b = c < p && sc.seen[c] > 0 ? max(sc.seen[c] - mx, -512) : 0;
      sc.b[0][c] = 0;
      sc.b[1][c] = b;
      mn = min(mn, b);
    }
    mn = __reduce_min_sync(0xffffffffu, mn);
    if (lane == 0) {
      sc.bmin = mn;
      sc.two = mn < -2;
      sc.slack = 4096;
      sc.bad = 0;
      sc.peaks = 0;
    }
  }
  __syncthreads();
}

// Scales F of the r coefficient columns (padded to rc), for both sets.  Coefficients of
// restarts and Ritz vectors are often a unit matrix with small entries beside it: the window
// of a column would hang on the one large coefficient, and whatever is small in P there be
// weak.  With PEAK a coefficient 8 times the others of its column stays out of the digits:
// its product is one FP64 multiply-add, and the window that of the others (500,000 rows, 35
// columns to 21, I + 1e-3 noise: 191 us for 415).
// sc.bad is set when a coefficient is not finite or a column is too small to be
// cut, sc.two is cleared when set 1 cannot hold the coefficients.
template <int NT, bool PEAK>
__device__ inline void coeff_scales(const double* __restrict__ Y, int ldy, int p, int r, int rc, Scales& sc, int tid) {
  const int warp = tid >> 5, lane = tid & 31;
  for (int c = warp; c < rc; c += NT / 32) {
    int f0 = 0, f1 = -4096, inf = 0, nz = 0, peak = -1;
    double y[2];                                 // (p <= 64)
#pragma unroll
    for (int u = 0; u < 2; ++u) y[u] = lane + 32 * u < p && c < r ? Y[lane + 32 * u + (size_t)c * ldy] : 0.0;
    if (PEAK && c < r) {
      // the lane's larger and smaller, by their high words
      const unsigned ma = (unsigned)__double2hiint(y[0]) & 0x7fffffffu;
      const unsigned mb = (unsigned)__double2hiint(y[1]) & 0x7fffffffu;
      const unsigned m0 = max(ma, mb), m1 = min(ma, mb);
      const unsigned top = __reduce_max_sync(0xffffffffu, m0);
      const int at = __ffs(__ballot_sync(0xffffffffu, m0 == top)) - 1;
      const unsigned next = __reduce_max_sync(0xffffffffu, lane == at ? m1 : m0);
      peak = __shfl_sync(0xffffffffu, mb > ma ? lane + 32 : lane, at);
      if (top < next + (3u << 20)) peak = -1;
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int k = lane + 32 * u, e = expo(y[u]);
      inf |= e == 0x7ff;
      if (y[u] == 0.0 || k == peak) continue;
      nz = 1;
      f0 = max(f0, e);
      f1 = max(f1, e + sc.b[1][k]);
    }
    f0 = __reduce_max_sync(0xffffffffu, f0);
    f1 = __reduce_max_sync(0xffffffffu, f1);
    inf = __any_sync(0xffffffffu, inf);
    nz = __any_sync(0xffffffffu, nz);
    const double ypeak = __shfl_sync(0xffffffffu, peak >= 32 ? y[1] : y[0], peak & 31);
    if (lane == 0) {
      if (inf || (nz && f0 < E_MIN)) sc.bad = 1;
      if (nz) {
        if (f1 < E_MIN) sc.two = 0;
        atomicMin(&sc.slack, f0 - f1);
      }
      sc.peak[c] = peak;
      if (peak >= 0) {
        sc.peaks = 1;
        sc.ypeak[c] = ypeak;
      }
      sc.F[0][c] = max(f0, E_MIN);
      sc.F[1][c] = max(f1, E_MIN);
    }
  }
  __syncthreads();
}

// Digits of the coefficients Y(k, c), k = k0, k0 + 4, k0 + 8, k0 + 12: the k
// of a lane in a step of 16 (the A and B fragments use the same order).
__device__ inline void coeff_lane(const double* __restrict__ Y, int ldy, int p, int r, int c, int k0,
                                  const Scales& sc, int set, unsigned (&d0)[NS], unsigned (&d1)[NS]) {
  double y[4];
  int b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int k = k0 + 4 * u;
    y[u] = (k < p && c < r && k != sc.peak[c]) ? Y[k + (size_t)c * ldy] : 0.0;
    b[u] = sc.F[set][c] - sc.b[set][k];
  }
  digits2(y[0], b[0], y[1], b[1], d0);
  digits2(y[2], b[2], y[3], b[3], d1);
}

// As B fragments (8 columns): Bs[(set * NS + s) * KT + kt][lane].
template <int KT, int NT>
__device__ inline void coeff_frag_b(const double* __restrict__ Y, int ldy, int p, int r, const Scales& sc, uint2* Bs,
                                    int tid) {
  for (int e = tid; e < KT * 32 * (sc.two ? 2 : 1); e += NT) {
    const int set = e / (KT * 32), kt = (e >> 5) % KT, ln = e & 31;
    unsigned d0[NS], d1[NS];
    coeff_lane(Y, ldy, p, r, ln >> 2, kt * 16 + (ln & 3), sc, set, d0, d1);
#pragma unroll
    for (int s = 0; s < NS; ++s) Bs[((set * NS + s) * KT + kt) * 32 + ln] = make_uint2(d0[s], d1[s]);
  }
  __syncthreads();
}
// As A fragments (16 columns per tile): As[((set * mt + tile) * KT + kt) * NS + s][lane].
template <int KT, int NT>
__device__ inline void coeff_frag_a(const double* __restrict__ Y, int ldy, int p, int r, int mt, const Scales& sc,
                                    uint4* As, int tid) {
  for (int e = tid; e < KT * mt * 32 * (sc.two ? 2 : 1); e += NT) {
    const int ln = e & 31, kt = (e >> 5) % KT, tile = (e >> 5) / KT % mt, set = (e >> 5) / KT / mt;
    unsigned d0[NS], d1[NS], d2[NS], d3[NS];
    coeff_lane(Y, ldy, p, r, tile * 16 + (ln >> 2), kt * 16 + (ln & 3), sc, set, d0, d2);
    coeff_lane(Y, ldy, p, r, tile * 16 + 8 + (ln >> 2), kt * 16 + (ln & 3), sc, set, d1, d3);
#pragma unroll
    for (int s = 0; s < NS; ++s)
      As[(((set * mt + tile) * KT + kt) * NS + s) * 32 + ln] = make_uint4(d0[s], d1[s], d2[s], d3[s]);
  }
  __syncthreads();
}

// Scales of NR rows of a tile (rows g + 8 v of the lane, columns 4k + t): the
// largest exponent, less the columns' scales of the set that is taken.
// Returns the set, or -1 when a row cannot be cut (for the whole warp alike).
template <int KT, int LDS_, int NR>
__device__ __forceinline__ int row_scales(const double* tile, const Scales& sc, int g, int t, int (&base)[NR]) {
  bool ok = true, small = false, zero[NR];
#pragma unroll
  for (int v = 0; v < NR; ++v) {
    unsigned m = 0;
#pragma unroll
    for (int k = 0; k < KT * 4; ++k)
      m = max(m, (unsigned)__double2hiint(tile[(k * 4 + t) * LDS_ + g + 8 * v]) & 0x7fffffffu);
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    base[v] = (int)(m >> 20);
    ok = ok && base[v] != 0x7ff;
    zero[v] = base[v] < E_MIN;                   // a row that passes below E_MIN is zero
    small = small || zero[v];
  }
  if (__any_sync(0xffffffffu, small)) {
#pragma unroll
    for (int v = 0; v < NR; ++v) {
      if (base[v] < E_MIN)
        for (int k = 0; k < KT * 4; ++k) ok = ok && tile[(k * 4 + t) * LDS_ + g + 8 * v] == 0.0;
      base[v] = max(base[v], E_MIN);
    }
  }
  if (!__all_sync(0xffffffffu, ok)) return -1;
  if (!sc.two) return 0;
  const int most = sc.slack + SCALE_LOSS;
  int w[NR];
  bool fits = true;
#pragma unroll
  for (int v = 0; v < NR; ++v) {
    int m = E_MIN - sc.bmin;
    for (int k = 0; k < KT * 4; ++k) m = max(m, expo(tile[(k * 4 + t) * LDS_ + g + 8 * v]) - sc.b[1][k * 4 + t]);
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
    m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
    w[v] = m;
    fits = fits && (zero[v] || m - base[v] <= most);
  }
  if (!__all_sync(0xffffffffu, fits)) return 0;
#pragma unroll
  for (int v = 0; v < NR; ++v) base[v] = w[v];
  return 1;
}

// Digits of row g of the tile, columns kt * 16 + t + {0, 4} and {8, 12}
template <int LDS_>
__device__ __forceinline__ void row_digits(const double* tile, const int* b, int kt, int g, int t, int base,
                                           unsigned (&d0)[NS], unsigned (&d1)[NS]) {
  const int c = kt * 16 + t;
  digits2(tile[c * LDS_ + g], base + b[c], tile[(c + 4) * LDS_ + g], base + b[c + 4], d0);
  digits2(tile[(c + 8) * LDS_ + g], base + b[c + 8], tile[(c + 12) * LDS_ + g], base + b[c + 12], d1);
}

// acc = the 16 x 8 products of 16 rows of a tile with 8 coefficient columns
template <int KT, int LDS_, bool ST>
__device__ __forceinline__ void rows_times_coeff(const double* tile, const Scales& sc, int set, const uint2* Bs, int g,
                                                 int t, int lane, const int (&base)[2], Acc& acc, Mag& mag) {
  acc.clear();
  mag.clear();
#pragma unroll 1
  for (int kt = 0; kt < KT; ++kt) {
    unsigned a[NS][4];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      unsigned d0[NS], d1[NS];
      row_digits<LDS_>(tile, sc.b[set], kt, g + 8 * v, t, base[v], d0, d1);
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        a[s][v] = d0[s];
        a[s][2 + v] = d1[s];
      }
    }
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      const uint2 b = Bs[((set * NS + q) * KT + kt) * 32 + lane];
      if (ST && q == 0) mag.add(a[0][0], a[0][1], a[0][2], a[0][3], b.x, b.y);
#pragma unroll
      for (int s = 0; s + q < NS; ++s) mma16(acc.c[acc_of(s, q)], a[s], b.x, b.y);
    }
  }
}
// Levels that make outputs 2 h, 2 h + 1 pass where they do not exist (columns 2 t, 2 t + 1 from q on).
__device__ __forceinline__ unsigned no_cols(int t, int q) {
  return (2 * t < q ? 0u : 31u) | (2 * t + 1 < q ? 0u : 31u << 16);
}
constexpr unsigned NO_ROW = 0x001f001fu;

// Whether the product of the kept-out coefficient y with x alone is large enough for the digits of
// the others, as a sum of moduli of 2^118 would be (their unit is 2^(base + F - 2168)).
__device__ __forceinline__ bool peak_holds(double x, double y, int base, int F) {
  return expo(x) + expo(y) + 4 >= base + F;
}

// ---------------------------------------------------------------------------
// Out = P Y [- Xs diag(theta)], optional column norms.  A warp takes 16-row
// tiles (loaded by cp.async; it reads a tile's rows before it writes them, so
// Out may be P).  With up to 8 output columns the rows are the 16 rows of the
// products (k_tall_rows): each step's digits are used once.  With more, the
// output columns are (k_tall_cols), 16 at a time, and 8 rows are the columns:
// the digits of those rows stay in registers for all output columns (half as
// many as for 16 rows, so that 16 warps fit an SM), and those of the
// coefficients come from shared memory.
// ---------------------------------------------------------------------------
constexpr int TS_R = 16, TS_LD = 20;   // rows of a tile; its column stride in shared memory (no bank conflicts)
// warps per CTA (the digits of 64 basis columns take more registers and shared memory)
__host__ __device__ constexpr int tall_warps(int KT) { return KT == 4 ? 12 : 16; }

struct TallSmem {
  size_t tiles, norms, total;
  TallSmem(int KT, int r, bool with_norms) {
    const int mt = (r + 15) / 16, W = tall_warps(KT);
    tiles = r <= 8 ? 2 * sizeof(uint2) * NS * KT * 32 : 2 * sizeof(uint4) * NS * KT * mt * 32;
    norms = tiles + sizeof(double) * W * KT * 16 * TS_LD;
    total = norms + (with_norms && r > 8 ? sizeof(double) * W * 64 * mt : 0);
  }
};

// A 16-row tile in plain FP64: lane = row and half of the columns;
// add_norm(c, v) is called by one lane per column.
template <typename F>
__device__ __noinline__ void tall_plain(const double* tile, int row0, int n, int p, const double* __restrict__ Y,
                                        int ldy, int r, double* Out, int ldo, const double* __restrict__ Xs, int ldx,
                                        const double* __restrict__ theta, int lane, F add_norm) {
  const int rr = lane & 15, i = row0 + rr;
  for (int c0 = 0; c0 < r; c0 += 2) {
    const int c = c0 + (lane >> 4);
    double o = 0.0;
    if (c < r && i < n) {
      for (int k = 0; k < p; ++k) o = fma(tile[k * TS_LD + rr], Y[k + (size_t)c * ldy], o);
      if (theta) o = fma(-theta[c], Xs[(size_t)c * ldx + i], o);
      Out[(size_t)c * ldo + i] = o;
    }
    double v = o * o;
#pragma unroll
    for (int q = 8; q > 0; q >>= 1) v += __shfl_xor_sync(0xffffffffu, v, q);
    if (c < r && rr == 0) add_norm(c, v);
    __syncwarp();
  }
}

// A CTA's first tiles, the scales of the columns and of the coefficients.
template <int KT, bool ST>
__device__ inline void tall_start(int n, const double* P, int ldp, int p, const double* __restrict__ Y, int ldy, int r,
                                  int rc, bool vec, double* buf, int tile, int ntiles, Scales& sc, int tid) {
  const int warp = tid >> 5, lane = tid & 31;
  for (int e = lane; e < KT * 16 * TS_LD; e += 32) buf[e] = 0.0;   // the columns past p stay zero
  if (tid < 64) sc.seen[tid] = 0;
  __syncthreads();
  if (tile < ntiles) load_cols<TS_R, TS_LD, 32>(P, ldp, p, n, tile * TS_R, vec, buf, lane);
  cp_commit();
  cp_wait<0>();
  __syncwarp();
  if (tile < ntiles) see_columns<TS_LD>(buf, p, sc, lane);
  __syncthreads();
  set_scales(p, sc, warp, lane);
  coeff_scales<tall_warps(KT) * 32, ST>(Y, ldy, p, r, rc, sc, tid);
}

template <int KT, bool ST>
__global__ void __launch_bounds__(tall_warps(KT) * 32, 1)
    k_tall_rows(int n, const double* P, int ldp, int p, const double* __restrict__ Y, int ldy, int r, double* Out,
                int ldo, const double* __restrict__ Xs, int ldx, const double* __restrict__ theta, double* norms2,
                bool vec, size_t off_tiles, RedWs rw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TS_W = tall_warps(KT);
  __shared__ Scales sc;
  __shared__ double wn[TS_W][8];
  __shared__ double part[8];
  __shared__ unsigned char list[TS_W][128];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  uint2* Bs = reinterpret_cast<uint2*>(smem_raw);
  double* buf = reinterpret_cast<double*>(smem_raw + off_tiles) + (size_t)warp * KT * 16 * TS_LD;
  const int ntiles = (n + TS_R - 1) / TS_R, stride = gridDim.x * TS_W;
  int tile = warp * gridDim.x + blockIdx.x;      // the first wave spreads over all CTAs
  if (lane < 8) wn[warp][lane] = 0.0;
  tall_start<KT, ST>(n, P, ldp, p, Y, ldy, r, 8, vec, buf, tile, ntiles, sc, tid);
  coeff_frag_b<KT, TS_W * 32>(Y, ldy, p, r, sc, Bs, tid);
  const bool plain = sc.bad != 0;
  const int c0 = 2 * t;
  int skip = 0;                                  // tiles to take in plain FP64
  const unsigned pad = no_cols(t, r);
  double sq[2] = {0.0, 0.0}, th[2] = {0.0, 0.0};
  if (theta)
    for (int u = 0; u < 2; ++u) th[u] = c0 + u < r ? theta[c0 + u] : 0.0;
  for (; tile < ntiles; tile += stride) {
    const int row0 = tile * TS_R, i0 = row0 + g, next = tile + stride;
    int base[2];
    const int set = row_scales<KT, TS_LD, 2>(buf, sc, g, t, base);
    if (set < 0 || plain || skip > 0) {
      --skip;
      tall_plain(buf, row0, n, p, Y, ldy, r, Out, ldo, Xs, ldx, theta, lane,
                 [&](int c, double v) { wn[warp][c] += v; });
      __syncwarp();
      if (next < ntiles) load_cols<TS_R, TS_LD, 32>(P, ldp, p, n, next * TS_R, vec, buf, lane);
      cp_commit();
    } else {
      double xs[4] = {0.0, 0.0, 0.0, 0.0};
      if (theta) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int c = c0 + (q & 1), i = i0 + (q < 2 ? 0 : 8);
          if (c < r && i < n) xs[q] = Xs[(size_t)c * ldx + i];
        }
      }
      Acc acc;
      Mag mag;
      rows_times_coeff<KT, TS_LD, ST>(buf, sc, set, Bs, g, t, lane, base, acc, mag);
      const unsigned l0 = mag.levels(0) | pad | (i0 < n ? 0u : NO_ROW);
      const unsigned l1 = mag.levels(1) | pad | (i0 + 8 < n ? 0u : NO_ROW);
      // what the kept-out coefficient of output q's column multiplies
      auto x_of = [&](int q) { return buf[sc.peak[c0 + (q & 1)] * TS_LD + g + (q < 2 ? 0 : 8)]; };
      auto finish = [&](int q, double o) {
        const int c = c0 + (q & 1), i = i0 + (q < 2 ? 0 : 8);
        if (theta) o = fma(-th[q & 1], xs[q], o);
        if (c < r && i < n) {
          Out[(size_t)c * ldo + i] = o;
          if (norms2) sq[q & 1] = fma(o, o, sq[q & 1]);
        }
      };
      unsigned need = 0u;
      if (ST && any_less2(__vminu2(l0, l1), MAG_MIN)) {
        need = less2(l0, MAG_MIN) | less2(l1, MAG_MIN) << 2;
        if (sc.peaks) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int c = c0 + (q & 1);
            if (sc.peak[c] >= 0 && peak_holds(x_of(q), sc.ypeak[c], base[q < 2 ? 0 : 1], sc.F[set][c]))
              need &= ~(1u << q);
          }
        }
        if (__any_sync(0xffffffffu, need)) {
          double fix[4];
          if (redo_list(need, buf, 1, TS_LD, Y, ldy, 1, p, list[warp], fix) > WEAK_MANY) skip = WEAK_SKIP;
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if ((need >> q) & 1u) finish(q, fix[q]);
        }
      }
      auto reload = [&] {
        __syncwarp();                            // every lane is done with the tile
        if (next < ntiles) load_cols<TS_R, TS_LD, 32>(P, ldp, p, n, next * TS_R, vec, buf, lane);
        cp_commit();
      };
      if (!ST || !sc.peaks) reload();                   // beside the sums (81 us; after them 87)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = c0 + (q & 1);
        double o = times_pow2(acc.sum(q), base[q < 2 ? 0 : 1] + sc.F[set][c] - E_OUT);
        if (ST && sc.peaks && sc.peak[c] >= 0) o = fma(x_of(q), sc.ypeak[c], o);
        if (!((need >> q) & 1u)) finish(q, o);
      }
      if (ST && sc.peaks) reload();
    }
    cp_wait<0>();
    __syncwarp();
  }
  if (norms2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int o = 4; o <= 16; o <<= 1) sq[u] += __shfl_xor_sync(0xffffffffu, sq[u], o);
      if (g == 0) wn[warp][c0 + u] += sq[u];
    }
    __syncthreads();
    if (tid < r) {
      double v = 0.0;
      for (int w = 0; w < TS_W; ++w) v += wn[w][tid];
      part[tid] = v;
    }
    __syncthreads();
    ordered_commit(part, r, norms2, 0, nullptr, rw);
  }
}

template <int KT, bool ST>
__global__ void __launch_bounds__(tall_warps(KT) * 32, 1)
    k_tall_cols(int n, const double* P, int ldp, int p, const double* __restrict__ Y, int ldy, int r, double* Out,
                int ldo, const double* __restrict__ Xs, int ldx, const double* __restrict__ theta, double* norms2,
                bool vec, bool vec_out, size_t off_tiles, size_t off_norms, RedWs rw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int TS_W = tall_warps(KT);
  __shared__ Scales sc;
  __shared__ double part[64];
  __shared__ unsigned char list[TS_W][128];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int mt = (r + 15) / 16;
  uint4* As = reinterpret_cast<uint4*>(smem_raw);
  double* buf = reinterpret_cast<double*>(smem_raw + off_tiles) + (size_t)warp * KT * 16 * TS_LD;
  double* slot = reinterpret_cast<double*>(smem_raw + off_norms) + (size_t)warp * mt * 64;   // [mt][lane][2]
  const int ntiles = (n + TS_R - 1) / TS_R, stride = gridDim.x * TS_W;
  int tile = warp * gridDim.x + blockIdx.x;
  if (norms2)
    for (int e = lane; e < mt * 64; e += 32) slot[e] = 0.0;
  tall_start<KT, ST>(n, P, ldp, p, Y, ldy, r, mt * 16, vec, buf, tile, ntiles, sc, tid);
  coeff_frag_a<KT, TS_W * 32>(Y, ldy, p, r, mt, sc, As, tid);
  const bool plain = sc.bad != 0;
  int skip = 0;
  for (; tile < ntiles; tile += stride) {
    const int row0 = tile * TS_R, next = tile + stride;
    int base[2];
    const int set = row_scales<KT, TS_LD, 2>(buf, sc, g, t, base);
    if (set < 0 || plain || skip > 0) {
      --skip;
      tall_plain(buf, row0, n, p, Y, ldy, r, Out, ldo, Xs, ldx, theta, lane, [&](int c, double v) {
        if (norms2) slot[(c >> 4) * 64 + (c & 7) * 8 + ((c >> 3) & 1)] += v;
      });
    } else {
      const int* F = sc.F[set];
      unsigned weak = 0u;                        // 4 bits per half of the rows and 16 columns
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        unsigned b[KT][NS][2];
        const int bh = h ? base[1] : base[0];
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
          unsigned d0[NS], d1[NS];
          row_digits<TS_LD>(buf + 8 * h, sc.b[set], kt, g, t, bh, d0, d1);
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            b[kt][s][0] = d0[s];
            b[kt][s][1] = d1[s];
          }
        }
        // scales of the output rows 2t, 2t + 1
        const int e0 = __shfl_sync(0xffffffffu, bh, 8 * t), e1 = __shfl_sync(0xffffffffu, bh, 8 * t + 4);
        const int i = row0 + 8 * h + 2 * t;
#pragma unroll 1
        for (int j = 0; j < mt; ++j) {
          const uint4* as = As + (size_t)(set * mt + j) * KT * NS * 32 + lane;
          Acc acc;
          Mag mag;
          acc.clear();
          mag.clear();
#pragma unroll
          for (int kt = 0; kt < KT; ++kt)
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              const uint4 v = as[(kt * NS + s) * 32];
              const unsigned a[4] = {v.x, v.y, v.z, v.w};
              if (ST && s == 0) mag.add(v.x, v.y, v.z, v.w, b[kt][0][0], b[kt][0][1]);
#pragma unroll
              for (int q = 0; s + q < NS; ++q) mma16(acc.c[acc_of(s, q)], a, b[kt][q][0], b[kt][q][1]);
            }
          const unsigned pad = no_cols(t, n - row0 - 8 * h);   // (here the rows run along t)
          const unsigned l0 = mag.levels(0) | pad | (j * 16 + g < r ? 0u : NO_ROW);
          const unsigned l1 = mag.levels(1) | pad | (j * 16 + g + 8 < r ? 0u : NO_ROW);
          unsigned need = 0u;
          if (ST && any_less2(__vminu2(l0, l1), MAG_MIN)) {
            need = less2(l0, MAG_MIN) | less2(l1, MAG_MIN) << 2;
            if (sc.peaks) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int c = j * 16 + g + 8 * (q >> 1), k = sc.peak[c];
                if (k >= 0 && peak_holds(buf[k * TS_LD + 8 * h + 2 * t + (q & 1)], sc.ypeak[c], q & 1 ? e1 : e0, F[c]))
                  need &= ~(1u << q);
              }
            }
            weak |= need << (16 * h + 4 * j);
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int c = j * 16 + g + 8 * u;
            double o0 = times_pow2(acc.sum(2 * u), e0 + F[c] - E_OUT);
            double o1 = times_pow2(acc.sum(2 * u + 1), e1 + F[c] - E_OUT);
            if (ST && sc.peaks && sc.peak[c] >= 0) {
              const double* x = buf + sc.peak[c] * TS_LD + 8 * h + 2 * t;
              o0 = fma(x[0], sc.ypeak[c], o0);
              o1 = fma(x[1], sc.ypeak[c], o1);
            }
            if (c < r && i < n) {
              if (theta) {
                const double th = theta[c];
                o0 = fma(-th, Xs[(size_t)c * ldx + i], o0);
                if (i + 1 < n) o1 = fma(-th, Xs[(size_t)c * ldx + i + 1], o1);
              }
              double* o = Out + (size_t)c * ldo + i;
              const unsigned w = (need >> (2 * u)) & 3u;   // the weak ones of the two are left out
              if (i + 1 >= n) o1 = 0.0;
              if (w == 0u && i + 1 < n && vec_out) {
                *reinterpret_cast<double2*>(o) = make_double2(o0, o1);
              } else {
                if (!(w & 1u)) o[0] = o0;
                if (!(w & 2u) && i + 1 < n) o[1] = o1;
              }
              if (w & 1u) o0 = 0.0;
              if (w & 2u) o1 = 0.0;
              if (norms2) slot[j * 64 + lane * 2 + u] += fma(o0, o0, o1 * o1);
            }
          }
        }
      }
      if (ST && __any_sync(0xffffffffu, weak)) {
        int most = 0;
        for (int h = 0; h < 2; ++h)
          for (int j = 0; j < mt; ++j) {
            const unsigned need = (weak >> (16 * h + 4 * j)) & 15u;
            if (!__any_sync(0xffffffffu, need)) continue;
            double fix[4];
            most = max(most, redo_list(need, Y + (size_t)j * 16 * ldy, ldy, 1, buf + 8 * h, 1, TS_LD, p, list[warp],
                                       fix));
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              if (!((need >> q) & 1u)) continue;
              const int c = j * 16 + g + 8 * (q >> 1), i = row0 + 8 * h + 2 * t + (q & 1);
              double o = fix[q];
              if (theta) o = fma(-theta[c], Xs[(size_t)c * ldx + i], o);
              Out[(size_t)c * ldo + i] = o;
              if (norms2) slot[j * 64 + lane * 2 + (q >> 1)] += o * o;
            }
          }
        if (most > WEAK_MANY) skip = WEAK_SKIP;
      }
    }
    __syncwarp();                                // every lane is done with the tile
    if (next < ntiles) load_cols<TS_R, TS_LD, 32>(P, ldp, p, n, next * TS_R, vec, buf, lane);
    cp_commit();
    cp_wait<0>();
    __syncwarp();
  }
  if (norms2) {
    __syncthreads();
    const double* slots = reinterpret_cast<double*>(smem_raw + off_norms);
    for (int c = tid; c < r; c += TS_W * 32) {
      double v = 0.0;
      for (int w = 0; w < TS_W; ++w)
        for (int q = 0; q < 4; ++q) v += slots[(size_t)w * mt * 64 + (c >> 4) * 64 + ((c & 7) * 4 + q) * 2 + ((c >> 3) & 1)];
      part[c] = v;
    }
    __syncthreads();
    ordered_commit(part, r, norms2, 0, nullptr, rw);
  }
}

// ---------------------------------------------------------------------------
// Block Gram-Schmidt pass: T <- T - P Gsub, Gout += P^T T, Tout += T^T T.  A CTA
// takes 128-row tiles (two CTAs per SM: one loads while the other computes):
//  * each of its 8 warps updates 16 rows of T with the digits of Gsub;
//  * each cuts its 16 rows of the updated T once, for all warps (the scale of
//    a column is that of its chunk of rows);
//  * then the rows are the contraction: the tile is cut into 16 basis columns x
//    a chunk of rows per warp (KT column groups x CH chunks).
// A tile's products are summed in FP64 over the tiles, the chunks and the CTAs,
// in a fixed order.
// ---------------------------------------------------------------------------
constexpr int CS_R = 128, CS_LD = 132, CS_W = 8;

// Largest exponent over a chunk's RC rows of a column (lane t holds rows t + 4u),
// at least E_MIN; ok is cleared when the column cannot be cut.
template <int RC>
__device__ __forceinline__ int col_scale(const double* col, int t, bool& ok) {
  unsigned m = 0;
#pragma unroll
  for (int u = 0; u < RC / 4; ++u) m = max(m, (unsigned)__double2hiint(col[t + 4 * u]) & 0x7fffffffu);
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
  int e = (int)(m >> 20);
  if (e == 0x7ff) ok = false;
  if (e < E_MIN) {
    for (int u = 0; u < RC / 4; ++u) ok = ok && col[t + 4 * u] == 0.0;
    e = E_MIN;
  }
  return e;
}

// For a pair of outputs (halves) of a chunk with the scales e and the levels l of its sums of
// moduli: top = the larger of it and e + l.  The chunk's digits will do where e + MAG_MIN <= top: they are
// then off by no more than the chain against the largest sum so far.  (A CTA takes a second
// tile only when there are more than 2 x 152, so that the errors of its chunks, each within (K + 4)
// 2^-52 of that sum, stay within n / 64 + 64 such parts of all.)
__device__ __forceinline__ unsigned raise(unsigned e, unsigned l, unsigned& top) {
  top = __vmaxu2(top, e + l);
  return e + MAG_MIN;
}

template <int KT, bool ST>
__global__ void __launch_bounds__(CS_W * 32, 2)
    k_cgs_split(int n, Basis<double> P, double* __restrict__ Tb, int ldt, int q, const double* __restrict__ Gsub,
                double* __restrict__ Gout, double* __restrict__ Tout, bool vec, bool vect, RedWs rw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int CH = KT >= 3 ? 2 : KT == 2 ? 4 : 8, RC = CS_R / CH, KS = RC / 16;   // chunks of RC rows, KS steps each
  __shared__ Scales sc;
  __shared__ int te[CH][8], tok[CH];
  __shared__ unsigned char list[CS_W][128];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int p = P.cols();
  uint2* Bs = reinterpret_cast<uint2*>(smem_raw);                    // Gsub, both sets of scales
  uint2* Td = Bs + 2 * NS * KT * 32;                                  // digits of T: [16-row step][s][lane]
  double* Ps = reinterpret_cast<double*>(Td + CS_W * NS * 32);        // [KT * 16][CS_LD]
  double* Ts = Ps + KT * 16 * CS_LD;                                  // [8][CS_LD]
  for (int e = tid; e < (KT * 16 + 8) * CS_LD; e += CS_W * 32) Ps[e] = 0.0;   // columns past p and q stay zero
  if (tid < 64) sc.seen[tid] = 0;
  __syncthreads();
  const int ntiles = (n + CS_R - 1) / CS_R;
  double gacc[4] = {0.0, 0.0, 0.0, 0.0}, tacc[2] = {0.0, 0.0};
  // level of the largest sum of moduli among the chunks so far, two outputs to a register:
  // a chunk that lies wholly below it needs no better than the digits give
  unsigned gtop[2] = {0u, 0u}, ttop = 0u;
  const unsigned pad = no_cols(t, q);
  const int ch = warp / KT, m = warp % KT;       // this warp's chunk and columns of P^T T (none when ch >= CH)
  const int tch = KT == 3 ? (warp >= 6 ? warp - 6 : -1) : (m == 0 ? ch : -1);   // its chunk of T^T T
  bool first = true;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int row0 = tile * CS_R;
    if (P.c1) load_cols<CS_R, CS_LD, CS_W * 32>(P.p1, P.ld1, P.c1, n, row0, vec, Ps, tid);
    if (P.c2) load_cols<CS_R, CS_LD, CS_W * 32>(P.p2, P.ld2, P.c2, n, row0, vec, Ps + P.c1 * CS_LD, tid);
    load_cols<CS_R, CS_LD, CS_W * 32>(Tb, ldt, q, n, row0, vect, Ts, tid);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    if (first && Gsub) {
      see_columns<CS_LD>(Ps + 16 * warp, p, sc, lane);
      __syncthreads();
      set_scales(p, sc, warp, lane);
      coeff_scales<CS_W * 32, false>(Gsub, p, p, q, 8, sc, tid);
      coeff_frag_b<KT, CS_W * 32>(Gsub, p, p, q, sc, Bs, tid);
    }
    first = false;
    // ---- T <- T - P Gsub
    if (Gsub) {
      const double* cur = Ps + 16 * warp;
      double* tw = Ts + 16 * warp;
      int base[2];
      const int set = row_scales<KT, CS_LD, 2>(cur, sc, g, t, base);
      if (set < 0 || sc.bad) {
        for (int e = lane; e < 16 * q; e += 32) {
          const int rr = e & 15, c = e >> 4;
          double v = tw[c * CS_LD + rr];
          for (int k = 0; k < p; ++k) v = fma(-cur[k * CS_LD + rr], Gsub[k + (size_t)c * p], v);
          tw[c * CS_LD + rr] = v;
        }
      } else {
        Acc acc;
        Mag mag;
        rows_times_coeff<KT, CS_LD, ST>(cur, sc, set, Bs, g, t, lane, base, acc, mag);
        const int i0 = row0 + 16 * warp + g;       // (rows past n are zero)
        const unsigned l0 = mag.levels(0) | pad | (i0 < n ? 0u : NO_ROW);
        const unsigned l1 = mag.levels(1) | pad | (i0 + 8 < n ? 0u : NO_ROW);
        double out[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          out[i] = times_pow2(acc.sum(i), base[i < 2 ? 0 : 1] + sc.F[set][2 * t + (i & 1)] - E_OUT);
        if (ST && any_less2(__vminu2(l0, l1), MAG_MIN)) {
          unsigned need = less2(l0, MAG_MIN) | less2(l1, MAG_MIN) << 2;
          // the digits' error, below 2^5 of the sum's last place, is no matter where it is below
          // half an ulp of T (their last place is 2^(base + F - E_OUT))
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 2 * t + (i & 1);
            if (expo(tw[c * CS_LD + g + (i < 2 ? 0 : 8)]) >= base[i < 2 ? 0 : 1] + sc.F[set][c] - E_OUT + 5 + 1023 + 53)
              need &= ~(1u << i);
          }
          if (__any_sync(0xffffffffu, need)) redo(need, cur, 1, CS_LD, Gsub, p, 1, p, list[warp], out);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) tw[(2 * t + (i & 1)) * CS_LD + g + (i < 2 ? 0 : 8)] -= out[i];
      }
      __syncwarp();
      for (int e = lane; e < q * 16; e += 32) {
        const int c = e >> 4, i = row0 + 16 * warp + (e & 15);
        if (i < n) Tb[(size_t)c * ldt + i] = tw[c * CS_LD + (e & 15)];
      }
    }
    // ---- P^T T and T^T T
    if (Gout || Tout) {
      __syncthreads();
      {
        const int mych = warp / KS;              // the chunk that holds this warp's 16 rows
        bool ok = true;
        const int e = col_scale<RC>(Ts + g * CS_LD + mych * RC, t, ok);
        ok = __all_sync(0xffffffffu, ok);
        if (t == 0) te[mych][g] = e;
        if (lane == 0) tok[mych] = ok;           // the same value from every warp of the chunk
        const double* x = Ts + g * CS_LD + 16 * warp + t;
        unsigned d0[NS], d1[NS];
        digits2(x[0], e, x[4], e, d0);
        digits2(x[8], e, x[12], e, d1);
#pragma unroll
        for (int s = 0; s < NS; ++s) Td[(warp * NS + s) * 32 + lane] = make_uint2(d0[s], d1[s]);
      }
      __syncthreads();
      if (Gout && ch < CH) {
        const double* x0 = Ps + (16 * m + g) * CS_LD + ch * RC;
        bool ok = tok[ch] != 0;
        const int e0 = col_scale<RC>(x0, t, ok), e1 = col_scale<RC>(x0 + 8 * CS_LD, t, ok);
        if (__all_sync(0xffffffffu, ok)) {
          Acc acc;
          Mag mag;
          acc.clear();
          mag.clear();
#pragma unroll 1
          for (int ks = 0; ks < KS; ++ks) {
            unsigned a[NS][4];
#pragma unroll
            for (int v = 0; v < 2; ++v) {
              const double* x = x0 + 8 * v * CS_LD + 16 * ks + t;
              const int e = v ? e1 : e0;
              unsigned d0[NS], d1[NS];
              digits2(x[0], e, x[4], e, d0);
              digits2(x[8], e, x[12], e, d1);
#pragma unroll
              for (int s = 0; s < NS; ++s) {
                a[s][v] = d0[s];
                a[s][2 + v] = d1[s];
              }
            }
#pragma unroll
            for (int k = 0; k < NS; ++k) {
              const uint2 b = Td[((ch * KS + ks) * NS + k) * 32 + lane];
              if (ST && k == 0) mag.add(a[0][0], a[0][1], a[0][2], a[0][3], b.x, b.y);
#pragma unroll
              for (int s = 0; s + k < NS; ++s) mma16(acc.c[acc_of(s, k)], a[s], b.x, b.y);
            }
          }
          const int s0 = te[ch][2 * t], s1 = te[ch][2 * t + 1];
          const unsigned s01 = (unsigned)s0 | (unsigned)s1 << 16;
          const unsigned l0 = mag.levels(0) | pad | (16 * m + g < p ? 0u : NO_ROW);
          const unsigned l1 = mag.levels(1) | pad | (16 * m + g + 8 < p ? 0u : NO_ROW);
          const unsigned w0 = raise(e0 * 0x10001u + s01, l0, gtop[0]), w1 = raise(e1 * 0x10001u + s01, l1, gtop[1]);
          double out[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            out[i] = times_pow2(acc.sum(i), (i < 2 ? e0 : e1) + (i & 1 ? s1 : s0) - E_OUT);
          if (ST && (any_less2(gtop[0], w0) || any_less2(gtop[1], w1)) && row0 + ch * RC < n)   // (zero past n)
            redo(less2(gtop[0], w0) | less2(gtop[1], w1) << 2, Ps + 16 * m * CS_LD + ch * RC, CS_LD, 1, Ts + ch * RC,
                 CS_LD, 1, RC, list[warp], out);
#pragma unroll
          for (int i = 0; i < 4; ++i) gacc[i] += out[i];
        } else {
#pragma unroll 1
          for (int i = 0; i < 4; ++i) {
            const double* x = x0 + (i < 2 ? 0 : 8 * CS_LD);
            const double* y = Ts + (2 * t + (i & 1)) * CS_LD + ch * RC;
            double v = 0.0;
            for (int rr = 0; rr < RC; ++rr) v = fma(x[rr], y[rr], v);
            if (i == 0) gacc[0] += v;
            if (i == 1) gacc[1] += v;
            if (i == 2) gacc[2] += v;
            if (i == 3) gacc[3] += v;
          }
        }
      }
      if (Tout && tch >= 0 && tch < CH) {
        if (tok[tch]) {
          Acc acc;
          Mag mag;
          acc.clear();
          mag.clear();
#pragma unroll 1
          for (int ks = 0; ks < KS; ++ks) {
            uint2 b[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) b[s] = Td[((tch * KS + ks) * NS + s) * 32 + lane];
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              const unsigned a[4] = {b[s].x, 0u, b[s].y, 0u};
              if (ST && s == 0) mag.add(b[0].x, 0u, b[0].y, 0u, b[0].x, b[0].y);
#pragma unroll
              for (int k = 0; s + k < NS; ++k) mma16(acc.c[acc_of(s, k)], a, b[k].x, b[k].y);
            }
          }
          const int e = te[tch][g], s0 = e + te[tch][2 * t], s1 = e + te[tch][2 * t + 1];
          const unsigned l0 = mag.levels(0) | pad | (g < q ? 0u : NO_ROW);
          const unsigned w = raise((unsigned)s0 | (unsigned)s1 << 16, l0, ttop);
          double out[4] = {times_pow2(acc.sum(0), s0 - E_OUT), times_pow2(acc.sum(1), s1 - E_OUT), 0.0, 0.0};
          if (ST && any_less2(ttop, w) && row0 + tch * RC < n)
            redo(less2(ttop, w), Ts + tch * RC, CS_LD, 1, Ts + tch * RC, CS_LD, 1, RC, list[warp], out);
          tacc[0] += out[0];
          tacc[1] += out[1];
        } else {
          for (int i = 0; i < 2; ++i) {
            const double *x = Ts + g * CS_LD + tch * RC, *y = Ts + (2 * t + i) * CS_LD + tch * RC;
            double v = 0.0;
            for (int rr = 0; rr < RC; ++rr) v = fma(x[rr], y[rr], v);
            if (i == 0) tacc[0] += v; else tacc[1] += v;
          }
        }
      }
    }
    __syncthreads();                             // every warp is done with the tile
  }
  // ---- over the chunks (fixed order), then over the CTAs
  const int n1 = Gout ? p * q : 0, n2 = Tout ? q * q : 0;
  if (n1 + n2 == 0) return;
  double* gr = Ps;                               // [CH][KT * 16][8], then [CH][8][8], then the sums
  double* tr = gr + CH * KT * 128;
  double* part = tr + CH * 64;
  if (ch < CH)
#pragma unroll
    for (int i = 0; i < 4; ++i) gr[(ch * KT * 16 + 16 * m + g + (i < 2 ? 0 : 8)) * 8 + 2 * t + (i & 1)] = gacc[i];
  if (tch >= 0 && tch < CH) {
    tr[tch * 64 + g * 8 + 2 * t] = tacc[0];
    tr[tch * 64 + g * 8 + 2 * t + 1] = tacc[1];
  }
  __syncthreads();
  for (int o = tid; o < n1 + n2; o += CS_W * 32) {
    double v = 0.0;
    if (o < n1) {
      for (int c = 0; c < CH; ++c) v += gr[(c * KT * 16 + o % p) * 8 + o / p];
    } else {
      const int a = (o - n1) % q, b = (o - n1) / q;
      for (int c = 0; c < CH; ++c) v += tr[c * 64 + min(a, b) * 8 + max(a, b)];   // exactly symmetric
    }
    part[o] = v;
  }
  __syncthreads();
  ordered_commit(part, n1, Gout, n2, Tout, rw);
}

int split_sms() {
  int dev = 0, v = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
  return v > 0 ? v : 152;
}
bool even16(const double* p, int ld) { return p == nullptr || (((uintptr_t)p & 15) == 0 && ld % 2 == 0); }
constexpr size_t SPLIT_SMEM = 220 * 1024;

template <int KT, bool ST>
void tall_go(cudaStream_t s, int n, const double* P, int ldp, int p, const double* Y, int ldy, int r, double* Out,
             int ldo, const double* Xs, int ldx, const double* theta, double* norms2) {
  const TallSmem sm(KT, r, norms2 != nullptr);
  static std::atomic<uint64_t> done{0};
  once_per_device(done, [&] {
    cudaFuncSetAttribute(k_tall_rows<KT, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SPLIT_SMEM);
    cudaFuncSetAttribute(k_tall_cols<KT, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SPLIT_SMEM);
  });
  const int grid = std::min(split_sms(), ceil_div(n, TS_R));
  const RedWs rw = norms2 ? red_ws((size_t)grid * r) : RedWs{};
  if (r <= 8)
    k_tall_rows<KT, ST><<<grid, tall_warps(KT) * 32, sm.total, s>>>(n, P, ldp, p, Y, ldy, r, Out, ldo, Xs, ldx, theta,
                                                                    norms2, even16(P, ldp), sm.tiles, rw);
  else
    k_tall_cols<KT, ST><<<grid, tall_warps(KT) * 32, sm.total, s>>>(n, P, ldp, p, Y, ldy, r, Out, ldo, Xs, ldx, theta,
                                                                    norms2, even16(P, ldp), even16(Out, ldo), sm.tiles,
                                                                    sm.norms, rw);
  count_launch();
  if (norms2) reduce_partials(s, rw, grid, r, norms2, 0, nullptr);
}

template <int KT, bool ST>
void cgs_go(cudaStream_t s, int n, const Basis<double>& P, double* Tb, int ldt, int q, const double* Gsub,
            double* Gout, double* Tout) {
  constexpr size_t smem = sizeof(uint2) * NS * 32 * (2 * KT + CS_W) + sizeof(double) * (KT * 16 + 8) * CS_LD;
  static std::atomic<uint64_t> done{0};
  once_per_device(done, [&] {
    cudaFuncSetAttribute(k_cgs_split<KT, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  const int grid = std::min(2 * split_sms(), ceil_div(n, CS_R));
  const int n1 = Gout ? P.cols() * q : 0, n2 = Tout ? q * q : 0;
  const RedWs rw = red_ws((size_t)grid * (n1 + n2));
  k_cgs_split<KT, ST><<<grid, CS_W * 32, smem, s>>>(n, P, Tb, ldt, q, Gsub, Gout, Tout,
                                                even16(P.p1, P.ld1) && even16(P.p2, P.ld2), even16(Tb, ldt), rw);
  count_launch();
  reduce_partials(s, rw, grid, n1, Gout, n2, Tout);
}

}  // namespace

// The lines between the forms, from both sides' times (us, FP64 pipe / here):
// V Y with 3 columns and more wins from the smallest sizes on (n = 600: p = 8,
// r = 3: 9.1 / 7.2; p = 35, r = 21: 50 / 17; n = 500,000, p = 10, r = 3: 76 / 42),
// one and two columns are nearer to their FP64 work in the streaming form.
bool tall_split(cudaStream_t s, int n, const double* P, int ldp, int p, const double* Y, int ldy, int r, double* Out,
                int ldo, const double* Xs, int ldx, const double* theta, double* norms2, bool strict) {
  const int KT = (p + 15) / 16;
  if (n < 512 || n > INT32_MAX - 256 || r < 3 || p < 8 || p > 64 || r > 64 ||
      TallSmem(KT, r, norms2 != nullptr).total > SPLIT_SMEM)
    return false;
  auto go = [&](auto kt) {
    (strict ? tall_go<kt(), true> : tall_go<kt(), false>)(s, n, P, ldp, p, Y, ldy, r, Out, ldo, Xs, ldx, theta, norms2);
  };
  switch (KT) {
    case 1: go(std::integral_constant<int, 1>()); break;
    case 2: go(std::integral_constant<int, 2>()); break;
    case 3: go(std::integral_constant<int, 3>()); break;
    default: go(std::integral_constant<int, 4>()); break;
  }
  return true;
}

// A pass costs the same for 1 to 8 columns here, and twice as much for 8 as for 4
// on the FP64 pipe: 5 columns and more win from the smallest sizes on (n = 600,
// p = 10, q = 8: 14.0 / 11.7), 3 and 4 with enough rows and basis columns
// (p = 35, q = 3: n = 4096: 14.7 / 16.7, n = 16,384: 25 / 19, n = 500,000:
// 267 / 195; p = 10, q = 3, n = 500,000: 86 / 101).
bool cgs_split(cudaStream_t s, int n, const Basis<double>& P, double* Tb, int ldt, int q, const double* Gsub,
               double* Gout, double* Tout, bool strict) {
  const int p = P.cols();
  if (n < (q >= 5 ? 512 : 8192) || n > INT32_MAX - 256 || q < 3 || p < (q >= 5 ? 10 : 16) || p > 64 ||
      !(Gsub || Gout))
    return false;
  auto go = [&](auto kt) {
    (strict ? cgs_go<kt(), true> : cgs_go<kt(), false>)(s, n, P, Tb, ldt, q, Gsub, Gout, Tout);
  };
  switch ((p + 15) / 16) {
    case 1: go(std::integral_constant<int, 1>()); break;
    case 2: go(std::integral_constant<int, 2>()); break;
    case 3: go(std::integral_constant<int, 3>()); break;
    default: go(std::integral_constant<int, 4>()); break;
  }
  return true;
}

}  // namespace ph
