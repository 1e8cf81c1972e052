// The hopping term of the FP64 Wilson operator in block fixed point on the integer pipes.
//
// What bounds the plain form: an SM issues two FP64 operations per clock and the stencil needs
// about 860 per (site, right-hand side): 430 clocks, 6.6 ms for ten fields of 24^3 x 32, against
// 0.3 ms of HBM traffic.  The same SM issues 32 32 x 32 -> 64-bit integer multiply-adds per clock
// (against 1.7 to 2 DFMA measured), 1824 per site, 57 clocks, so the stencil runs on integers:
//   * fx_convert_kernel turns a field into integers once per application: a real x of a site whose
//     largest real has biased exponent X becomes q = x 2^(1082 - X), |q| < 2^60 (the mantissa
//     shifted by X - exponent; all 53 bits survive down to 2^-7 of the site's largest entry).
//     Converting the half spinor of each direction inside the stencil (tried) costs 96 conversions
//     of 15 instructions per site, and the two FP64 operations of each projection;
//   * links become q_u = u 2^(1082 - X_u), once per call (fx_links_kernel);
//   * spin projections are 64-bit additions; a half spinor is shifted right by E - X_u - X - 1 to the
//     exponent E >= X_u + X + 2 that all eight directions of the thread share, leaving |h| < 2^60;
//   * both factors are split as hi 2^32 + lo with signed lo: a product needs hi hi and
//     (hi lo + lo hi) / 2^32, three mad.wide; lo lo / 2^64, a quarter of the unit that is kept at most, is dropped.  Six
//     products are summed exactly (|hi hi| sum < 2^59, |mixed| sum < 2^63), the mixed sum enters by
//     its high word (one mad.wide), and the eight directions are added as 64-bit integers (< 2^62).
// FP64 arithmetic is left with the last p - kappa acc (24 conversions, 24 DFMA).
// Error: with the exponent of the largest product around the site, the unit kept is 2^-53 to 2^-55 (by the
// mantissas) of largest link entry x largest field entry.  A real of the result has 48 dropped lo lo, at most a
// quarter of it each (12 units; random signs make it about one), 8 roundings of half a unit and the truncated
// inputs.  Measured against extended precision the error is below that of the FP64 chain
// (tests/test_gpu_fxhop.py).
// Sites or links with a NaN, an Inf, or a scale near the ends of the exponent range carry the exponent
// FX_BAD, those with entries far apart FX_WIDE; the threads that meet one run the plain FP64 stencil.
//
// Layout: blocks of 32 sites, [block][component][site of the block] with 16 bytes each (components: the
// 12 of a field; 9 entries of each of the four links), so that a warp reads 512 contiguous bytes and
// one address serves all components; the canonical layout (192 bytes per site) would cost 32 cache
// lines per load.  The canonical side goes through a warp-private shared buffer with 208 bytes per
// site (conflict-free) in memory order.
#pragma once

#include "spin.cuh"

namespace fx {

using spin::Cx;
using spin::mk;

struct Links {
  const int4 *q;   // [site / 32][mu 4][entry 9][site % 32]: (re hi, re lo, im hi, im lo)
  const int *ex;   // [mu 4][site]: biased exponent X_u of the link's largest real, or FX_BAD
};
struct Field {
  longlong2 *q;    // [right-hand side][site / 32][component 12][site % 32]
  int *ex;         // [right-hand side][site]: X, or FX_BAD
};
__host__ __device__ __forceinline__ long long blocks32(long long S) { return (S + 31) >> 5; }
// first component of site s in an array with per components per site
__device__ __forceinline__ long long slot(int s, int per) { return (long long)(s >> 5) * (32 * per) + (s & 31); }
constexpr int FX_BAD = 1 << 20;       // exponent that sends the thread to the FP64 stencil
constexpr int FX_MINX = 64;           // X of a block of zeros (and the least a shift may start from)
constexpr int FX_MIN_FIELD = 400, FX_MIN_LINK = 700;   // smaller non-zero blocks are FX_BAD
// Entries far apart: the integers hold an entry to 2^-60 of its block's largest, where FP64 holds each to its own
// 53 bits.  A block with a non-zero complex entry below 2^-12 of the largest real, or a real below 2^-24, has
// FX_WIDE added to its exponent, and the stencil and the contraction read it in FP64; so do sites whose
// neighbours' products are more than FX_SPREAD binary orders apart.  The lines lie where fields of Gaussian
// entries hardly ever cross them: 3e-6 of the sites, so that one warp in a thousand of the stencil (32 sites and
// their neighbours) takes its FP64 form; at 2^-8 and 2^-16 one in four would.  Sums over a site (fxblas.cu)
// use the integers.
constexpr int FX_WIDE = 1 << 16, FX_ENTRY = 12, FX_REAL = 24, FX_SPREAD = 8;
constexpr int SITE_BYTES = 208;       // 192 + 16: lanes of a quarter warp fall on distinct banks
constexpr int WARP_BYTES = 32 * SITE_BYTES;

__device__ __forceinline__ unsigned long long shr64(unsigned long long a, int n) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));  // shifts above 63 give 0
  return r;
}
__device__ __forceinline__ long long sar64(long long a, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
}
// acc + a b: this form becomes one multiply-add; inline mad.wide.s32 becomes two instructions, and the
// plain C++ product in between
__device__ __forceinline__ long long madw(long long acc, int a, int b) {
  long long p;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
  return acc + p;
}

// mantissa of x left aligned in 64 bits.  Zeros and denormals have exponent field 0, so that a shift
// by base - exponent >= 64 (FX_MINX) takes their (wrong) implicit one out.
__device__ __forceinline__ unsigned long long mantissa(double x) {
  return (((unsigned long long)((__double2hiint(x) & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x)) << 11;
}
__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// for maxima over a block: its exponent field is that of the largest real, and 0 means that all are zero
__device__ __forceinline__ int mag(double x) { return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0); }
// Exponent of a block of complex entries, as it is stored: X [+ FX_WIDE], or FX_BAD
struct Range {
  int mx = 0;                              // largest magnitude word
  unsigned entry = ~0u, real = ~0u;        // smallest of the non-zero entries and reals, minus 1
  __device__ __forceinline__ void add(double2 v) {
    const int a = mag(v.x), b = mag(v.y), m = max(a, b);
    mx = max(mx, m);
    entry = min(entry, (unsigned)m - 1u);
    real = min(real, min((unsigned)a - 1u, (unsigned)b - 1u));
  }
  __device__ __forceinline__ int X() const { return max(mx >> 20, FX_MINX); }
  __device__ __forceinline__ int stored(int least) const {
    const int x = X();
    if (x == 0x7ff || (mx != 0 && x < least)) return FX_BAD;
    const bool wide = mx != 0 && ((int)((entry + 1) >> 20) < x - FX_ENTRY || (int)((real + 1) >> 20) < x - FX_REAL);
    return wide ? x + FX_WIDE : x;
  }
};
// x -> trunc(x 2^(1086 - base)), base = X + 4 for 60 bits
__device__ __forceinline__ long long fixed(double x, int base) {
  const long long s = __double2hiint(x) >> 31;
  return ((long long)shr64(mantissa(x), base - exponent(x)) ^ s) - s;
}
// q = hi 2^32 + lo with lo in [-2^31, 2^31)
__device__ __forceinline__ void split(long long q, int &hi, int &lo) {
  lo = (int)q;
  hi = (int)(q >> 32) + (int)((unsigned)lo >> 31);
}

__device__ __forceinline__ void cp_async16(unsigned sa, const void *g) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(g) : "memory");
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void wait_but() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Warp-private staging of 32 site blocks (12 double2 each): chunk i = lane + 32 j of the 384 belongs to
// site i / 12, component i % 12; 96 chunks are 8 sites, so three (site, component) pairs serve all j.
struct Stage {
  int lane;
  int site[3], comp[3];
  unsigned sm;      // shared address of the warp's buffer
  char *smp;
  __device__ __forceinline__ void init(char *warp_smem) {
    lane = threadIdx.x & 31;
    smp = warp_smem;
    sm = (unsigned)__cvta_generic_to_shared(warp_smem);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int i = lane + 32 * r;
      site[r] = i / 12;
      comp[r] = i - 12 * site[r];
    }
  }
  // copy the 192-byte blocks of the lanes' sites m (each lane names its own) into the buffer
  // (SPLIT = 4: warp part of the four that share the sites copies a quarter)
  template <int SPLIT = 1>
  __device__ __forceinline__ void load(const double2 *src, int m, int part = 0) const {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int j = 0; j < 4 / SPLIT; ++j) {
        const int q = SPLIT == 1 ? j : part;
        const int ms = __shfl_sync(0xffffffffu, m, site[r] + 8 * q);
        cp_async16(sm + (site[r] + 8 * q) * SITE_BYTES + comp[r] * 16,
                   src + (long long)ms * 12 + comp[r]);
      }
    commit();
  }
  // write the blocks of the buffer to the lanes' sites m of dst; lanes with m < 0 write nothing
  template <int SPLIT = 1>
  __device__ __forceinline__ void store(double2 *dst, int m, int part = 0) const {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int j = 0; j < 4 / SPLIT; ++j) {
        const int q = SPLIT == 1 ? j : part;
        const int ms = __shfl_sync(0xffffffffu, m, site[r] + 8 * q);
        if (ms >= 0)
          dst[(long long)ms * 12 + comp[r]] =
              *(const double2 *)(smp + (site[r] + 8 * q) * SITE_BYTES + comp[r] * 16);
      }
  }
  __device__ __forceinline__ double2 *mine() const {
    return (double2 *)(smp + lane * SITE_BYTES);
  }
};

struct Acc {
  long long v[4][3][2];   // [spin][colour][re, im], unit 2^(E - 2101)
  int E;
  bool bad;
};

__device__ __forceinline__ void add2(long long a[2], long long re, long long im) { a[0] += re; a[1] += im; }

// Colour product of one direction d (2 mu: U h of (1 - g) p, 2 mu + 1: U^dag h of (1 + g) p) for the two
// components of a half spinor: q: the field's integers at p, of which the half spinor is shifted by sh; u: the
// links of the site that holds the link; pu, pl: component offsets of the upper and lower spin pair
// (exchanged: -gamma_5 times the field).  With sh = E - X_u - X - 1 the unit of o is 2^(E - 2101).
__device__ __forceinline__ void half_product(int d, const longlong2 *__restrict__ q, int pu, int pl, int sh,
                                             const int4 *__restrict__ u, long long o[2][3][2]) {
  const int mu = d >> 1, bwd = d & 1;
  // half spinor (table at the head of spin.cuh), shifted and split; the t projection is 2 p of one pair
  longlong2 h[2][3];
  if (mu == 3) {
    sh -= 1;
    const longlong2 *p = q + (bwd ? pu : pl);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      h[0][c] = __ldg(p + c * 32);
      h[1][c] = __ldg(p + (3 + c) * 32);
    }
  } else {
    const longlong2 *p = q + pu, *w0 = q + pl + (mu == 2 ? 0 : 96), *w1 = q + pl + (mu == 2 ? 96 : 0);
    longlong2 w[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      h[0][c] = __ldg(p + c * 32);
      h[1][c] = __ldg(p + (3 + c) * 32);
      w[0][c] = __ldg(w0 + c * 32);
      w[1][c] = __ldg(w1 + c * 32);
    }
    // (h0, h1) += phases (i, i), (1, -1), (i, -i) of x, y, z, the negatives backward
    switch (d) {
#define LQCD_FX_CASE(D, X0, Y0, X1, Y1)                                     \
  case D:                                                                   \
    _Pragma("unroll") for (int c = 0; c < 3; ++c) {                         \
      h[0][c].x += X0; h[0][c].y += Y0; h[1][c].x += X1; h[1][c].y += Y1;   \
    }                                                                       \
    break;
      LQCD_FX_CASE(0, -w[0][c].y, w[0][c].x, -w[1][c].y, w[1][c].x)
      LQCD_FX_CASE(1, w[0][c].y, -w[0][c].x, w[1][c].y, -w[1][c].x)
      LQCD_FX_CASE(2, w[0][c].x, w[0][c].y, -w[1][c].x, -w[1][c].y)
      LQCD_FX_CASE(3, -w[0][c].x, -w[0][c].y, w[1][c].x, w[1][c].y)
      LQCD_FX_CASE(4, -w[0][c].y, w[0][c].x, w[1][c].y, -w[1][c].x)
      default:
      LQCD_FX_CASE(5, w[0][c].y, -w[0][c].x, -w[1][c].y, w[1][c].x)
#undef LQCD_FX_CASE
    }
  }
  int hi[2][3][2], lo[2][3][2];
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      split(sar64(h[k][c].x, sh), hi[k][c][0], lo[k][c][0]);
      split(sar64(h[k][c].y, sh), hi[k][c][1], lo[k][c][1]);
    }
  // o_a = sum_b U_ab h_b (forward) or conj(U_ba) h_b (backward)
  const int4 *um = u + mu * 288;
  const int ea = bwd ? 32 : 96, eb = bwd ? 96 : 32, cs = bwd ? -1 : 1;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    long long hh[2][2], md[2][2];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        hh[k][z] = 0;
        md[k][z] = 1ll << 31;   // rounds to the high word
      }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 v = __ldg(um + a * ea + b * eb);
      // (re, im) += (v_re, +-v_im) (h_re, h_im); v is the factor that is negated, since its lo is
      // never -2^31 (fx_links_kernel)
      const int ih = v.z * cs, il = v.w * cs, nh = -ih, nl = -il;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int rh = hi[k][b][0], rl = lo[k][b][0], mh = hi[k][b][1], ml = lo[k][b][1];
        hh[k][0] = madw(hh[k][0], v.x, rh);
        md[k][0] = madw(md[k][0], v.x, rl);
        md[k][0] = madw(md[k][0], v.y, rh);
        hh[k][0] = madw(hh[k][0], nh, mh);
        md[k][0] = madw(md[k][0], nh, ml);
        md[k][0] = madw(md[k][0], nl, mh);
        hh[k][1] = madw(hh[k][1], v.x, mh);
        md[k][1] = madw(md[k][1], v.x, ml);
        md[k][1] = madw(md[k][1], v.y, mh);
        hh[k][1] = madw(hh[k][1], ih, rh);
        md[k][1] = madw(md[k][1], ih, rl);
        md[k][1] = madw(md[k][1], il, rh);
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int z = 0; z < 2; ++z) o[k][a][z] = madw(hh[k][z], (int)(md[k][z] >> 32), 1);
  }
}

// Adds direction d (x + mu, x - mu) to A; arguments as half_product.  d is a run-time value, the same in all
// threads: the loop over the directions stays rolled, since eight unrolled copies (100 kB of
// instructions) missed the instruction cache on one issue in six.
__device__ __forceinline__ void direction(int d, const longlong2 *__restrict__ q, int pu, int pl, int sh,
                                          const int4 *__restrict__ u, Acc &A) {
  long long o[2][3][2];
  half_product(d, q, pu, pl, sh, u, o);
  if (d != 6) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      add2(A.v[0][c], o[0][c][0], o[0][c][1]);
      add2(A.v[1][c], o[1][c][0], o[1][c][1]);
    }
  }
  // the lower pair is the upper one (exchanged for x and y) times the conjugate phases
  switch (d) {
#define LQCD_FX_CASE(D, X2, Y2, X3, Y3)                                                           \
  case D:                                                                                         \
    _Pragma("unroll") for (int c = 0; c < 3; ++c) {                                               \
      const long long *o0 = o[0][c], *o1 = o[1][c];                                               \
      add2(A.v[2][c], X2, Y2);                                                                    \
      add2(A.v[3][c], X3, Y3);                                                                    \
    }                                                                                             \
    break;
    LQCD_FX_CASE(0, o1[1], -o1[0], o0[1], -o0[0])
    LQCD_FX_CASE(1, -o1[1], o1[0], -o0[1], o0[0])
    LQCD_FX_CASE(2, -o1[0], -o1[1], o0[0], o0[1])
    LQCD_FX_CASE(3, o1[0], o1[1], -o0[0], -o0[1])
    LQCD_FX_CASE(4, o0[1], -o0[0], -o1[1], o1[0])
    LQCD_FX_CASE(5, -o0[1], o0[0], o1[1], -o1[0])
    LQCD_FX_CASE(6, o0[0], o0[1], o1[0], o1[1])
#undef LQCD_FX_CASE
    default: break;
  }
}

// A = sum over the directions d0 .. d1 - 1 of the hopping term at link-lattice site s for right-hand side
// r of the field f (S sites), at the exponent E of all eight; with g5 the spins are read exchanged, which is -gamma_5 times the field
// (finish flips the sign).  nbr(d): link-lattice index of the neighbour; COMPACT: the field holds one
// parity (index = neighbour >> 1).
template <bool COMPACT, typename Nbr>
__device__ __forceinline__ void hop(const Field &f, int r, long long S, bool g5, const Links &L, long long VL, int s,
                                    const Nbr &nbr, int d0, int d1, Acc &A) {
  const longlong2 *q = f.q + (long long)r * blocks32(S) * 384;
  const int *ex = f.ex + (long long)r * S;
  A.E = 0;
  int low = 1 << 30;   // the least of the products that are not zero
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const int n = nbr(d);
    const int xf = __ldg(ex + (COMPACT ? n >> 1 : n)), xl = __ldg(L.ex + (d >> 1) * VL + ((d & 1) ? n : s));
    A.E = max(A.E, xf + xl + 2);
    if (xf != FX_MINX && xl != FX_MINX) low = min(low, xf + xl + 2);
  }
  // FX_BAD or FX_WIDE among them, products far apart, or kappa 2^(E - 2101) without room to the end of the range
  A.bad = A.E > 2900 || A.E - low > FX_SPREAD;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) A.v[a][c][0] = A.v[a][c][1] = 0;
  if (__all_sync(0xffffffffu, A.bad)) return;
#pragma unroll 1
  for (int d = d0; d < d1; ++d) {
    const int n = nbr(d), m = COMPACT ? n >> 1 : n, l = (d & 1) ? n : s;
    const int X = __ldg(ex + m) + __ldg(L.ex + (d >> 1) * VL + l);
    direction(d, q + slot(m, 12), g5 ? 192 : 0, g5 ? 0 : 192, A.E - X - 1, L.q + slot(l, 36), A);
  }
}

// acc += direction d of the hopping term in FP64 at link-lattice site s, with the factor -gamma_5 that g5 stands for
template <bool COMPACT, typename Nbr>
__device__ __forceinline__ void direction_fp64(int d, const double2 *U, const double2 *src, long long VL, int s, bool g5,
                                               const Nbr &nbr, Cx<double> acc[4][3]) {
  using namespace spin;
  Cx<double> p[4][3], u[9];
  const int n = nbr(d);
  load_spinor<double, false>(src + 12LL * (COMPACT ? n >> 1 : n), p);
  if (g5) {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Cx<double> v = p[a][c];
        p[a][c] = p[a + 2][c];
        p[a + 2][c] = v;
      }
  }
  load_link<double>(U, (d >> 1) * VL + ((d & 1) ? n : s), u);
  switch (d) {
    case 0: term_fwd<double, 0>(p, u, acc); break;
    case 1: term_bwd<double, 0>(p, u, acc); break;
    case 2: term_fwd<double, 1>(p, u, acc); break;
    case 3: term_bwd<double, 1>(p, u, acc); break;
    case 4: term_fwd<double, 2>(p, u, acc); break;
    case 5: term_bwd<double, 2>(p, u, acc); break;
    case 6: term_fwd<double, 3>(p, u, acc); break;
    default: term_bwd<double, 3>(p, u, acc); break;
  }
}

// The whole sum in FP64
template <bool COMPACT, typename Nbr>
__device__ __forceinline__ void hop_fp64(const double2 *U, const double2 *src, long long VL, int s, bool g5,
                                         const Nbr &nbr, Cx<double> acc[4][3]) {
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[a][c] = mk<double>(0.0, 0.0);
#pragma unroll 1
  for (int d = 0; d < 8; ++d) direction_fp64<COMPACT>(d, U, src, VL, s, g5, nbr, acc);
}

// The same by four warps (run<4>): the upper pairs of directions d0 and d0 + 1 (the lower one of d = 6, whose upper pair
// is zero), 24 reals 32 slots apart, and their sum for spin a in the order of the whole sum, with its bits.
template <bool COMPACT, typename Nbr>
__device__ __noinline__ void halves_fp64(const double2 *U, const double2 *src, long long VL, int s, bool g5, Nbr nbr,
                                         int d0, double *o) {
#pragma unroll 1
  for (int d = d0; d < d0 + 2; ++d, o += 12 * 32) {
    Cx<double> acc[4][3];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[a][c] = mk<double>(0.0, 0.0);
    direction_fp64<COMPACT>(d, U, src, VL, s, g5, nbr, acc);
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Cx<double> v = d == 6 ? acc[2 + k][c] : acc[k][c];
        o[(6 * k + 2 * c) * 32] = v.x;
        o[(6 * k + 2 * c + 1) * 32] = v.y;
      }
  }
}
// (o: stride doubles between the reals)
__device__ __forceinline__ Cx<double> sum_halves(const double *o, int stride, int a, int c) {
  using namespace spin;
  Cx<double> acc = mk<double>(0.0, 0.0);
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    if (a < 2 ? d == 6 : d == 7) continue;
    const int k = a < 2 ? a : (a == 2) == (d < 4) ? 1 : 0;   // x and y exchange the pair
    Cx<double> v = mk<double>(o[(12 * d + 6 * k + 2 * c) * stride], o[(12 * d + 6 * k + 2 * c + 1) * stride]);
    if (a >= 2) {   // conjugate phases of the lower pair: -i, i, (-, +), (+, -), (-i, i), (i, -i)
      if (d == 0 || d == 1 || d == 4 || d == 5) v = ti(v);
      if (d == 0 || d == (a == 2 ? 2 : 3) || d == (a == 2 ? 4 : 5)) v = neg(v);
    }
    acc = acc + v;
  }
  return acc;
}

// Half spinor component k of direction d, multiplied by the link, for one site by one lane, without branches on d:
// lanes of a warp take the 16 (d, k) of a site in turn where a warp has few (FEW) bad ones.  Ordinary fields have a bad
// site in one warp of a thousand, and an FP64 instruction holds the pipe for 16 clocks however many lanes take part: the
// whole sum by one lane was a tail of 20 us at the end of a launch.  Four fields of 12^3 x 24, conversions
// included: M 134.7 us with it, 109.3 so (113.6 with no such sites), the even/odd hop 94.5 and 73.0.  More
// than FEW take a lane per site (10 fields of 24^3 x 32, all sites: 7.26 ms, 6.62 in the plain FP64 kernel before the
// integers).  n: link-lattice index of the neighbour; o as in halves_fp64.
constexpr int FEW = 8;
template <bool COMPACT>
__device__ __noinline__ void half_fp64(const double2 *U, const double2 *src, long long VL, int s, int n, bool g5, int d,
                                       int k, double *o, int stride) {
  using namespace spin;
  const int mu = d >> 1, bwd = d & 1;
  const double2 *p = src + 12LL * (COMPACT ? n >> 1 : n);
  const double2 *u = U + (mu * VL + (bwd ? n : s)) * 9;
  // h = p_a + phase p_b (table at the head of spin.cuh); the t projection is 2 p of one pair
  const int up = g5 ? 2 : 0;   // exchanged spins
  const int a = mu == 3 ? (bwd ? k : 2 + k) : k, b = mu == 3 ? a : mu == 2 ? 2 + k : 3 - k;
  const bool rot = mu == 0 || mu == 2, minus = mu != 3 && ((bwd != 0) != (mu != 0 && k == 1));
  Cx<double> h[3], m[9], r[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const Cx<double> x = load_c<double>(p + 3 * (a ^ up) + c), y = load_c<double>(p + 3 * (b ^ up) + c);
    const Cx<double> t = rot ? ti(y) : y;
    h[c] = minus ? x - t : x + t;
  }
#pragma unroll
  for (int e = 0; e < 3; ++e)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const Cx<double> v = load_c<double>(u + (bwd ? 3 * c + e : 3 * e + c));
      m[3 * e + c] = mk<double>(v.x, bwd ? -v.y : v.y);
    }
  mul_u<double>(m, h, r);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    o[(12 * d + 6 * k + 2 * c) * stride] = r[c].x;
    o[(12 * d + 6 * k + 2 * c + 1) * stride] = r[c].y;
  }
}

// The results of the lanes in bad, self + sc * (the sum in FP64), in the place of self in their blocks of the warp's
// buffer smp (self: 0 none; 1; 2 with gamma_5; left: gamma_5 on the result; as in run); o: 96 reals of the warp
template <bool COMPACT, typename Nbr>
__device__ __noinline__ void sites_fp64(char *smp, double *o, const double2 *U, const double2 *src, long long VL, int s,
                                        bool g5, Nbr nbr, int self, bool left, double sc, unsigned bad) {
  const int lane = threadIdx.x & 31;
  auto get = [&](const double2 *m, int i) {
    const double2 x = m[self == 2 ? (i + 6) % 12 : i];
    return self == 0 ? make_double2(0.0, 0.0) : self == 1 ? x : make_double2(-x.x, -x.y);
  };
  auto put = [&](double2 *m, int i, double2 x, Cx<double> v) {
    const double2 y = make_double2(fma(sc, v.x, x.x), fma(sc, v.y, x.y));
    m[left ? (i + 6) % 12 : i] = left ? make_double2(-y.x, -y.y) : y;
  };
  if (__popc(bad) > FEW) {
    if (!(bad >> lane & 1)) return;
    Cx<double> acc[4][3];
    hop_fp64<COMPACT>(U, src, VL, s, g5, nbr, acc);
    double2 *m = (double2 *)(smp + lane * SITE_BYTES), x[12];
#pragma unroll
    for (int i = 0; i < 12; ++i) x[i] = get(m, i);
#pragma unroll
    for (int i = 0; i < 12; ++i) put(m, i, x[i], acc[i / 3][i % 3]);
    return;
  }
  for (unsigned todo = bad; todo; todo &= todo - 1) {
    const int b = __ffs(todo) - 1, sb = __shfl_sync(0xffffffffu, s, b);
    int n = 0;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const int nb = __shfl_sync(0xffffffffu, nbr(d), b);
      if (d == lane >> 1) n = nb;
    }
    if (lane < 16) half_fp64<COMPACT>(U, src, VL, sb, n, g5, lane >> 1, lane & 1, o, 1);
    __syncwarp();
    double2 *m = (double2 *)(smp + b * SITE_BYTES), x = make_double2(0.0, 0.0);
    if (lane < 12) x = get(m, lane);
    __syncwarp();
    if (lane < 12) put(m, lane, x, sum_halves(o, 1, lane / 3, lane % 3));
    __syncwarp();
  }
}

// Neighbours of a site on a periodic Lx x Ly x Lz x Lt lattice
struct Torus {
  int Lx, Ly, Lz, Lt, x, y, z, t, s;
  __device__ __forceinline__ Torus(int lx, int ly, int lz, int lt, int site) : Lx(lx), Ly(ly), Lz(lz), Lt(lt), s(site) {
    x = s % Lx;
    int q = s / Lx;
    y = q % Ly;
    q /= Ly;
    z = q % Lz;
    t = q / Lz;
  }
  __device__ __forceinline__ int operator()(int d) const {
    switch (d) {
      case 0: return x + 1 == Lx ? s - (Lx - 1) : s + 1;
      case 1: return x == 0 ? s + (Lx - 1) : s - 1;
      case 2: return y + 1 == Ly ? s - (Ly - 1) * Lx : s + Lx;
      case 3: return y == 0 ? s + (Ly - 1) * Lx : s - Lx;
      case 4: return z + 1 == Lz ? s - (Lz - 1) * Lx * Ly : s + Lx * Ly;
      case 5: return z == 0 ? s + (Lz - 1) * Lx * Ly : s - Lx * Ly;
      case 6: return t + 1 == Lt ? s - (Lt - 1) * Lx * Ly * Lz : s + Lx * Ly * Lz;
      default: return t == 0 ? s + (Lt - 1) * Lx * Ly * Lz : s - Lx * Ly * Lz;
    }
  }
};

// Shared bytes of a block of 128 threads in run
template <int SPLIT> constexpr int SMEM_BYTES = SPLIT == 1 ? 4 * (WARP_BYTES + 96 * 8) : WARP_BYTES + 4 * 24 * 32 * 8;

// One application for this thread: out[out_i] = self[self_i] + coef * hopping term (self may be NULL; the
// gamma_5 flags: on the hopping input, on self, on the result).  src: the canonical field f was
// converted from.  A lane with out_i < 0 (its site repeats another's) helps and stores nothing.
// SPLIT = 1: one thread per site.  SPLIT = 4, for fields that leave most of the chip idle: the four
// warps of a block share 32 sites, warp w adds the two directions of mu = w and finishes spin w; the
// sums are integers at one exponent, so both forms give the same bits, and FP64 sites add the directions in one order.
template <int SPLIT, bool COMPACT, typename Nbr>
__device__ __forceinline__ void run(char *smem, const double2 *U, const Links &L, long long VL, int s, const Nbr &nbr,
                                    const Field &f, int r, long long S, const double2 *src, bool g5,
                                    const double2 *self, int self_i, bool self_g5, double coef, bool left_g5,
                                    double2 *out, int out_i) {
  const int warp = threadIdx.x >> 5;
  Stage st;
  st.init(smem + (SPLIT == 1 ? warp * WARP_BYTES : 0));
  if (self) st.load<SPLIT>(self, self_i, warp);
  Acc A;
  hop<COMPACT>(f, r, S, g5, L, VL, s, nbr, SPLIT == 1 ? 0 : 2 * warp, SPLIT == 1 ? 8 : 2 * warp + 2, A);
  // E is above 1100 unless every block was zero (FX_MIN_FIELD, FX_MIN_LINK); the exchanged spins of g5
  // are -gamma_5 times the field
  const double sc = g5 ? -coef : coef;
  const double k = A.E > 1080 ? sc * __hiloint2double((A.E - 2101 + 1023) << 20, 0) : 0.0;
  double2 *m = st.mine();
  if constexpr (SPLIT == 1) {
    wait_all();
    __syncwarp();
    if (!A.bad) {
      double2 p[12];
#pragma unroll
      for (int i = 0; i < 12; ++i)
        p[i] = !self ? make_double2(0.0, 0.0) : self_g5 ? make_double2(-m[(i + 6) % 12].x, -m[(i + 6) % 12].y) : m[i];
#pragma unroll
      for (int i = 0; i < 12; ++i) {
        p[i].x = fma(k, (double)A.v[i / 3][i % 3][0], p[i].x);
        p[i].y = fma(k, (double)A.v[i / 3][i % 3][1], p[i].y);
      }
#pragma unroll
      for (int i = 0; i < 12; ++i) m[i] = left_g5 ? make_double2(-p[(i + 6) % 12].x, -p[(i + 6) % 12].y) : p[i];
    }
    const unsigned bad = __ballot_sync(0xffffffffu, A.bad);
    if (bad)
      sites_fp64<COMPACT>(st.smp, (double *)(smem + 4 * WARP_BYTES) + 96 * warp, U, src, VL, s, g5, nbr,
                          !self ? 0 : self_g5 ? 2 : 1, left_g5, sc, bad);
    __syncwarp();
    st.store<SPLIT>(out, out_i);
  } else {
    long long *red = (long long *)(smem + WARP_BYTES);   // [warp][real 24][lane 32]
    if (!A.bad) {
#pragma unroll
      for (int i = 0; i < 24; ++i) red[(warp * 24 + i) * 32 + st.lane] = A.v[i / 6][i / 2 % 3][i & 1];
    }
    const unsigned bad = __ballot_sync(0xffffffffu, A.bad);   // the same in the four warps, and as with SPLIT = 1
    if (__popc(bad) > FEW) {
      if (A.bad) halves_fp64<COMPACT>(U, src, VL, s, g5, nbr, 2 * warp, (double *)red + warp * 24 * 32 + st.lane);
    } else if (bad) {
      // lane 4 i + j: half spinor j of the warp's four, of the i-th bad site
      unsigned rest = bad;
      for (int i = 0; i < st.lane >> 2; ++i) rest &= rest - 1;
      const int b = rest ? __ffs(rest) - 1 : 0, sb = __shfl_sync(0xffffffffu, s, b), d = 2 * warp + (st.lane >> 1 & 1);
      const int n0 = __shfl_sync(0xffffffffu, nbr(2 * warp), b), n1 = __shfl_sync(0xffffffffu, nbr(2 * warp + 1), b);
      if (rest) half_fp64<COMPACT>(U, src, VL, sb, d & 1 ? n1 : n0, g5, d, st.lane & 1, (double *)red + b, 32);
    }
    wait_all();
    __syncthreads();
    double2 p[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int i = 3 * warp + c;
      p[c] = !self ? make_double2(0.0, 0.0) : self_g5 ? make_double2(-m[(i + 6) % 12].x, -m[(i + 6) % 12].y) : m[i];
      if (!A.bad) {
        long long re = 0, im = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          re += red[(w * 24 + 2 * i) * 32 + st.lane];
          im += red[(w * 24 + 2 * i + 1) * 32 + st.lane];
        }
        p[c] = make_double2(fma(k, (double)re, p[c].x), fma(k, (double)im, p[c].y));
      } else {
        const Cx<double> h = sum_halves((const double *)red + st.lane, 32, warp, c);
        p[c] = make_double2(fma(sc, h.x, p[c].x), fma(sc, h.y, p[c].y));
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int i = 3 * warp + c;
      m[left_g5 ? (i + 6) % 12 : i] = left_g5 ? make_double2(-p[c].x, -p[c].y) : p[c];
    }
    __syncthreads();
    st.store<SPLIT>(out, out_i, warp);
  }
}

// Whether n sites of nrhs right-hand sides take the split form: up to 8 warps per SM of the plain one.  Measured
// on 8^3 x 16 (256 warps a right-hand side, 152 SMs): 12.5 against 21.2 us for one, 24.6 against 27.6 for
// four; eight (37.9 us) are past the line and gain nothing.
inline bool use_split(long long n, int nrhs, int sms) { return blocks32(n) * nrhs <= 8LL * sms; }

}  // namespace fx
