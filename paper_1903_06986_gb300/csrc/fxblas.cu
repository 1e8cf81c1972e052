// Gram-Schmidt of the FP64 Krylov cycles on the integer form of the basis (fxhop.cuh).
//
// What bounds the plain kernels (blas.cu): four DFMA per complex element and basis vector, two per clock
// and SM: 2 clocks an element, where HBM delivers one (16 bytes) in 0.69 and L2 in less.  The operator
// has every basis vector in block fixed point already (60-bit integers, one exponent per site), so the
// solver keeps those and the inner products and updates read them: twelve 32 x 32 -> 64-bit
// multiply-adds an element (0.38 clocks) with no conversion, and both kernels become memory bound.
//
// Inner products: the 12 components of a site are summed exactly as integers at the exponent X_V + X_w of
// the site (w is converted once per group of vectors), then added to an FP64 sum per thread: four FP64
// operations per site instead of 48.  The unit kept is 2^-54 to 2^-56 (by the mantissas) of
// the product of the largest entries; a real has 24 dropped low products of at most a quarter unit (6 units; about
// one half with random signs), where the FP64 chain rounds 24 times.
// Updates: sum_i V_i h_i of a site is one integer per real, at an exponent that all vectors of the sum
// share (found in a first pass over the exponents alone); V_i is shifted to it.  The unit kept is 2^-53 to
// 2^-55 of the largest |V_i h_i| of the site, coarser where 64 and more vectors of that size need room (the exponent
// of the sum grows with log2 of their number less 6); two low products of at most a quarter unit are dropped per
// vector, and one FP64 multiply-add per real ends the sum, where the FP64 chain rounds 2 nvec times.
// Sites with an entry that the integers cannot hold (FX_BAD, products near the ends of the exponent range)
// and non-finite coefficients take the FP64 sums, from the FP64 basis beside the integers.
#include <algorithm>

#include "common.cuh"
#include "fxhop.cuh"

namespace {

using namespace fx;

constexpr int FB = 128;      // threads per block
constexpr int FG = 8;        // basis vectors per block of the inner products
constexpr int X_LOW = 1100, X_HIGH = 2900;   // sums of two exponents that give normal FP64 scales

__device__ __forceinline__ double pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// h[i * nrhs + r] = <V_i^r, w^r>: block (chunk c, group g, right-hand side r), one thread per site and
// step; last-block sums in a fixed order as in multidot_kernel.  A warp copies the 6 KB of its 32 sites of
// the next two vectors into its ring of three shared stages (cp.async) while it multiplies the current
// one: two blocks per SM keep about 100 KB of loads in flight whatever the registers hold (loads straight
// to registers reached 3.0 TB/s on 50 right-hand sides of 8^3 x 16, this 4.1, the FP64 sums 1.0).
constexpr int DRING = 3, DSTAGE = 32 * 12 * 16;
constexpr int DOT_SMEM = FB / 32 * (WARP_BYTES + DRING * DSTAGE);
__global__ void __launch_bounds__(FB, 2) fx_multidot_kernel(Field f, const double2 *__restrict__ V,
                                                            const double2 *__restrict__ w, int S, int nvec, int nrhs,
                                                            int nchunk, double2 *__restrict__ partial,
                                                            unsigned *__restrict__ counters, double2 *__restrict__ h) {
  extern __shared__ __align__(16) char dyn[];
  __shared__ double red[FB / 32][2 * FG];
  __shared__ bool last;
  const int c = blockIdx.x % nchunk;
  const int ngroup = (nvec + FG - 1) / FG;
  const int g0 = (blockIdx.x / nchunk) % ngroup, r = blockIdx.x / (nchunk * ngroup);
  const int i0 = g0 * FG, ng = min(FG, nvec - i0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long fq = blocks32(S) * 384;
  const double2 *wr = w + (long long)r * S * 12;
  Stage st;
  st.init(dyn + warp * WARP_BYTES);
  char *ring = dyn + FB / 32 * WARP_BYTES + warp * DRING * DSTAGE;
  const unsigned ring_sm = (unsigned)__cvta_generic_to_shared(ring) + lane * 16;
  double acc[2 * FG];
#pragma unroll
  for (int j = 0; j < 2 * FG; ++j) acc[j] = 0.0;
  // whole warps of 32 sites: warp strips strided by the chunks, so that neighbours read neighbours
  for (int b = c * (FB / 32) + warp; b < (S + 31) / 32; b += nchunk * (FB / 32)) {
    const int s0 = b * 32 + lane, s = min(s0, S - 1);
    auto issue = [&](int j) {
      if (j < ng) {
        const longlong2 *q = f.q + ((long long)(i0 + j) * nrhs + r) * fq + (long long)b * 384 + lane;
#pragma unroll
        for (int e = 0; e < 12; ++e) cp_async16(ring_sm + (j % DRING) * DSTAGE + e * 512, q + e * 32);
      }
      commit();
    };
    __syncwarp();
    st.load(wr, s);
    issue(0);
    issue(1);
    wait_but<2>();
    __syncwarp();
    const double2 *m = st.mine();
    int mx = 0;
#pragma unroll
    for (int e = 0; e < 12; ++e) mx = max(mx, max(mag(m[e].x), mag(m[e].y)));
    const int Xw = mx >> 20;
    const bool held = Xw >= FX_MINX && Xw < 0x7ff;   // the integers of w are its values
    int wh[12][2], wl[12][2];
#pragma unroll
    for (int e = 0; e < 12; ++e) {
      split(fixed(m[e].x, 4 + Xw), wh[e][0], wl[e][0]);
      split(fixed(m[e].y, 4 + Xw), wh[e][1], wl[e][1]);
    }
#pragma unroll
    for (int j = 0; j < FG; ++j) {
      if (j >= ng) break;
      issue(j + 2);
      const long long fld = (long long)(i0 + j) * nrhs + r;
      const int xv = __ldg(f.ex + fld * S + s) & ~FX_WIDE, X = xv + Xw;
      wait_but<2>();
      __syncwarp();
      const longlong2 *q = (const longlong2 *)(ring + (j % DRING) * DSTAGE) + lane;
      long long re = 0, im = 0;
#pragma unroll
      for (int e3 = 0; e3 < 12; e3 += 3) {
        long long mr = 1ll << 31, mi = 1ll << 31;
#pragma unroll
        for (int e = e3; e < e3 + 3; ++e) {
          const longlong2 v = q[e * 32];
          int rh, rl, ih, il;
          split(v.x, rh, rl);
          split(v.y, ih, il);
          // conj(v) w = (vr wr + vi wi, vr wi - vi wr); lo may be -2^31, so in a cross product the negated
          // factor is a hi
          re = madw(re, rh, wh[e][0]);
          im = madw(im, rh, wh[e][1]);
          mr = madw(mr, rh, wl[e][0]);
          mi = madw(mi, rh, wl[e][1]);
          mr = madw(mr, rl, wh[e][0]);
          mi = madw(mi, rl, wh[e][1]);
          re = madw(re, ih, wh[e][1]);
          im = madw(im, -ih, wh[e][0]);
          mr = madw(mr, ih, wl[e][1]);
          mi = madw(mi, -ih, wl[e][0]);
          mr = madw(mr, il, wh[e][1]);
          mi = madw(mi, il, -wh[e][0]);
        }
        re = madw(re, (int)(mr >> 32), 1);
        im = madw(im, (int)(mi >> 32), 1);
      }
      if (s0 < S) {
        if (held && X >= X_LOW && X <= X_HIGH) {
          const double k = pow2(X - 2100);
          acc[2 * j] = fma((double)re, k, acc[2 * j]);
          acc[2 * j + 1] = fma((double)im, k, acc[2 * j + 1]);
        } else if (mx == 0 ? xv == FX_BAD : xv != FX_MINX || Xw == 0x7ff) {   // no block of zeros, or one against NaN, Inf
          const double2 *v = V + (fld * S + s) * 12;
          double dr = 0.0, di = 0.0;
#pragma unroll 1
          for (int e = 0; e < 12; ++e) {
            const double2 a = v[e], o = m[e];
            dr = fma(a.x, o.x, dr);
            dr = fma(a.y, o.y, dr);
            di = fma(a.x, o.y, di);
            di = fma(-a.y, o.x, di);
          }
          acc[2 * j] += dr;
          acc[2 * j + 1] += di;
        }
      }
      __syncwarp();   // the stage is filled again two vectors on
    }
  }
  wait_but<0>();
  // 16 sums over 32 lanes by halves: lane pairs end up with one of the sums each
#pragma unroll
  for (int n = FG, o = 16; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const double send = up ? acc[j] : acc[j + n], keep = up ? acc[j + n] : acc[j];
      acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
  static_assert(FG == 8, "16 sums over the lane bits 16, 8, 4, 2");
  if ((lane & 1) == 0) red[warp][lane >> 1] = acc[0];
  __syncthreads();
  if (threadIdx.x < ng) {
    double2 sum = make_double2(0.0, 0.0);
    for (int k = 0; k < FB / 32; ++k) {
      sum.x += red[k][2 * threadIdx.x];
      sum.y += red[k][2 * threadIdx.x + 1];
    }
    partial[((long long)(i0 + threadIdx.x) * nrhs + r) * nchunk + c] = sum;
  }
  __threadfence();
  __syncthreads();
  unsigned *cnt = counters + (long long)r * ngroup + g0;
  if (threadIdx.x == 0) last = (atomicAdd(cnt, 1u) == (unsigned)(nchunk - 1));
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int j = warp; j < ng; j += FB / 32) {
    const double2 *pp = partial + ((long long)(i0 + j) * nrhs + r) * nchunk;
    double2 sum = make_double2(0.0, 0.0);
    for (int q = lane; q < nchunk; q += 32) sum = cadd(sum, __ldcg(pp + q));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
      sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
    }
    if (lane == 0) h[(long long)(i0 + j) * nrhs + r] = sum;
  }
  if (threadIdx.x == 0) *cnt = 0u;
}

// w^r += sign * sum_i V_i^r h[i * nrhs + r].  Block: 32 sites of one right-hand side, warp = spin, so that a
// thread sums three complex components.  Coefficients as 59-bit integers with one exponent each.
// VS > 1, for fields that leave most of the chip idle: VS = 4 such groups of four warps share the sites and
// take every fourth vector, and their integers at the one exponent are added.
// Eight blocks per SM (64 registers): 4.8 TB/s on 50 right-hand sides of 8^3 x 16, 4.1 to 4.4 with four to
// six; the FP64 sums ran at 1.3.
constexpr int FAXPY_MAXV = 512;
template <int VS>
__global__ void __launch_bounds__(FB * VS, 8 / VS) fx_multiaxpy_kernel(Field f, const double2 *__restrict__ V,
                                                             const double2 *__restrict__ h, double sign,
                                                             double2 *__restrict__ w, int S, int nvec, int nrhs) {
  extern __shared__ __align__(16) char dyn[];   // coefficients int4[nvec], exponents int[nvec]
  __shared__ __align__(16) char sm[WARP_BYTES];
  int4 *cf = (int4 *)dyn;
  int *cx = (int *)(cf + nvec);
  const int r = blockIdx.x % nrhs;
  const int lane = threadIdx.x & 31, gw = threadIdx.x >> 5, warp = gw % 4, vg = gw / 4;   // spin, vector group
  const int s0 = (blockIdx.x / nrhs) * 32 + lane, s = min(s0, S - 1);
  double2 *wr = w + (long long)r * S * 12;
  Stage st;
  st.init(sm);
  if (vg == 0) st.load<4>(wr, s, warp);
  bool odd = false;   // a coefficient outside the range of the integers
  for (int i = threadIdx.x; i < nvec; i += FB * VS) {
    const double2 a = h[(long long)i * nrhs + r];
    const int X = max(mag(a.x), mag(a.y)) >> 20;
    const bool zero = a.x == 0.0 && a.y == 0.0;
    odd = odd || X >= 0x7fe || (X < FX_MIN_FIELD && !zero);
    int4 c;
    split(fixed(sign * a.x, 5 + max(X, FX_MINX)), c.x, c.y);
    split(fixed(sign * a.y, 5 + max(X, FX_MINX)), c.z, c.w);
    c.w = max(c.w, -0x7fffffff);   // its negative is used below
    cf[i] = c;
    cx[i] = zero ? 0 : X;
  }
  wait_all();
  odd = __syncthreads_or(odd) != 0;
  const long long fq = blocks32(S) * 384;
  // the exponent of the sum: sum_i 2^(X_i) <= 2^(E + 6) with X_i = X_V + X_h, E at least their largest.
  // Zero blocks and coefficients have no share.  Each warp looks at its share of the vectors.
  __shared__ float s_tot[4 * VS][32];
  __shared__ int s_E[4 * VS][32];
  int E = 0;
  float tot = 0.f;
  auto share = [](int &E, float &tot, int X, float n) {   // (E, tot) += n 2^X
    const int d = X - E;
    if (d > 0) {
      tot = (d > 100 ? 0.f : tot * __int_as_float((127 - d) << 23)) + n;
      E = X;
    } else if (d > -100) {
      tot += n * __int_as_float((127 + d) << 23);
    }
  };
#pragma unroll 4
  for (int i = gw; i < nvec; i += 4 * VS) {
    const int xv = __ldg(f.ex + ((long long)i * nrhs + r) * S + s) & ~FX_WIDE, xh = cx[i];
    if (xv == FX_MINX || (xh == 0 && xv != FX_BAD)) continue;
    const int X = xv + xh;
    odd = odd || X > X_HIGH || X < X_LOW;
    share(E, tot, X, 1.f);
  }
  s_E[gw][lane] = E;
  s_tot[gw][lane] = odd ? INFINITY : tot;
  __syncthreads();
  E = 0;
  tot = 0.f;
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 4 * VS; ++k) {
    bad = bad || isinf(s_tot[k][lane]);
    if (s_E[k][lane] > 0) share(E, tot, s_E[k][lane], s_tot[k][lane]);
  }
  E += max(0, (__float_as_int(tot) >> 23) - 127 + 1 - 6);
  double2 *m = st.mine() + 3 * warp;
  long long hh[3][2], md[3][2];
#pragma unroll
  for (int c = 0; c < 3; ++c) hh[c][0] = hh[c][1] = 0, md[c][0] = md[c][1] = 1ll << 31;
  if (!bad) {
    const longlong2 *q = f.q + ((long long)vg * nrhs + r) * fq + slot(s, 12) + 3 * warp * 32;
    const int *ex = f.ex + ((long long)vg * nrhs + r) * S + s;
#pragma unroll 4
    for (int i = vg; i < nvec; i += VS, q += (long long)VS * nrhs * fq, ex += (long long)VS * nrhs * S) {
      const int4 k = cf[i];
      const int sh = max(0, min(E - (__ldg(ex) & ~FX_WIDE) - cx[i], 63));   // out of 0..63 only where the product is 0
      const int nzh = -k.z, nzl = -k.w;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const longlong2 v = __ldg(q + c * 32);
        int rh, rl, ih, il;
        split(v.x >> sh, rh, rl);
        split(v.y >> sh, ih, il);
        hh[c][0] = madw(hh[c][0], k.x, rh);
        hh[c][1] = madw(hh[c][1], k.x, ih);
        md[c][0] = madw(md[c][0], k.x, rl);
        md[c][1] = madw(md[c][1], k.x, il);
        md[c][0] = madw(md[c][0], k.y, rh);
        md[c][1] = madw(md[c][1], k.y, ih);
        hh[c][0] = madw(hh[c][0], nzh, ih);
        hh[c][1] = madw(hh[c][1], k.z, rh);
        md[c][0] = madw(md[c][0], nzh, il);
        md[c][1] = madw(md[c][1], k.z, rl);
        md[c][0] = madw(md[c][0], nzl, ih);
        md[c][1] = madw(md[c][1], k.w, rh);
      }
      if ((i / VS & 3) == 3) {   // four vectors: |md| < 2^63
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            hh[c][z] = madw(hh[c][z], (int)(md[c][z] >> 32), 1);
            md[c][z] &= 0xffffffffll;
          }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int z = 0; z < 2; ++z) hh[c][z] = madw(hh[c][z], (int)(md[c][z] >> 32), 1);
  }
  if constexpr (VS > 1) {
    __shared__ long long part[VS - 1][6][FB];
    if (vg > 0) {
#pragma unroll
      for (int z = 0; z < 6; ++z) part[vg - 1][z][threadIdx.x % FB] = hh[z / 2][z % 2];
    }
    __syncthreads();
    if (vg == 0) {
#pragma unroll
      for (int g = 0; g < VS - 1; ++g)
#pragma unroll
        for (int z = 0; z < 6; ++z) hh[z / 2][z % 2] += part[g][z][threadIdx.x];
    }
  }
  if (vg > 0) {
    // the first group ends the sum
  } else if (!bad) {
    // E = 0: every share was zero
    const double k = E >= X_LOW ? pow2(E - 2099) : 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const long long re = hh[c][0], im = hh[c][1];
      const double2 o = m[c];
      m[c] = make_double2(fma((double)re, k, o.x), fma((double)im, k, o.y));
    }
  } else {
    double2 a[3] = {m[0], m[1], m[2]};
#pragma unroll 1
    for (int i = 0; i < nvec; ++i) {
      const double2 *v = V + (((long long)i * nrhs + r) * S + s) * 12 + 3 * warp, k = cscale(h[(long long)i * nrhs + r], sign);
#pragma unroll
      for (int c = 0; c < 3; ++c) cfma(a[c], v[c], k);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) m[c] = a[c];
  }
  __syncthreads();
  if (vg == 0) st.store<4>(wr, s0 < S ? s : -1, warp);
}

// blocks per (right-hand side, vector group): about 12 blocks per SM, six resident rounds; at least one
// warp strip each
int dot_chunks(const lqcd_ctx *ctx, long long S, int nrhs, int nvec) {
  const long long ngroup = (nvec + FG - 1) / FG, most = (blocks32(S) + FB / 32 - 1) / (FB / 32);
  return (int)std::max<long long>(1, std::min<long long>(most, (12LL * ctx->sms + nrhs * ngroup - 1) / (nrhs * ngroup)));
}

}  // namespace

lqcd_status fx_blas_reserve(lqcd_ctx *ctx, long long S, int nrhs, int max_nvec) {
  size_t need = 0;
  for (int v = 1; v <= max_nvec; ++v) need = std::max(need, sizeof(double2) * (size_t)dot_chunks(ctx, S, nrhs, v) * nrhs * v);
  void *p;
  return ws_get(ctx, WS_PARTIAL, need, &p);
}

lqcd_status fx_multidot(lqcd_ctx *ctx, const fx::Field &f, const double2 *V, const double2 *w, long long S, int nvec,
                        int nrhs, double2 *h) {
  const int ngroup = (nvec + FG - 1) / FG, nchunk = dot_chunks(ctx, S, nrhs, nvec);
  const long long grid = (long long)nchunk * ngroup * nrhs;
  if (grid > 0x7fffffffLL) return set_err(ctx, LQCD_ERR_INVALID_ARG, "fx_multidot: grid too large");
  void *p;
  unsigned *cnt;
  LQCD_TRY(ws_get(ctx, WS_PARTIAL, sizeof(double2) * (size_t)nchunk * nrhs * nvec, &p));
  LQCD_TRY(reduction_counters(ctx, nrhs * ngroup, &cnt));
  LQCD_CUDA(ctx, cudaFuncSetAttribute(fx_multidot_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DOT_SMEM));
  kbegin(ctx);
  fx_multidot_kernel<<<(unsigned)grid, FB, DOT_SMEM, ctx->stream>>>(f, V, w, (int)S, nvec, nrhs, nchunk, (double2 *)p, cnt, h);
  return launch_check_bytes(ctx, "fx_multidot_kernel", K_DOT, 12.0 * S * nrhs * nvec, 196.0 * S * nrhs * nvec + 192.0 * S * nrhs);
}

lqcd_status fx_multiaxpy(lqcd_ctx *ctx, const fx::Field &f, const double2 *V, const double2 *h, double sign, double2 *w,
                         long long S, int nvec, int nrhs) {
  if (nvec > FAXPY_MAXV) return set_err(ctx, LQCD_ERR_INVALID_ARG, "fx_multiaxpy: at most %d vectors", FAXPY_MAXV);
  const long long grid = fx::blocks32(S) * nrhs;
  if (grid > 0x7fffffffLL) return set_err(ctx, LQCD_ERR_INVALID_ARG, "fx_multiaxpy: grid too large");
  kbegin(ctx);
  const int vs = grid < 4LL * ctx->sms && nvec > 1 ? 4 : 1;   // fewer than 16 warps per SM
  (vs == 4 ? fx_multiaxpy_kernel<4> : fx_multiaxpy_kernel<1>)
      <<<(unsigned)grid, FB * vs, nvec * (sizeof(int4) + sizeof(int)), ctx->stream>>>(f, V, h, sign, w, (int)S, nvec, nrhs);
  return launch_check_bytes(ctx, "fx_multiaxpy_kernel", K_AXPY, 12.0 * S * nrhs * nvec, 196.0 * S * nrhs * nvec + 384.0 * S * nrhs);
}

// Integers of nvec x nrhs canonical fields V in WS_FX_BASIS
static lqcd_status basis_field(lqcd_ctx *ctx, const double2 *V, int nvec, int nrhs, fx::Field *f) {
  const long long S = ctx->V, cnt = (long long)nvec * nrhs;
  if ((S / 32 + 1) * cnt > 0x7fffffffLL) return set_err(ctx, LQCD_ERR_INVALID_ARG, "basis product: too many vectors");
  const size_t qb = (size_t)cnt * fx::blocks32(S) * 384 * sizeof(longlong2);
  char *p;
  LQCD_TRY(ws_get(ctx, WS_FX_BASIS, qb + (size_t)cnt * S * sizeof(int), (void **)&p));
  f->q = (longlong2 *)p;
  f->ex = (int *)(p + qb);
  return fx_convert(ctx, V, *f, S, (int)cnt);
}

extern "C" lqcd_status lqcd_basis_dot(lqcd_ctx *ctx, const double *V, int nvec, const double *w, int nrhs, double *h) {
  if (!ctx) return LQCD_ERR_INVALID_ARG;
  if (!V || !w || !h || nvec < 1 || nvec > FAXPY_MAXV || nrhs < 1 || nrhs > 65535)
    return set_err(ctx, LQCD_ERR_INVALID_ARG, "basis_dot: bad arguments");
  FxScope scope(ctx);
  fx::Field f;
  LQCD_TRY(fx_blas_reserve(ctx, ctx->V, nrhs, nvec));
  LQCD_TRY(basis_field(ctx, (const double2 *)V, nvec, nrhs, &f));
  return fx_multidot(ctx, f, (const double2 *)V, (const double2 *)w, ctx->V, nvec, nrhs, (double2 *)h);
}

extern "C" lqcd_status lqcd_basis_update(lqcd_ctx *ctx, const double *V, int nvec, const double *h, double *w, int nrhs) {
  if (!ctx) return LQCD_ERR_INVALID_ARG;
  if (!V || !w || !h || nvec < 1 || nvec > FAXPY_MAXV || nrhs < 1 || nrhs > 65535)
    return set_err(ctx, LQCD_ERR_INVALID_ARG, "basis_update: bad arguments");
  FxScope scope(ctx);
  fx::Field f;
  LQCD_TRY(basis_field(ctx, (const double2 *)V, nvec, nrhs, &f));
  return fx_multiaxpy(ctx, f, (const double2 *)V, (const double2 *)h, -1.0, (double2 *)w, ctx->V, nvec, nrhs);
}
