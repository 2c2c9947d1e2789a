// FP64-accurate stencil arithmetic on the integer units.
//
// GB300 issues 2 FP64 operations per SM and clock (DFMA 1.9, conversions to and from
// FP64 as well, measured) but 22 32 x 32 + 64 bit multiply-adds (mad.wide.s32), 60
// 64-bit additions and 30 64-bit shifts.  A complex product of 64-bit numbers takes 12
// of the first, half a clock, against 2 clocks for its 4 DFMA.  The operators here are linear with coefficients known in advance (links, Galerkin
// blocks), so their inputs are carried as 64-bit integers with one power-of-two
// scale per site:
//   value = v * 2^(e - FX_BIAS),  |v| < 2^FX_BITS,
// e the largest biased FP64 exponent of the site's components.  A sum over
// neighbours is formed at the largest exponent among its terms: each is
// computed at its own site's scale and shifted right by the difference.  Hop
// terms are smaller than their site by 2 diag: their coefficients are held times
// 2^k and their exponents are e - k.  The absolute error of a result is then a few
// units of 2^-58 of the largest term, below the 2^-53 roundings of the same sum in
// FP64, whatever the range of the field elsewhere.
// Results do not depend on the tiling.  Components below the FP64 normal range
// count as zero next to larger ones; sites holding infinities or NaN, or whose
// exponents lie outside [FX_EMIN, FX_EMAX] (sites of subnormals alone among them: the
// test for those takes 0.6% of 256^2 x 64, and telling them apart per tile or per
// result took as much), get the exponent FX_BAD, which every sum over neighbours
// inherits: their results are recomputed in FP64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace mgk {

static constexpr int FX_BITS = 58;
static constexpr int FX_BIAS = 1022 + FX_BITS;
static constexpr int FX_EMIN = 200, FX_EMAX = 1800, FX_BAD = 1 << 14;

struct FxC { long long re, im; };                    // a complex fixed-point number
struct FxSpinor { FxC a, b; int e; };                // both spin components of a site

// A component (FP64 words hi, lo) as a 64-bit integer; kmax = the largest exponent field
// (hi & 0x7ff00000) of the site, at least 64 << 20 so that zeros shift out.
__host__ __device__ __forceinline__ long long fx_component(uint32_t hi, uint32_t lo, uint32_t kmax) {
  const uint32_t mh = (hi & 0xfffff) | 0x100000;
  unsigned long long m = (((unsigned long long)mh << 32) | lo) << (FX_BITS - 53);
  const int sh = (int)((kmax - (hi & 0x7ff00000)) >> 20);
  m >>= sh > 63 ? 63 : sh;
  return (int)hi < 0 ? -(long long)m : (long long)m;
}

// a site's two spin components (re, im, re, im) as FP64 bit patterns
__host__ __device__ __forceinline__ FxSpinor fx_spinor(const uint32_t (&hi)[4], const uint32_t (&lo)[4]) {
  const uint32_t k = 0x7ff00000;
  uint32_t m = hi[0] & k, n = hi[1] & k, p = hi[2] & k, q = hi[3] & k;
  m = m > n ? m : n;
  p = p > q ? p : q;
  m = m > p ? m : p;
  const int e = (int)(m >> 20);
  m = m > (64u << 20) ? m : (64u << 20);
  FxSpinor f;
  f.a.re = fx_component(hi[0], lo[0], m);
  f.a.im = fx_component(hi[1], lo[1], m);
  f.b.re = fx_component(hi[2], lo[2], m);
  f.b.im = fx_component(hi[3], lo[3], m);
  if (e == 0)                                          // a zero site, or subnormals alone
    f.e = ((hi[0] | hi[1] | hi[2] | hi[3]) & 0xfffff) | lo[0] | lo[1] | lo[2] | lo[3] ? FX_BAD : 0;
  else
    f.e = (unsigned)(e - FX_EMIN) > FX_EMAX - FX_EMIN ? FX_BAD : e;
  return f;
}

__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)a * b + c;
#endif
}

// v = hi * 2^32 + lo with lo signed
__host__ __device__ __forceinline__ int fx_lo(long long v) { return (int)v; }
__host__ __device__ __forceinline__ int fx_hi(long long v) {
  return (int)(v >> 32) + (int)((uint32_t)v >> 31);
}

// A complex coefficient w * 2^64 split into signed words {re_lo, re_hi, im_lo, im_hi}.
// (w h) and (conj(w) h) without the product of the low words (2^-62 of the largest
// product).  With |w| <= 1/3 and |h| components below 2^61.3 no sum leaves 64 bits:
// the words of w are below 2^30.5 and 2^31, those of h below 2^29.3 and 2^31, so the
// four middle products add to less than 2^62.7.
__host__ __device__ __forceinline__ FxC fx_cmul(int4 w, FxC h, bool conj) {
  const int rl = fx_lo(h.re), rh = fx_hi(h.re), il = fx_lo(h.im), ih = fx_hi(h.im);
  const int pl = conj ? -w.z : w.z, ph = conj ? -w.w : w.w;      // Im of the factor
  const int nl = conj ? w.z : -w.z, nh = conj ? w.w : -w.w;      // and its negative
  long long m = fx_mad(w.y, rl, fx_mad(w.x, rh, fx_mad(nh, il, (long long)nl * ih)));
  FxC r;
  r.re = fx_mad(w.y, rh, fx_mad(nh, ih, m >> 32));
  m = fx_mad(w.y, il, fx_mad(w.x, ih, fx_mad(ph, rl, (long long)pl * rh)));
  r.im = fx_mad(w.y, ih, fx_mad(ph, rh, m >> 32));
  return r;
}

__host__ __device__ __forceinline__ FxC fx_shr(FxC p, int s) { return {p.re >> s, p.im >> s}; }
__host__ __device__ __forceinline__ int fx_gap(int f, int e) { return f - e > 63 ? 63 : f - e; }

// Hop terms of the Wilson stencil from the spinor f, S = +1: projector (1 - sigma),
// S = -1: (1 + sigma); w = 2^k link / (2 diag), CONJ for the backward hop.  Returned at
// the scale of f over 2^k (fx_hop_*), and added to the row sum (fx_add_*): with
// D psi / diag = psi - sum w (1 -+ sigma) psi, the hops enter with a minus sign.
template <int S, bool CONJ>
__host__ __device__ __forceinline__ FxC fx_hop_x(int4 w, const FxSpinor& f) {
  const FxC h = S > 0 ? FxC{f.a.re - f.b.re, f.a.im - f.b.im} : FxC{f.a.re + f.b.re, f.a.im + f.b.im};
  return fx_cmul(w, h, CONJ);
}
template <int S, bool CONJ>
__host__ __device__ __forceinline__ FxC fx_hop_t(int4 w, const FxSpinor& f) {
  const FxC h = S > 0 ? FxC{f.a.re - f.b.im, f.a.im + f.b.re} : FxC{f.a.re + f.b.im, f.a.im - f.b.re};
  return fx_cmul(w, h, CONJ);
}
// row sum of D (S = +1) or D^dagger (S = -1) over diag: forward hops with (1 - S sigma),
// backward hops with (1 + S sigma); c the site's own spinor, all at one scale
template <int S>
__host__ __device__ __forceinline__ void fx_row(FxSpinor& r, const FxSpinor& c, FxC xf, FxC xb,
                                                FxC tf, FxC tb) {
  const FxC xs = {xf.re + xb.re, xf.im + xb.im}, ts = {tf.re + tb.re, tf.im + tb.im};
  const FxC xd = {xf.re - xb.re, xf.im - xb.im}, td = {tf.re - tb.re, tf.im - tb.im};
  r.a.re = c.a.re - xs.re - ts.re;
  r.a.im = c.a.im - xs.im - ts.im;
  if (S > 0) {
    r.b.re = c.b.re + xd.re - td.im;
    r.b.im = c.b.im + xd.im + td.re;
  } else {
    r.b.re = c.b.re - xd.re + td.im;
    r.b.im = c.b.im - xd.im - td.re;
  }
}

// Output scale: y * ca * diag^2 as FP64, the factor as q * 2^(exp - 64) in split words.
struct FxScale { int lo, hi; int exp; };             // exp: added to the site exponent
__host__ __device__ __forceinline__ long long fx_scale(long long y, FxScale q) {
  const int yl = fx_lo(y), yh = fx_hi(y);
  const long long m = fx_mad(q.hi, yl, (long long)q.lo * yh);
  return fx_mad(q.hi, yh, m >> 32);
}
// factor = q * 2^(exp - 64), |q| about 2^62 .. 2^63 - 2^31: the carry of the low word has to fit
// into the high one.  A q above that (ca diag^2 less than 2^-32 of itself below a power of
// two, or rounded up to one) is halved.
inline FxScale make_scale(double ca, double diag) {
  int ex;
  const double f = std::frexp(diag * diag, &ex);       // the product's rounding is recovered below
  const double lo = std::ldexp(std::fma(diag, diag, -diag * diag), -ex);
  int ec;
  const double c = std::frexp(std::fabs(ca), &ec);
  double ph = f * c, pl = std::fma(f, c, -ph) + lo * c;
  if (ph < 0.5) { ph *= 2; pl *= 2; --ex; }
  unsigned long long m = (unsigned long long)std::ldexp(ph, 63) + (long long)std::llrint(std::ldexp(pl, 63));
  if (m >= (1ull << 63) - (1ull << 31)) {
    m = (m + 1) >> 1;
    ++ex;
  }
  const long long q = ca < 0 ? -(long long)m : (long long)m;
  return FxScale{fx_lo(q), fx_hi(q), ex + ec + 1};
}
// v * 2^(e + shift) of an FP64-representable size
__device__ __forceinline__ double fx_double(long long v, int e) {
  const double d = (double)v;
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
}

// k: the largest with |w| = 2^k / (2 |diag|) <= 1/3, where the products stay in range.  With 0
// everywhere, fields that fall by 1 / diag per site kept 44 bits at |diag| = 64; below 6 they
// keep 50 or more (two hops are 1 / (4 diag^2) of a site), and k stays 0.
inline int fixed_shift(double diag) {
  const double a = std::fabs(diag);
  return a < 6.0 ? 0 : std::ilogb(a / 1.5);
}
// |diag| from 1.5 to 64 (k = 5).
__host__ __device__ __forceinline__ bool fixed_diag_ok(double diag) {
  const double a = diag < 0 ? -diag : diag;
  return a >= 1.5 && a <= 64.0;
}

}  // namespace mgk
