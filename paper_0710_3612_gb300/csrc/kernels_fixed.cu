// Fine-lattice A = D^dagger D on FP64 vectors with the integer arithmetic of
// fixed.cuh: FP64 instructions are left only for the output conversion (4 per
// site) and the optional epilogue, so the kernel is bound by integer issue and
// HBM instead of the 2 FP64 operations per SM and clock.
#include <cmath>

#include "fixed.cuh"
#include "kernels.h"
#include "wilson.cuh"

namespace mgk {

namespace {

__device__ __forceinline__ FxSpinor to_fixed(const double2& a, const double2& b) {
  const uint32_t hi[4] = {(uint32_t)__double2hiint(a.x), (uint32_t)__double2hiint(a.y),
                          (uint32_t)__double2hiint(b.x), (uint32_t)__double2hiint(b.y)};
  const uint32_t lo[4] = {(uint32_t)__double2loint(a.x), (uint32_t)__double2loint(a.y),
                          (uint32_t)__double2loint(b.x), (uint32_t)__double2loint(b.y)};
  return fx_spinor(hi, lo);
}

// (A psi)(x, t) in FP64 from global memory: the sites whose neighbourhood holds
// infinities, NaN or extreme exponents.
__device__ __noinline__ void wilson_A_site64(const double2* in, const double2* U, double diag, int x,
                                             int t, int Lx, int Lt, double2* o) {
  const int V = Lx * Lt, site = x + Lx * t;
  const int x1 = x + 1 == Lx ? 0 : x + 1, x0 = x == 0 ? Lx - 1 : x - 1;
  const int t1 = t + 1 == Lt ? 0 : t + 1, t0 = t == 0 ? Lt - 1 : t - 1;
  double2 a0 = mk(0.0, 0.0), a1 = mk(0.0, 0.0), f0, f1;
  wilson_site<double, false>(in, U, diag, x1, t, Lx, Lt, f0, f1);
  hop_x<double>(a0, a1, U[site], f0, f1, -1.0);
  wilson_site<double, false>(in, U, diag, x0, t, Lx, Lt, f0, f1);
  hop_x<double>(a0, a1, cconj(U[x0 + Lx * t]), f0, f1, 1.0);
  wilson_site<double, false>(in, U, diag, x, t1, Lx, Lt, f0, f1);
  hop_t<double>(a0, a1, U[V + site], f0, f1, -1.0);
  wilson_site<double, false>(in, U, diag, x, t0, Lx, Lt, f0, f1);
  hop_t<double>(a0, a1, cconj(U[V + x + Lx * t0]), f0, f1, 1.0);
  wilson_site<double, false>(in, U, diag, x, t, Lx, Lt, f0, f1);
  o[0] = mk(diag * f0.x - 0.5 * a0.x, diag * f0.y - 0.5 * a0.y);
  o[1] = mk(diag * f1.x - 0.5 * a1.x, diag * f1.y - 0.5 * a1.y);
}

struct FxArgs {
  const double2* in;
  double2* out;
  const double2* U;
  const int4* W;
  FxScale q;
  double diag;
  int k;                                               // of the hop terms (fixed_shift)
  int Lx, Lt;
  Epilogue ep;
};
static constexpr int FX_BAD_SUM = FX_BAD / 2;          // sums inherit FX_BAD less 2 k at most

// What follows the stencil at a site: nothing, out = ca y + cu U (+ cw W), or the dot
// with psi (its real part, or both parts).  Separate kernels: a skipped FP64
// instruction still takes its slot on the FP64 pipe (plain 256^2 x 64: 221 us with
// all epilogues predicated into one kernel).
enum { FX_PLAIN = 0, FX_EPI, FX_DOT_RE, FX_DOT };

// y = ca A psi from the fixed-point sum (ca is part of the output scale), then the
// rest of the epilogue.  off: first entry of the vector.
template <int MODE>
__device__ __forceinline__ void fx_output(const FxArgs& a, const FxSpinor& y, int x, int t, long long off,
                                          double& dre, double& dim) {
  const long long g = off + 2LL * (x + a.Lx * t);
  double2 y0, y1;
  if (y.e >= FX_BAD_SUM) {
    double2 o[2];
    wilson_A_site64(a.in + off, a.U, a.diag, x, t, a.Lx, a.Lt, o);
    y0 = mk(a.ep.ca * o[0].x, a.ep.ca * o[0].y);
    y1 = mk(a.ep.ca * o[1].x, a.ep.ca * o[1].y);
  } else {
    const int e = y.e - FX_BIAS + a.q.exp;
    y0 = mk(fx_double(fx_scale(y.a.re, a.q), e), fx_double(fx_scale(y.a.im, a.q), e));
    y1 = mk(fx_double(fx_scale(y.b.re, a.q), e), fx_double(fx_scale(y.b.im, a.q), e));
  }
  if (MODE >= FX_DOT_RE) {
    double2 p0, p1;
    split(ld_spinor(a.in + g), p0, p1);
    dre += p0.x * y0.x + p0.y * y0.y + p1.x * y1.x + p1.y * y1.y;
    if (MODE == FX_DOT) dim += p0.x * y0.y - p0.y * y0.x + p1.x * y1.y - p1.y * y1.x;
  }
  if (MODE == FX_EPI) {
    const Epilogue& ep = a.ep;
    double2 u0, u1;
    split(ld_spinor((const double2*)ep.U + g), u0, u1);
    y0 = mk(y0.x + ep.cu * u0.x, y0.y + ep.cu * u0.y);
    y1 = mk(y1.x + ep.cu * u1.x, y1.y + ep.cu * u1.y);
    if (ep.W) {
      split(ld_spinor((const double2*)ep.W + g), u0, u1);
      y0 = mk(y0.x + ep.cw * u0.x, y0.y + ep.cw * u0.y);
      y1 = mk(y1.x + ep.cw * u1.x, y1.y + ep.cw * u1.y);
    }
  }
  st_spinor(a.out + g, join(y0, y1));
}

// One row sum of D (S = +1) or D^dagger (S = -1) from the site's spinor and the
// four hop products, each with its own site's exponent (k above the product's).
template <int S>
__device__ __forceinline__ FxSpinor fx_sum(FxSpinor c, FxC xf, int exf, FxC xb, int exb, FxC tf, int etf,
                                           FxC tb, int etb, int k) {
  FxSpinor r;
  r.e = max(max(max(exf, exb), max(etf, etb)) - k, c.e);
  const int sc = fx_gap(r.e, c.e), h = r.e + k;
  c.a = fx_shr(c.a, sc);
  c.b = fx_shr(c.b, sc);
  fx_row<S>(r, c, fx_shr(xf, fx_gap(h, exf)), fx_shr(xb, fx_gap(h, exb)), fx_shr(tf, fx_gap(h, etf)),
            fx_shr(tb, fx_gap(h, etb)));
  return r;
}

// Shared-memory field of fixed-point spinors: 16-byte halves and exponents apart,
// so that the lanes of a warp read consecutive words.
struct FxField {
  longlong2 *a, *b;
  int* e;
  __device__ __forceinline__ FxSpinor get(int i) const {
    const longlong2 u = a[i], v = b[i];
    return {{u.x, u.y}, {v.x, v.y}, e[i]};
  }
  __device__ __forceinline__ void put(int i, const FxSpinor& s) const {
    a[i] = make_longlong2(s.a.re, s.a.im);
    b[i] = make_longlong2(s.b.re, s.b.im);
    e[i] = s.e;
  }
};

template <int S>
__device__ __forceinline__ FxSpinor fx_stencil(const FxField& f, int c, int row, const int4* wx,
                                               const int4* wt, int u, int urow, int k) {
  const FxSpinor xp = f.get(c + 1), xm = f.get(c - 1), tp = f.get(c + row), tm = f.get(c - row);
  return fx_sum<S>(f.get(c), fx_hop_x<S, false>(wx[u], xp), xp.e, fx_hop_x<-S, true>(wx[u - 1], xm), xm.e,
                   fx_hop_t<S, false>(wt[u], tp), tp.e, fx_hop_t<-S, true>(wt[u - urow], tm), tm.e, k);
}

template <int TX, int TY, int RPT>
struct FxTile {
  static constexpr int TT = TY * RPT;
  static constexpr int PW = TX + 4, PH = TT + 4, DW = TX + 2, DH = TT + 2, UW = TX + 3, UH = TT + 3;
  static constexpr int NP = PW * PH, ND = DW * DH, NU = UW * UH;
  static constexpr int BYTES = 36 * (NP + ND) + 32 * NU;
};

// Tile kernel (the layout of k_wilson_A): psi with a 2-site halo converted to fixed
// point in shared memory, D psi on the tile plus a 1-site halo, D^dagger on the tile.
// 905 instructions per site at 32 x 16 (426 of them on the 64-wide ALU pipe: shifts,
// masks, comparisons), 22 mad.wide per clock: bound by those two pipes.  256^2 x 64:
// 167 us against 1024 us in FP64 (137 FP64 instructions per site), 128^2 4.2 against
// 10.2 us, 210 x 90 x 12 12.8 against 71.6 us; with the fused dot 207 against 1254 us.
// A warp-streaming form (rows in registers, shuffles along x) took 260 us there.  SHIFT: hop
// terms with k > 0 (1.1% more).
template <int TX, int TY, int RPT, int MINB, int MODE, bool SHIFT>
__global__ void __launch_bounds__(TX* TY, MINB) k_wilson_A_fx(const FxArgs a, int dependent) {
  pdl_wait(dependent);
  using T = FxTile<TX, TY, RPT>;
  extern __shared__ __align__(16) unsigned char fsm[];
  longlong2* p16 = (longlong2*)fsm;
  const FxField fp{p16, p16 + T::NP, (int*)(p16 + 2 * T::NP + 2 * T::ND + 2 * T::NU)};
  const FxField fd{p16 + 2 * T::NP, p16 + 2 * T::NP + T::ND, fp.e + T::NP};
  int4* wx = (int4*)(p16 + 2 * T::NP + 2 * T::ND);
  int4* wt = wx + T::NU;
  const int V = a.Lx * a.Lt;
  const int x0 = blockIdx.x * TX, t0 = blockIdx.y * T::TT;
  const long long off = (long long)blockIdx.z * V * 2;
  const int tid = threadIdx.x;
  for (int q = tid; q < T::NU; q += TX * TY) {
    const int g = wrap_tile(x0 + q % T::UW - 2, a.Lx) + a.Lx * wrap_tile(t0 + q / T::UW - 2, a.Lt);
    wx[q] = a.W[g];
    wt[q] = a.W[V + g];
  }
#pragma unroll 2
  for (int q = tid; q < T::NP; q += TX * TY) {
    const int g = wrap_tile(x0 + q % T::PW - 2, a.Lx) + a.Lx * wrap_tile(t0 + q / T::PW - 2, a.Lt);
    const double2* p = a.in + off + 2LL * g;
    fp.put(q, to_fixed(p[0], p[1]));
  }
  __syncthreads();
  for (int q = tid; q < T::ND; q += TX * TY) {
    const int lx = q % T::DW + 1, lt = q / T::DW + 1;
    fd.put(q, fx_stencil<1>(fp, lt * T::PW + lx, T::PW, wx, wt, lt * T::UW + lx, T::UW, SHIFT ? a.k : 0));
  }
  __syncthreads();
  double dre = 0.0, dim = 0.0;
  const int lx = tid % TX, gx = x0 + lx;
#pragma unroll 1
  for (int k = 0; k < RPT; ++k) {
    const int lt = tid / TX + TY * k, gt = t0 + lt;
    if (gx >= a.Lx || gt >= a.Lt) continue;
    const FxSpinor y = fx_stencil<-1>(fd, (lt + 1) * T::DW + lx + 1, T::DW, wx, wt,
                                      (lt + 2) * T::UW + lx + 2, T::UW, SHIFT ? a.k : 0);
    fx_output<MODE>(a, y, gx, gt, off, dre, dim);
  }
  if (MODE >= FX_DOT_RE) {
    constexpr int N = MODE == FX_DOT ? 2 : 1;
    __shared__ double sh[N * TX * TY];
    finish_reduction_g<N>(dre, dim, a.ep.dot_ws, a.ep.dot_out, sh, blockIdx.z,
                          blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
  }
}

// Links over 2 diag, times 2^k, as split 64-bit words; scale = 2^(63 + k).  The quotient is
// carried to 2^-106 by the division's remainder, so a word is exact to one unit of 2^-63.
__device__ __forceinline__ long long fx_link_word(double u, double diag, double scale) {
  const double q = u / diag, r = fma(-q, diag, u) / diag;
  long long w = (long long)(q * scale) + __double2ll_rn(r * scale);
  if ((int)w == INT32_MIN) ++w;                        // the low word is negated for conj(w)
  return w;
}

__global__ void k_fixed_links(const double2* __restrict__ U, int4* __restrict__ W, double diag, double scale, int n,
                              int dependent) {
  pdl_wait(dependent, U, W);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double2 u = U[i];
  const long long a = fx_link_word(u.x, diag, scale), b = fx_link_word(u.y, diag, scale);
  W[i] = make_int4(fx_lo(a), fx_hi(a), fx_lo(b), fx_hi(b));
}

template <int TX, int TY, int RPT, int MINB, int MODE, bool SHIFT>
cudaError_t launch_shift(const FxArgs& a, int nrhs, cudaStream_t s) {
  using T = FxTile<TX, TY, RPT>;
  static SmemLimit limit;
  const cudaError_t e = limit.raise(k_wilson_A_fx<TX, TY, RPT, MINB, MODE, SHIFT>, T::BYTES);
  if (e != cudaSuccess) return e;
  const dim3 grid((a.Lx + TX - 1) / TX, (a.Lt + T::TT - 1) / T::TT, nrhs);
  launch_after(k_wilson_A_fx<TX, TY, RPT, MINB, MODE, SHIFT>, grid, TX * TY, T::BYTES, s, a);
  return cudaGetLastError();
}

template <int TX, int TY, int RPT, int MINB, int MODE>
cudaError_t launch_mode(const FxArgs& a, int nrhs, cudaStream_t s) {
  return a.k ? launch_shift<TX, TY, RPT, MINB, MODE, true>(a, nrhs, s)
             : launch_shift<TX, TY, RPT, MINB, MODE, false>(a, nrhs, s);
}

template <int TX, int TY, int RPT, int MINB>
cudaError_t launch_tile(const FxArgs& a, int nrhs, cudaStream_t s) {
  if (a.ep.dot_out)
    return a.ep.dot_real ? launch_mode<TX, TY, RPT, MINB, FX_DOT_RE>(a, nrhs, s)
                         : launch_mode<TX, TY, RPT, MINB, FX_DOT>(a, nrhs, s);
  return a.ep.U ? launch_mode<TX, TY, RPT, MINB, FX_EPI>(a, nrhs, s)
                : launch_mode<TX, TY, RPT, MINB, FX_PLAIN>(a, nrhs, s);
}

}  // namespace

cudaError_t fixed_links(const void* U64, void* W, double diag, int Lx, int Lt, cudaStream_t s) {
  const int n = 2 * Lx * Lt;
  launch_after(k_fixed_links, (n + 255) / 256, 256, 0, s, (const double2*)U64, (int4*)W, diag,
               std::ldexp(1.0, 63 + fixed_shift(diag)), n);
  count_launch();
  return cudaGetLastError();
}

// Factors ca of 2^-120 .. 2^120: a result's exponent field is at least 133 + q.exp (hops from a
// site at FX_EMIN, one unit left of their sum) and at most 1805 + q.exp, with q.exp within 14 of ca's.
bool wilson_A_fx_ok(const void* W, double diag, const Epilogue& ep) {
  return W && fixed_diag_ok(diag) && !ep.zq_q && std::fabs(ep.ca) <= 0x1p120 &&
         std::fabs(ep.ca) >= 0x1p-120 && (ep.U || !ep.W) && !(ep.dot_out && (ep.U || ep.ca != 1.0));
}

cudaError_t wilson_A_fx(int tx, int ty, const void* in, void* out, const void* U64, const void* W,
                        double diag, int Lx, int Lt, int nrhs, const Epilogue& ep, cudaStream_t s) {
  const FxArgs a{(const double2*)in, (double2*)out, (const double2*)U64, (const int4*)W,
                 make_scale(ep.ca, diag), diag, fixed_shift(diag), Lx, Lt, ep};
  if (tx == 16 && ty == 8) return launch_tile<16, 8, 1, 4>(a, nrhs, s);
  if (tx == 32 && ty == 8) return launch_tile<32, 8, 1, 3>(a, nrhs, s);
  if (tx == 32 && ty == 16) return launch_tile<32, 8, 2, 3>(a, nrhs, s);
  return cudaErrorInvalidValue;
}

}  // namespace mgk
