// FP64 coarse stencil apply, y(j)[r] = sum_d sum_c A[j][d][r][c] x(j + d)[c], by the
// 64-bit integer arithmetic of fixed.cuh.  A site and right-hand side takes 36 n^2
// FMAs; at 2 FP64 operations per SM and clock k_coarse_apply<double> is bound by them
// (256 sites of 16 dof, 64 right-hand sides: 300 us, 252 us of it FMA issue).
//
// Every block row (site, d, r) gets the exponent of its largest entry, every
// neighbour vector that of its largest component; entries are 56-bit integers at
// those scales, as two signed words of 28 bits.  A complex product takes three real ones,
//   k1 = ar (xr + xi), k2 = xr (ai - ar), k3 = xi (ar + ai); Re = k1 - k3, Im = k1 + k2,
// each accumulated over the row as high and middle partial products (three mad.wide;
// the product of the low words is below 2^-57 of the largest term), so a row's
// dot product is exact to a few units of 2^-56 of its largest entry times the
// largest x, against FP64's 2^-53 per addition.  The nine displacements are then added
// at the largest of their exponents.  Rows or vectors outside the exponent range,
// infinities and NaN take the FP64 path of their right-hand side.  So does a row whose nine
// sums are below 2^-8 of largest times largest: the largest components then meet none but
// small entries, and units of the largest product are coarser than FP64's roundings of those
// (2.5e-10 of the result for a unit vector at mass 60).  Of 2.5 million rows of operators at
// masses -2 to 0.05 on random, smooth and solution vectors none is below 2^-7.
#include "fixed.cuh"
#include "kernels.h"
#include "common.cuh"

namespace mgk {

namespace {

static constexpr int CF_BITS = 56;
// Words: |low| <= 2^27, |high| <= 2^28, sums of two twice that; the high and middle sums
// over 32 columns then stay within 2^62.
static constexpr int CF_NMAX = 32;
static constexpr int CF_ZERO = -(1 << 20);           // exponent of an all-zero row or vector
static constexpr int CF_BAD = 1 << 20;
// range of a row's plus a vector's exponent whose product is a normal FP64 number
static constexpr int CF_SMIN = 1300, CF_SMAX = 2800;
// the nine sums' magnitudes, in units of 2^36 of the 2^56 that largest times largest has at most
static constexpr int CF_SMALL = 1 << (CF_BITS - 8 - 36);

// The larger exponent field; 1 for subnormal numbers, so that rows or vectors of those alone
// are told from zeros (and lie outside the range).
__device__ __forceinline__ uint32_t exp_field(double2 v) {
  const uint32_t hx = (uint32_t)__double2hiint(v.x) & 0x7fffffffu, hy = (uint32_t)__double2hiint(v.y) & 0x7fffffffu;
  const uint32_t k = max(hx, hy) & 0x7ff00000u, lo = (uint32_t)__double2loint(v.x) | (uint32_t)__double2loint(v.y);
  return k == 0 && (hx | hy | lo) ? 1u << 20 : k;
}
// exponent of a row or vector from the largest exponent field of its entries
__device__ __forceinline__ int scale_of(uint32_t k) {
  const int e = (int)(k >> 20);
  return e == 0 ? CF_ZERO : (e < FX_EMIN || e > FX_EMAX) ? CF_BAD : e;
}
__device__ __forceinline__ int2 entry(double v, uint32_t k) {   // {low, high} word
  const uint32_t hi = (uint32_t)__double2hiint(v);
  unsigned long long m = (((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) |
                          (uint32_t)__double2loint(v)) << (CF_BITS - 53);
  const int sh = (int)((k - (hi & 0x7ff00000)) >> 20);
  m >>= sh > 63 ? 63 : sh;
  const long long w = (int)hi < 0 ? -(long long)m : (long long)m;
  const int lo = (int)((uint32_t)w << 4) >> 4;
  return make_int2(lo, (int)((w - lo) >> 28));
}

// high and middle sums of products of split words
struct CfAcc { long long h, m; };
__device__ __forceinline__ void cf_mac(CfAcc& a, int al, int ah, int xl, int xh) {
  a.h = fx_mad(ah, xh, a.h);
  a.m = fx_mad(ah, xl, a.m);
  a.m = fx_mad(al, xh, a.m);
}
// the sum in units of 2^CF_BITS (of the 2^(2 CF_BITS) scale of a product)
__device__ __forceinline__ long long cf_value(CfAcc a) { return a.h + (a.m >> 28); }

// Row `row` of site j for one right-hand side: the nine row sums added at their largest
// exponent (or the FP64 path when `bad`), then out = ca y + cu U + cw W.
__device__ __forceinline__ void cf_output(const double2* in, double2* out, const double2* Aj, int Lx, int Lt,
                                          int n, int j, int rhs, int row, int bad, const longlong2* sp,
                                          const int* pe, const Epilogue& ep) {
  const long long V = (long long)Lx * Lt;
  double2 y = make_double2(0.0, 0.0);
  if (!bad) {
    int f = CF_ZERO;
#pragma unroll
    for (int dd = 0; dd < 9; ++dd) f = max(f, pe[dd * n + row]);
    if (f != CF_ZERO) {
      long long hr = 0, hi = 0;                      // the sums in units of 16, and the
      int lr = 0, li = 0, mag = 0;                   // remainders: nine 63-bit terms
#pragma unroll
      for (int dd = 0; dd < 9; ++dd) {
        const int i = dd * n + row, sh = fx_gap(f, pe[i]);
        const long long vr = sp[i].x >> sh, vi = sp[i].y >> sh;
        hr += vr >> 4;
        hi += vi >> 4;
        lr += (int)vr & 15;
        li += (int)vi & 15;
        mag += abs((int)(vr >> 36)) + abs((int)(vi >> 36));
      }
      const double sc = __hiloint2double((f - 2044 - CF_BITS + 1023) << 20, 0);
      y = make_double2(fma((double)hr, 16.0, (double)lr) * sc, fma((double)hi, 16.0, (double)li) * sc);
      bad = mag < CF_SMALL;
    }
  }
  if (bad) {
    y = make_double2(0.0, 0.0);
    for (int dd = 0; dd < 9; ++dd) {
      int xn = j % Lx + dd % 3 - 1, tn = j / Lx + dd / 3 - 1;
      xn = xn < 0 ? xn + Lx : (xn >= Lx ? xn - Lx : xn);
      tn = tn < 0 ? tn + Lt : (tn >= Lt ? tn - Lt : tn);
      const double2* xs = in + (rhs * V + xn + Lx * tn) * n;
      double2 acc = make_double2(0.0, 0.0);
      for (int c = 0; c < n; ++c) cfma(acc, Aj[(dd * n + row) * n + c], xs[c]);
      y = cadd(y, acc);
    }
  }
  const long long gi = (rhs * V + j) * n + row;
  y = make_double2(ep.ca * y.x, ep.ca * y.y);
  if (ep.U) {
    const double2 u = ((const double2*)ep.U)[gi];
    y = make_double2(y.x + ep.cu * u.x, y.y + ep.cu * u.y);
  }
  if (ep.W) {
    const double2 w = ((const double2*)ep.W)[gi];
    y = make_double2(y.x + ep.cw * w.x, y.y + ep.cw * w.y);
  }
  out[gi] = y;
}

// Everything derived from the FP64 blocks of a level, one CTA per site: with COMB, the
// blocks themselves as G0 + m G1 + m^2 I; their FP32 and BF16 copies; and their words,
// column by column (the 9 n rows of a column consecutive, so that the threads of the
// apply, one per row, read whole lines), with the exponent of every row.  One pass over
// the blocks; separate combination and conversion kernels took 47 us for 1024 sites of
// 16 dof, this one 35 us with the words.  Lanes of a power of two >= n share a row.
template <bool COMB>
__global__ void __launch_bounds__(256) k_coarse_finish(const double2* __restrict__ G0,
                                                       const double2* __restrict__ G1, double m,
                                                       double2* __restrict__ A64, float2* __restrict__ A32,
                                                       __nv_bfloat162* __restrict__ A16, int4* __restrict__ W,
                                                       int* __restrict__ E, int n, int P, int dependent) {
  pdl_wait(dependent, G0, G1, A64, A32, A16, W, E);
  extern __shared__ int4 wsm[];                      // [9 n][n | 1]
  const int NR = 9 * n, LD = n | 1;
  const int c = threadIdx.x & (P - 1), step = 256 / P;
  const long long base = (long long)blockIdx.x * NR * n;
  for (int q0 = 0; q0 < NR; q0 += step) {
    const int q = q0 + threadIdx.x / P;
    const bool in = q < NR && c < n;
    const long long i = base + q * n + c;
    double2 v = make_double2(0.0, 0.0);
    if (in) {
      if (COMB) {
        const double2 x = G0[i], y = G1[i];
        v = make_double2(x.x + m * y.x, x.y + m * y.y);
        if (q / n == 4 && q % n == c) v.x += m * m;
        A64[i] = v;
      } else {
        v = A64[i];
      }
      A32[i] = make_float2((float)v.x, (float)v.y);
      A16[i] = __floats2bfloat162_rn((float)v.x, (float)v.y);
    }
    if (!W) continue;
    uint32_t k = exp_field(v);
    for (int o = P >> 1; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
    if (!in) continue;
    if (c == 0) E[(long long)blockIdx.x * NR + q] = scale_of(k);
    k = max(k, 64u << 20);                           // zeros of a zero row shift out
    const int2 re = entry(v.x, k), im = entry(v.y, k);
    wsm[q * LD + c] = make_int4(re.x, re.y, im.x, im.y);
  }
  if (!W) return;
  __syncthreads();
  for (int e = threadIdx.x; e < NR * n; e += 256) W[base + e] = wsm[(e % NR) * LD + e / NR];
}

// One CTA per (coarse site, rpc right-hand sides), one thread per row, RG right-hand sides
// at a time sharing every block entry read.  Bound by mad.wide (9 per complex product, 22
// a clock) and the latency of its four phases.  16 dof, us (k_coarse_apply<double>): 256
// sites 8.2 (10.1), x 16 28 (65), x 64 88 (300); 1024 sites 14.5 (24.6), x 8 49 (153);
// 4096 sites 45 (90).  Splitting a row over 2 or 4 threads for one right-hand side was
// slower (16.4, 26.7 us at 1024 sites: fewer CTAs per SM).
template <int RG>
__global__ void __launch_bounds__(288, RG == 1 ? 1 : 2) k_coarse_fx(const double2* __restrict__ in, double2* out, const double2* __restrict__ A,
                            const int4* __restrict__ W, const int* __restrict__ E, int Lx, int Lt, int n,
                            int nrhs, int rpc, Epilogue ep, int dependent) {
  pdl_wait(dependent, in, out, A, W, E);
  extern __shared__ __align__(16) unsigned char csm[];
  const int NR = 9 * n;
  longlong2* sp = (longlong2*)csm;                   // [RG][NR] row sums
  int4* sx = (int4*)(sp + RG * NR);              // [RG][NR] xr, xi as split words
  int2* ss = (int2*)(sx + RG * NR);                  // [RG][NR] xr + xi
  int* pe = (int*)(ss + RG * NR);                    // [RG][NR] exponent of a row sum
  uint32_t* kx = (uint32_t*)(pe + RG * NR);          // [RG][9]
  int* bad = (int*)(kx + RG * 9);                    // [RG]
  const int j = blockIdx.x, jx = j % Lx, jt = j / Lx, tid = threadIdx.x;
  const long long V = (long long)Lx * Lt;
  const int q = tid, d = q / n, r = q - d * n;
  const bool row = q < NR;
  const int4* Wj = W + (long long)j * n * NR + q;
  int ea = CF_ZERO;
  long long nb = 0;                                  // first entry of x(j + d)
  if (row) {
    ea = E[(long long)j * NR + q];
    int xn = jx + d % 3 - 1, tn = jt + d / 3 - 1;
    xn = xn < 0 ? xn + Lx : (xn >= Lx ? xn - Lx : xn);
    tn = tn < 0 ? tn + Lt : (tn >= Lt ? tn - Lt : tn);
    nb = (long long)(xn + Lx * tn) * n;
  }
  const int r1 = min((int)(blockIdx.y + 1) * rpc, nrhs);
  for (int r0 = blockIdx.y * rpc; r0 < r1; r0 += RG) {
    double2 xv[RG];
#pragma unroll
    for (int g = 0; g < RG; ++g)                     // thread (d, r) loads component r of x(j + d)
      xv[g] = row && r0 + g < r1 ? in[(r0 + g) * V * n + nb + r] : make_double2(0.0, 0.0);
    for (int i = tid; i < RG * 9; i += blockDim.x) kx[i] = 0;   // more than a warp; n = 2 has one
    __syncthreads();                                 // kx cleared; the previous group's sums are read
    if (tid < RG) bad[tid] = 0;
#pragma unroll
    for (int g = 0; g < RG; ++g)
      if (row) atomicMax(&kx[g * 9 + d], exp_field(xv[g]));
    __syncthreads();
    if (row) {
#pragma unroll
      for (int g = 0; g < RG; ++g) {
        const uint32_t k = kx[g * 9 + d], km = max(k, 64u << 20);
        const int ex = scale_of(k), e = ea + ex;
        const int2 xr = entry(xv[g].x, km), xi = entry(xv[g].y, km);
        sx[g * NR + q] = make_int4(xr.x, xr.y, xi.x, xi.y);
        ss[g * NR + q] = make_int2(xr.x + xi.x, xr.y + xi.y);
        const bool zero = ea == CF_ZERO || ex == CF_ZERO;
        pe[g * NR + q] = zero ? CF_ZERO : e;
        if (ea == CF_BAD || ex == CF_BAD || (!zero && (e < CF_SMIN || e > CF_SMAX))) bad[g] = 1;
      }
    }
    __syncthreads();
    if (row) {
      CfAcc k1[RG], k2[RG], k3[RG];
#pragma unroll
      for (int g = 0; g < RG; ++g) k1[g] = k2[g] = k3[g] = CfAcc{0, 0};
      const int4* xg = sx + d * n;
      const int2* sg = ss + d * n;
#pragma unroll 4
      for (int c = 0; c < n; ++c) {
        const int4 a = Wj[c * NR];                   // sums and differences word by word
        const int dl = a.z - a.x, dh = a.w - a.y, sl = a.x + a.z, sh = a.y + a.w;
#pragma unroll
        for (int g = 0; g < RG; ++g) {
          const int4 x = xg[g * NR + c];
          const int2 s = sg[g * NR + c];
          cf_mac(k1[g], a.x, a.y, s.x, s.y);
          cf_mac(k2[g], dl, dh, x.x, x.y);
          cf_mac(k3[g], sl, sh, x.z, x.w);
        }
      }
#pragma unroll
      for (int g = 0; g < RG; ++g) {
        const long long v1 = cf_value(k1[g]);
        sp[g * NR + q] = make_longlong2(v1 - cf_value(k3[g]), v1 + cf_value(k2[g]));
      }
    }
    __syncthreads();
    for (int o = tid; o < RG * n; o += blockDim.x) {
      const int g = o / n, orow = o - g * n;
      if (r0 + g >= r1) break;
      cf_output(in, out, A + (long long)j * NR * n, Lx, Lt, n, j, r0 + g, orow, bad[g], sp + g * NR,
                pe + g * NR, ep);
    }
  }
}

template <int RG>
cudaError_t launch(const double2* x, double2* y, const double2* A, const int4* W, const int* E, int Lx,
                   int Lt, int n, int nrhs, int rpc, const Epilogue& ep, cudaStream_t s) {
  const int NR = 9 * n;
  const size_t smem = (size_t)RG * (NR * (16 + 16 + 8 + 4) + 40);   // at most 51 KB
  static SmemLimit limit;
  const cudaError_t e = limit.raise(k_coarse_fx<RG>, 64 * 1024);
  if (e != cudaSuccess) return e;
  launch_after(k_coarse_fx<RG>, dim3(Lx * Lt, (nrhs + rpc - 1) / rpc), (NR + 31) & ~31, smem, s, x, y, A, W,
               E, Lx, Lt, n, nrhs, rpc, ep);
  return cudaGetLastError();
}

}  // namespace

long long coarse_words_bytes(long long sites, int n) {
  return n <= CF_NMAX ? sites * 9 * n * (n * (long long)sizeof(int4) + (long long)sizeof(int)) : 0;
}

cudaError_t coarse_finish(const void* G0, const void* G1, double m, void* A64, void* A32, void* A16,
                          void* words, long long sites, int n, cudaStream_t s) {
  int4* W = (int4*)words;
  int* E = W ? (int*)(W + sites * 9 * n * n) : nullptr;
  const size_t smem = W ? (size_t)9 * n * (n | 1) * sizeof(int4) : 0;   // at most 152 KB
  int P = 2;
  while (P < n) P *= 2;
  if (P > 256) return cudaErrorInvalidValue;
  static SmemLimit limit0, limit1;
  const cudaError_t e = G0 ? limit1.raise(k_coarse_finish<true>, 160 * 1024)
                           : limit0.raise(k_coarse_finish<false>, 160 * 1024);
  if (e != cudaSuccess) return e;
  if (G0)
    launch_after(k_coarse_finish<true>, (unsigned)sites, 256, smem, s, (const double2*)G0, (const double2*)G1,
                 m, (double2*)A64, (float2*)A32, (__nv_bfloat162*)A16, W, E, n, P);
  else
    launch_after(k_coarse_finish<false>, (unsigned)sites, 256, smem, s, nullptr, nullptr, 0.0, (double2*)A64,
                 (float2*)A32, (__nv_bfloat162*)A16, W, E, n, P);
  count_launch();
  return cudaGetLastError();
}

cudaError_t coarse_apply_fx(const void* in, void* out, const void* A64, const void* words, int Lx, int Lt,
                            int n, int nrhs, const Epilogue& ep, cudaStream_t s) {
  const double2 *x = (const double2*)in, *a = (const double2*)A64;
  const int4* W = (const int4*)words;
  const int* E = (const int*)(W + (long long)Lx * Lt * 9 * n * n);
  // up to 8 right-hand sides per CTA beyond 8 (4, 8 and 16 measure within 5%)
  const cudaError_t e =
      nrhs == 1 ? launch<1>(x, (double2*)out, a, W, E, Lx, Lt, n, 1, 1, ep, s)
                : launch<4>(x, (double2*)out, a, W, E, Lx, Lt, n, nrhs, nrhs > 8 ? 8 : 4, ep, s);
  count_launch();
  return e;
}

}  // namespace mgk
