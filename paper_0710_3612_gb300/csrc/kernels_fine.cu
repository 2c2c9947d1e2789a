// Fine-lattice Wilson-Dirac operator D and D^dagger (Sec. 1 of the paper,
// display after Eq. 1), 2D, U(1) links, gamma_1 = sigma_1 (x), gamma_2 =
// sigma_2 (t), diagonal 4 + m, t antiperiodic (sign folded into the t link at
// t = Lt - 1 by fold_links).
//
// Spin projection: (1 - s sigma_1) phi = (phi0 - s phi1) (1, -s)^T and
// (1 - s sigma_2) phi = (phi0 + i s phi1) (1, -i s)^T, so each hop is one
// complex projection, one link multiply and a rank-1 reconstruction.
// D uses s = +1 forward (x + mu) and s = -1 backward; D^dagger swaps them.
#include <map>
#include <mutex>
#include <tuple>

#include "kernels.h"
#include "wilson.cuh"

namespace mgk {

template <typename R, bool DAG>
__global__ void __launch_bounds__(256) k_wilson_D(const cplx_t<R>* __restrict__ in,
                                                  cplx_t<R>* __restrict__ out,
                                                  const cplx_t<R>* __restrict__ U, R diag, int Lx,
                                                  int Lt, int dependent) {
  pdl_wait(dependent, in, out, U);
  const int V = Lx * Lt;
  const int site = blockIdx.x * blockDim.x + threadIdx.x;
  if (site >= V) return;
  const long long off = (long long)blockIdx.y * V * 2;
  cplx_t<R> o0, o1;
  wilson_site<R, DAG>(in + off, U, diag, site % Lx, site / Lx, Lx, Lt, o0, o1);
  out[off + 2 * site] = o0;
  out[off + 2 * site + 1] = o1;
}

template <typename R>
cudaError_t wilson_D(const void* in, void* out, const void* U, double diag, int Lx, int Lt,
                     int nrhs, bool dagger, cudaStream_t s) {
  const int V = Lx * Lt;
  dim3 grid((V + 255) / 256, nrhs);
  if (dagger)
    launch_after(k_wilson_D<R, true>, grid, 256, 0, s, (const cplx_t<R>*)in, (cplx_t<R>*)out,
                 (const cplx_t<R>*)U, (R)diag, Lx, Lt);
  else
    launch_after(k_wilson_D<R, false>, grid, 256, 0, s, (const cplx_t<R>*)in, (cplx_t<R>*)out,
                 (const cplx_t<R>*)U, (R)diag, Lx, Lt);
  count_launch();
  return cudaGetLastError();
}

// Fused A = D^dagger D.  A CTA of TX x TY threads owns a TX x (TY * RPT) tile
// of output sites (each thread RPT sites of one column).  It stages psi on the
// tile plus a 2-site halo and the links on the tile plus a 2-site halo below /
// 1-site halo above in shared memory, forms D psi on the tile plus a 1-site
// halo, and applies D^dagger to it -- one pass over psi and the links.
// Coordinates wrap periodically (the antiperiodic sign sits in the links), so
// lattices that are not multiples of the tile work unchanged.
// Tile geometry: TX x (TY * RPT) sites per CTA of TX x TY threads.  Large
// lattices use 32 x 16 (FP32, two rows per thread) or 32 x 8 (FP64, shared
// memory below 48 KB); lattices with fewer than two tiles per SM use 16 x 8
// tiles so that every SM gets work.

template <typename R, int TX, int TY, int RPT>
__global__ void __launch_bounds__(TX* TY) k_wilson_A(const cplx_t<R>* __restrict__ in,
                                                     cplx_t<R>* out,
                                                     const cplx_t<R>* __restrict__ U, R diag,
                                                     int Lx, int Lt, Epilogue ep, int dependent) {
  pdl_wait(dependent, in, out, U);
  constexpr int TT = TY * RPT;
  constexpr int PW = TX + 4, PH = TT + 4;     // psi region [-2, TX+1] x [-2, TT+1]
  constexpr int DW = TX + 2, DH = TT + 2;     // D psi region [-1, TX] x [-1, TT]
  constexpr int UW = TX + 3, UH = TT + 3;     // link region [-2, TX] x [-2, TT]
  using C = cplx_t<R>;
  using S = typename spinor_t<R>::type;
  __shared__ S sp[PH * PW];
  __shared__ S sd[DH * DW];
  __shared__ C su[UH * UW][2];
  const int V = Lx * Lt;
  const int x0 = blockIdx.x * TX, t0 = blockIdx.y * TT;
  const long long off = (long long)blockIdx.z * V * 2;
  const int tid = threadIdx.x;
  for (int q = tid; q < PH * PW; q += TX * TY) {
    const int gx = wrap_tile(x0 + q % PW - 2, Lx), gt = wrap_tile(t0 + q / PW - 2, Lt);
    sp[q] = ld_spinor(in + off + 2LL * (gx + Lx * gt));
  }
  for (int q = tid; q < UH * UW; q += TX * TY) {
    const int gx = wrap_tile(x0 + q % UW - 2, Lx), gt = wrap_tile(t0 + q / UW - 2, Lt);
    const int g = gx + Lx * gt;
    su[q][0] = U[g];
    su[q][1] = U[V + g];
  }
  __syncthreads();
  // D psi on [-1, TX] x [-1, TT]
  for (int q = tid; q < DH * DW; q += TX * TY) {
    const int lx = q % DW - 1, lt = q / DW - 1;
    const int pc = (lt + 2) * PW + (lx + 2);
    const int uc = (lt + 2) * UW + (lx + 2);
    C a0 = mk((R)0, (R)0), a1 = mk((R)0, (R)0), f0, f1;
    split(sp[pc + 1], f0, f1);
    hop_x<R>(a0, a1, su[uc][0], f0, f1, (R)1);
    split(sp[pc - 1], f0, f1);
    hop_x<R>(a0, a1, cconj(su[uc - 1][0]), f0, f1, (R)-1);
    split(sp[pc + PW], f0, f1);
    hop_t<R>(a0, a1, su[uc][1], f0, f1, (R)1);
    split(sp[pc - PW], f0, f1);
    hop_t<R>(a0, a1, cconj(su[uc - UW][1]), f0, f1, (R)-1);
    split(sp[pc], f0, f1);
    sd[q] = join(mk(diag * f0.x - (R)0.5 * a0.x, diag * f0.y - (R)0.5 * a0.y),
                 mk(diag * f1.x - (R)0.5 * a1.x, diag * f1.y - (R)0.5 * a1.y));
  }
  __syncthreads();
  // D^dagger on the tile, then the epilogue
  const int lx = tid % TX;
  const int gx = x0 + lx;
  const R ca = (R)ep.ca, cu = (R)ep.cu, cw = (R)ep.cw;
  const C* EU = (const C*)ep.U;
  const C* EW = (const C*)ep.W;
  double zq = 0.0, rz = 0.0;     // the dot (a site's sum in the stencil's precision) or the flexible-CG pair
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    const int lt = tid / TX + TY * k;
    const int gt = t0 + lt;
    if (gx >= Lx || gt >= Lt) continue;
    const int dc = (lt + 1) * DW + (lx + 1);
    const int uc = (lt + 2) * UW + (lx + 2);
    C a0 = mk((R)0, (R)0), a1 = mk((R)0, (R)0), f0, f1;
    split(sd[dc + 1], f0, f1);
    hop_x<R>(a0, a1, su[uc][0], f0, f1, (R)-1);
    split(sd[dc - 1], f0, f1);
    hop_x<R>(a0, a1, cconj(su[uc - 1][0]), f0, f1, (R)1);
    split(sd[dc + DW], f0, f1);
    hop_t<R>(a0, a1, su[uc][1], f0, f1, (R)-1);
    split(sd[dc - DW], f0, f1);
    hop_t<R>(a0, a1, cconj(su[uc - UW][1]), f0, f1, (R)1);
    split(sd[dc], f0, f1);
    C y0 = mk(diag * f0.x - (R)0.5 * a0.x, diag * f0.y - (R)0.5 * a0.y);
    C y1 = mk(diag * f1.x - (R)0.5 * a1.x, diag * f1.y - (R)0.5 * a1.y);
    const long long g = off + 2LL * (gx + Lx * gt);
    if (ep.dot_out && !ep.zq_q) {
      C p0, p1;
      split(sp[(lt + 2) * PW + (lx + 2)], p0, p1);
      zq += (double)(p0.x * y0.x + p0.y * y0.y + p1.x * y1.x + p1.y * y1.y);
      rz += (double)(p0.x * y0.y - p0.y * y0.x + p1.x * y1.y - p1.y * y1.x);
    }
    y0 = mk(ca * y0.x, ca * y0.y);
    y1 = mk(ca * y1.x, ca * y1.y);
    if (EU) {
      const S u = ld_spinor(EU + g);
      C u0, u1;
      split(u, u0, u1);
      y0 = mk(y0.x + cu * u0.x, y0.y + cu * u0.y);
      y1 = mk(y1.x + cu * u1.x, y1.y + cu * u1.y);
    }
    if (EW) {
      const S w = ld_spinor(EW + g);
      C w0, w1;
      split(w, w0, w1);
      y0 = mk(y0.x + cw * w0.x, y0.y + cw * w0.y);
      y1 = mk(y1.x + cw * w1.x, y1.y + cw * w1.y);
    }
    if (ep.zq_q) {
      const double2* Q = (const double2*)ep.zq_q + g;
      const double2* Rv = (const double2*)ep.zq_r + g;
      const double2 q0 = Q[0], q1 = Q[1], r0 = Rv[0], r1 = Rv[1];
      zq += (double)y0.x * q0.x + (double)y0.y * q0.y + (double)y1.x * q1.x + (double)y1.y * q1.y;
      rz += r0.x * (double)y0.x + r0.y * (double)y0.y + r1.x * (double)y1.x + r1.y * (double)y1.y;
    }
    st_spinor(out + g, join(y0, y1));
  }
  if (ep.dot_out) {
    // the tile's shared memory is free again: it holds the block sums
    static_assert(sizeof(sp) >= 2 * TX * TY * sizeof(double), "room for the block sums");
    __syncthreads();
    finish_reduction_g<2>(zq, rz, ep.dot_ws, ep.dot_out, (double*)sp, blockIdx.z,
                          blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y);
  }
}

// Register-streaming A = D^dagger D on FP64 vectors for large lattices (masses the integer
// kernel does not take).  A warp owns a strip
// of 32 consecutive x sites (lanes 2..29 produce output, lanes 0, 1, 30, 31
// are halo) and marches along t over SROWS output rows, keeping three rows of
// psi, two rows of D psi and the needed link rows in registers; x neighbours
// come from warp shuffles, t neighbours from the row window.  No shared
// memory and no block barriers: every loaded byte is used from registers.
// Row r + 2 of psi and the links of row r + 1 are prefetched one step ahead.
static constexpr int SROWS = 32;
static constexpr int SOUT = 28;            // output lanes per warp

template <typename C>
__device__ __forceinline__ C shfl_c(C v, int delta, bool up) {
  C r;
  if (up) {
    r.x = __shfl_up_sync(0xffffffffu, v.x, delta);
    r.y = __shfl_up_sync(0xffffffffu, v.y, delta);
  } else {
    r.x = __shfl_down_sync(0xffffffffu, v.x, delta);
    r.y = __shfl_down_sync(0xffffffffu, v.y, delta);
  }
  return r;
}

// D (sf = +1) or D^dagger (sf = -1) at this lane's site for one row: (f0, f1)
// the row's spinor, fu / fd the rows t+1 / t-1 at this x, ux and ut the links
// here, utm the t link one row below; the x-hop terms come from the adjacent
// lanes.
template <typename R>
__device__ __forceinline__ void dslash_row(cplx_t<R> f0, cplx_t<R> f1, cplx_t<R> fu0,
                                           cplx_t<R> fu1, cplx_t<R> fd0, cplx_t<R> fd1,
                                           cplx_t<R> ux, cplx_t<R> ut, cplx_t<R> utm, R diag,
                                           R sf, cplx_t<R>& o0, cplx_t<R>& o1) {
  using C = cplx_t<R>;
  // x hops: each lane forms the projections of its own site and the lane
  // x - 1 also applies its link, so only one complex per direction moves.
  const C q = mk(f0.x - sf * f1.x, f0.y - sf * f1.y);               // (1 - sf s1) projection
  const C g = cmul(cconj(ux), mk(f0.x + sf * f1.x, f0.y + sf * f1.y));
  const C qn = shfl_c(q, 1, false);                                 // from x + 1
  const C gp = shfl_c(g, 1, true);                                  // U_x(x-1)^* (...)(x - 1)
  const C hf = cmul(ux, qn);
  C a0 = cadd(hf, gp);
  C a1 = mk(-sf * hf.x + sf * gp.x, -sf * hf.y + sf * gp.y);
  hop_t<R>(a0, a1, ut, fu0, fu1, sf);
  hop_t<R>(a0, a1, cconj(utm), fd0, fd1, -sf);
  o0 = mk(diag * f0.x - (R)0.5 * a0.x, diag * f0.y - (R)0.5 * a0.y);
  o1 = mk(diag * f1.x - (R)0.5 * a1.x, diag * f1.y - (R)0.5 * a1.y);
}

// Asynchronous row prefetch for the streaming stencil: each lane copies its
// own spinor and links of a future row into a per-warp ring of SNB slots in
// shared memory (cp.async), SNB - 1 iterations ahead of use.
static constexpr int SNB = 4;

__global__ void __launch_bounds__(128, 3) k_wilson_A_stream(const double2* __restrict__ in, double2* out,
                                                           const double2* __restrict__ U, double diag,
                                                           int Lx, int Lt, Epilogue ep, int dependent) {
  pdl_wait(dependent, in, out, U);
  using R = double;
  using C = double2;
  using S = double4_32a;
  __shared__ S ring_psi[4][SNB][32];           // [warp][slot][lane]
  __shared__ C ring_u[4][SNB][32][2];
  const int V = Lx * Lt;
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const int strips = (Lx + SOUT - 1) / SOUT;
  const int w = blockIdx.x * (blockDim.x >> 5) + wl;
  const int row_blocks = (Lt + SROWS - 1) / SROWS;
  if (w >= strips * row_blocks) return;                  // whole warp
  const int strip = w % strips, t0 = (w / strips) * SROWS;
  const int xu = strip * SOUT - 2 + lane;                // unwrapped x
  const int x = wrap(xu, Lx);
  const bool writer = lane >= 2 && lane < 30 && xu < Lx;
  const long long off = (long long)blockIdx.y * V * 2;
  const int t1 = min(t0 + SROWS, Lt);                    // output rows [t0, t1)
  auto ld_psi = [&](int t, C& a, C& b) {
    split(ld_spinor(in + off + 2LL * (x + Lx * wrap(t, Lt))), a, b);
  };
  auto ld_u = [&](int t, C& ux, C& ut) {
    const int g = x + Lx * wrap(t, Lt);
    ux = U[g];
    ut = U[V + g];
  };
  // group for loop step r: psi(r + 2) and links(r + 1), into slot
  // (r - t0 + 1) mod SNB; empty past the last step that reads one
  auto issue = [&](int r) {
    if (r < t1) {
      const int slot = (r - t0 + 1 + SNB) % SNB;
      const C* ps = in + off + 2LL * (x + Lx * wrap(r + 2, Lt));
      char* dst = (char*)&ring_psi[wl][slot][lane];
      cp_async16(dst, ps);
      cp_async16(dst + 16, ps + 1);
      const int g = x + Lx * wrap(r + 1, Lt);
      cp_async16(&ring_u[wl][slot][lane][0], U + g);
      cp_async16(&ring_u[wl][slot][lane][1], U + V + g);
    }
    cp_commit();
  };
  C pm0, pm1, pc0, pc1, pp0, pp1;          // psi rows r-1, r, r+1
  C dm0, dm1, dc0, dc1;                    // D psi rows r-2, r-1
  C uxc, utc, utm;                         // U_x(r), U_t(r), U_t(r-1)
  C uxo, uto, utmo;                        // the same one row earlier (for D^dagger)
  C dummy;
  ld_psi(t0 - 2, pm0, pm1);
  ld_psi(t0 - 1, pc0, pc1);
  ld_psi(t0, pp0, pp1);
  ld_u(t0 - 2, dummy, utm);
  ld_u(t0 - 1, uxc, utc);
  for (int k = 0; k < SNB - 1; ++k) issue(t0 - 1 + k);
  dm0 = dm1 = dc0 = dc1 = mk((R)0, (R)0);
  uxo = uto = utmo = mk((R)0, (R)0);
  const R ca = (R)ep.ca, cu = (R)ep.cu, cw = (R)ep.cw;
  const C* EU = (const C*)ep.U;
  const C* EW = (const C*)ep.W;
  for (int r = t0 - 1; r <= t1; ++r) {
    C e0, e1;                                            // D psi at row r
    dslash_row<R>(pc0, pc1, pp0, pp1, pm0, pm1, uxc, utc, utm, diag, (R)1, e0, e1);
    if (r >= t0 + 1) {                                   // output row r - 1
      C o0, o1;
      dslash_row<R>(dc0, dc1, e0, e1, dm0, dm1, uxo, uto, utmo, diag, (R)-1, o0, o1);
      if (writer) {
        const long long g = off + 2LL * (x + Lx * (r - 1));
        o0 = mk(ca * o0.x, ca * o0.y);
        o1 = mk(ca * o1.x, ca * o1.y);
        if (EU) {
          C u0, u1;
          split(ld_spinor(EU + g), u0, u1);
          o0 = mk(o0.x + cu * u0.x, o0.y + cu * u0.y);
          o1 = mk(o1.x + cu * u1.x, o1.y + cu * u1.y);
        }
        if (EW) {
          C w0, w1;
          split(ld_spinor(EW + g), w0, w1);
          o0 = mk(o0.x + cw * w0.x, o0.y + cw * w0.y);
          o1 = mk(o1.x + cw * w1.x, o1.y + cw * w1.y);
        }
        st_spinor(out + g, join(o0, o1));
      }
    }
    dm0 = dc0; dm1 = dc1; dc0 = e0; dc1 = e1;            // shift: row r becomes r - 1
    uxo = uxc; uto = utc; utmo = utm;
    pm0 = pc0; pm1 = pc1; pc0 = pp0; pc1 = pp1;
    utm = utc;
    if (r + 1 <= t1) {                                   // psi(r + 2), links(r + 1)
      cp_wait<SNB - 2>();
      const int slot = (r - t0 + 1 + SNB) % SNB;
      split(ring_psi[wl][slot][lane], pp0, pp1);
      uxc = ring_u[wl][slot][lane][0];
      utc = ring_u[wl][slot][lane][1];
    }
    issue(r + SNB - 1);
  }
  cp_wait<0>();
}

// Register-streaming A on FP32 vectors, two sites per lane.  Both sites of a lane go through
// every operation together as packed pairs (fma.rn.f32x2: one issue slot for two FMAs), so a
// row step takes 40 packed operations for two sites where k_wilson_A_stream takes 88, and
// only one shuffle per component and direction; a warp owns 64 sites of a row, 60 of them
// outputs.  Its links are stored as -U / 2, so that D is diag psi + the sum of hops and nothing
// leaves the range that the result has.  The t-backward product of a row is formed when the row
// is current and carried.  Bound by FMA issue (72% of the heavy pipe) and HBM: 4096^2 128 us (0.93
// of the copy bandwidth; 144 us with one site per lane), 1024^2 x 16 117 (146), 256^2 x 64 40 (68
// with tiles).
using P2 = unsigned long long;                       // two floats, low = first site

__device__ __forceinline__ P2 p2(float a, float b) {
  P2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lo(P2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi(P2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) {
  P2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ P2 mul2(P2 a, P2 b) {
  P2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ P2 add2(P2 a, P2 b) {
  P2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ P2 sub2(P2 a, P2 b) { return fma2(b, 0xBF800000BF800000ull, a); }

struct C2 { P2 x, y; };                              // complex numbers of two sites
struct S2 { C2 a, b; };                              // their spinors
struct L2 { P2 x, y, n; };                           // their links: re, im, -im

__device__ __forceinline__ C2 add2(C2 a, C2 b) { return {add2(a.x, b.x), add2(a.y, b.y)}; }
__device__ __forceinline__ C2 sub2(C2 a, C2 b) { return {sub2(a.x, b.x), sub2(a.y, b.y)}; }
__device__ __forceinline__ C2 mul2(const L2& u, C2 h) {
  return {fma2(u.n, h.y, mul2(u.x, h.x)), fma2(u.y, h.x, mul2(u.x, h.y))};
}
__device__ __forceinline__ C2 mulc2(const L2& u, C2 h) {   // conj(u) h
  return {fma2(u.y, h.y, mul2(u.x, h.x)), fma2(u.n, h.x, mul2(u.x, h.y))};
}
__device__ __forceinline__ S2 spinors(float4 p, float4 q) {
  return {{p2(p.x, q.x), p2(p.y, q.y)}, {p2(p.z, q.z), p2(p.w, q.w)}};
}
__device__ __forceinline__ L2 links(float4 u) {
  const P2 y = p2(u.y, u.w);
  return {p2(u.x, u.z), y, y ^ 0x8000000080000000ull};
}
// f0 + i s f1
template <int S>
__device__ __forceinline__ C2 proj_t(const S2& f) {
  return S > 0 ? C2{sub2(f.a.x, f.b.y), add2(f.a.y, f.b.x)} : C2{add2(f.a.x, f.b.y), sub2(f.a.y, f.b.x)};
}
// the pair one site to the right / left of each site's value
__device__ __forceinline__ P2 from_right(P2 v) { return p2(hi(v), __shfl_down_sync(0xffffffffu, lo(v), 1)); }
__device__ __forceinline__ P2 from_left(P2 v) { return p2(__shfl_up_sync(0xffffffffu, hi(v), 1), lo(v)); }

// D (S = 1) or D^dagger (S = -1) of one row; f the row, up the next one, tb the t-backward
// product, ux and ut the links times -1/2.
template <int S>
__device__ __forceinline__ S2 row2(const S2& f, const S2& up, const L2& ux, const L2& ut, C2 tb, P2 diag) {
  const C2 q = S > 0 ? sub2(f.a, f.b) : add2(f.a, f.b);
  const C2 g = mulc2(ux, S > 0 ? add2(f.a, f.b) : sub2(f.a, f.b));
  const C2 X = mul2(ux, C2{from_right(q.x), from_right(q.y)});
  const C2 Y = {from_left(g.x), from_left(g.y)};
  const C2 Z = mul2(ut, proj_t<S>(up));
  const C2 s = add2(add2(add2(X, Y), Z), tb);
  const C2 d = S > 0 ? sub2(Y, X) : sub2(X, Y), e = S > 0 ? sub2(Z, tb) : sub2(tb, Z);
  return {{fma2(diag, f.a.x, s.x), fma2(diag, f.a.y, s.y)},
          {fma2(diag, f.b.x, add2(d.x, e.y)), fma2(diag, f.b.y, sub2(d.y, e.x))}};
}

static constexpr int SOUT2 = 60;           // output sites per warp

__global__ void __launch_bounds__(128, 4) k_wilson_A_stream2(const float2* __restrict__ in, float2* out,
                                                             const float2* __restrict__ W, float diag,
                                                             int Lx, int Lt, int rows, Epilogue ep, int dependent) {
  pdl_wait(dependent, in, out, W);
  __shared__ float4 ring_psi[4][SNB][2][32];           // [warp][slot][site][lane]
  __shared__ float4 ring_u[4][SNB][2][32];             // [warp][slot][direction][lane]
  const int V = Lx * Lt;
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
  const int strips = (Lx + SOUT2 - 1) / SOUT2, row_blocks = (Lt + rows - 1) / rows;
  const int w = blockIdx.x * 4 + wl;
  if (w >= strips * row_blocks) return;                // whole warp
  const int strip = w % strips, t0 = (w / strips) * rows, t1 = min(t0 + rows, Lt);
  const int xu = strip * SOUT2 - 2 + 2 * lane;
  const int x = min(wrap(xu, Lx), Lx - 2);             // Lx is even: both sites wrap together
  const bool writer = lane >= 1 && lane < 31 && xu < Lx;
  const long long off = (long long)blockIdx.y * V * 2;
  const float2* col = in + off + 2 * x;
  auto issue = [&](int r) {                            // psi(r + 2) and links(r + 1) for step r
    if (r < t1) {
      const int slot = (r - t0 + 1 + SNB) % SNB;
      const float2* ps = col + 2LL * Lx * wrap(r + 2, Lt);
      cp_async16(&ring_psi[wl][slot][0][lane], ps);
      cp_async16(&ring_psi[wl][slot][1][lane], ps + 2);
      const float2* pu = W + x + Lx * wrap(r + 1, Lt);
      cp_async16(&ring_u[wl][slot][0][lane], pu);
      cp_async16(&ring_u[wl][slot][1][lane], pu + V);
    }
    cp_commit();
  };
  auto ld_psi = [&](int t) {
    const float4* p = (const float4*)(col + 2LL * Lx * wrap(t, Lt));
    return spinors(p[0], p[1]);
  };
  auto ld_u = [&](int mu, int t) { return links(*(const float4*)(W + mu * V + x + Lx * wrap(t, Lt))); };
  for (int k = 0; k < SNB - 1; ++k) issue(t0 - 1 + k);
  const P2 d2 = p2(diag, diag);
  C2 tb = mulc2(ld_u(1, t0 - 2), proj_t<-1>(ld_psi(t0 - 2)));
  S2 pc = ld_psi(t0 - 1), pp = ld_psi(t0), dc = {{0, 0}, {0, 0}};
  L2 ux = ld_u(0, t0 - 1), ut = ld_u(1, t0 - 1), uxo = {0, 0, 0}, uto = {0, 0, 0};
  C2 db = {0, 0};
  const float ca = (float)ep.ca, cu = (float)ep.cu, cw = (float)ep.cw;
  const float2 *EU = (const float2*)ep.U, *EW = (const float2*)ep.W;
#pragma unroll 2                                       // the row window rotates by renaming
  for (int r = t0 - 1; r <= t1; ++r) {
    const S2 e = row2<1>(pc, pp, ux, ut, tb, d2);      // D psi at row r
    if (r > t0) {                                      // output row r - 1
      const S2 y = row2<-1>(dc, e, uxo, uto, db, d2);
      if (writer) {
        const long long g = off + 2LL * (x + Lx * (r - 1));
        const P2 c = p2(ca, ca);
        S2 o = {{mul2(c, y.a.x), mul2(c, y.a.y)}, {mul2(c, y.b.x), mul2(c, y.b.y)}};
        auto axpy = [&](float k, const float2* v) {
          const float4* p = (const float4*)(v + g);
          const S2 u = spinors(p[0], p[1]);
          const P2 kk = p2(k, k);
          o = {{fma2(kk, u.a.x, o.a.x), fma2(kk, u.a.y, o.a.y)}, {fma2(kk, u.b.x, o.b.x), fma2(kk, u.b.y, o.b.y)}};
        };
        if (EU) axpy(cu, EU);
        if (EW) axpy(cw, EW);
        float4* po = (float4*)(out + g);
        po[0] = make_float4(lo(o.a.x), lo(o.a.y), lo(o.b.x), lo(o.b.y));
        po[1] = make_float4(hi(o.a.x), hi(o.a.y), hi(o.b.x), hi(o.b.y));
      }
    }
    db = mulc2(uto, proj_t<1>(dc));                    // into D^dagger's row r
    tb = mulc2(ut, proj_t<-1>(pc));                    // into D's row r + 1
    dc = e;
    uxo = ux;
    uto = ut;
    pc = pp;
    if (r < t1) {                                      // psi(r + 2), links(r + 1)
      cp_wait<SNB - 2>();
      const int slot = (r - t0 + 1 + SNB) % SNB;
      pp = spinors(ring_psi[wl][slot][0][lane], ring_psi[wl][slot][1][lane]);
      ux = links(ring_u[wl][slot][0][lane]);
      ut = links(ring_u[wl][slot][1][lane]);
    }
    issue(r + SNB - 1);
  }
  cp_wait<0>();
}

// The FP64 streaming kernel serves lattices with enough strips to fill the GPU.
static bool streamed64(int Lx, int Lt) {
  const long long warps = (long long)((Lx + SOUT - 1) / SOUT) * ((Lt + SROWS - 1) / SROWS);
  return Lx >= 64 && Lt >= 2 * SROWS && warps >= 4LL * 152;
}

// The FP32 one: launches with 12 warps per SM at 8 rows each (at 256^2 x 16 it takes 16.4 us
// against 18.6 with tiles, at 512^2 x 4 14.1 against 18.5, at 512^2 8.2 against 8.3), then the
// most rows per warp that leave two rounds of 16 warps per SM: more rows repeat less of the
// 4-row halo (1024^2 x 16: 133, 121, 119 us with 8, 16, 32), fewer fill the GPU (256^2 x 64:
// 41, 40, 43 us).
static long long stream32_warps(int Lx, int Lt, int nrhs, int rows) {
  return (long long)((Lx + SOUT2 - 1) / SOUT2) * ((Lt + rows - 1) / rows) * nrhs;
}
static bool streamed32(int Lx, int Lt, int nrhs) {
  return Lx >= 64 && Lt >= 16 && stream32_warps(Lx, Lt, nrhs, 8) >= 12LL * 152;
}
static int stream32_rows(int Lx, int Lt, int nrhs) {
  int rows = 32;
  while (rows > 8 && stream32_warps(Lx, Lt, nrhs, rows) < 2LL * 16 * 152) rows /= 2;
  return rows;
}

// Tile choice of the fused kernel: 32 x 8 (FP64) or 32 x 16 (FP32) when that
// gives two CTAs per SM, else 16 x 8 (smaller tiles measured slower: more halo).
int wilson_A_ctas(int Lx, int Lt, bool f64) {
  const int big = ((Lx + 31) / 32) * ((Lt + (f64 ? 7 : 15)) / (f64 ? 8 : 16));
  if (big >= 2 * 152) return big;
  return ((Lx + 15) / 16) * ((Lt + 7) / 8);
}

template <typename R, int TX, int TY, int RPT>
static void launch_wilson_A(const void* in, void* out, const void* U, double diag, int Lx, int Lt,
                            int nrhs, const Epilogue& ep, cudaStream_t s) {
  static_assert(sizeof(R) * 4 * ((TY * RPT + 4) * (TX + 4) + (TY * RPT + 2) * (TX + 2)) +
                        sizeof(R) * 4 * (TY * RPT + 3) * (TX + 3) <= 48 * 1024,
                "tile above the static shared-memory limit");
  dim3 grid((Lx + TX - 1) / TX, (Lt + TY * RPT - 1) / (TY * RPT), nrhs);
  launch_after(k_wilson_A<R, TX, TY, RPT>, grid, TX * TY, 0, s, (const cplx_t<R>*)in, (cplx_t<R>*)out,
               (const cplx_t<R>*)U, (R)diag, Lx, Lt, ep);
}

// ---------------------------------------------------------------------------
// Launch shapes of the fused A and their autotuner.  A shape is admitted by the
// tuner only if it reproduces the default shape's output bit for bit: the tiles
// share their per-site arithmetic (wilson_site order), the integer kernel's do not
// depend on the tile; the FP32 streaming kernel associates its sums otherwise and
// is admitted only where it is the default (wide lattices and batches, so that an
// FP32 result's last bits may depend on the number of right-hand sides).  The
// tuner keeps the fastest admitted shape per (precision, Lx, Lt, nrhs) when it
// beats the default shape by more than 3%; it takes 62 launches of every admitted
// shape in the first set-up of a shape in a process.
// Launches with the fused <in, A in> epilogue keep the default shape (their
// partial sums depend on the tiling).
// ---------------------------------------------------------------------------
enum { WV_STREAM = 0, WV_16x8, WV_32x8, WV_32x8x2, WV_16x16, WV_64x4, WV_64x4x2, WV_COUNT };
static const int WV_SHAPE[WV_COUNT][3] = {{0, 0, 0}, {16, 8, 1}, {32, 8, 1}, {32, 8, 2},
                                          {16, 16, 1}, {64, 4, 1}, {64, 4, 2}};

// The default shape (the choice made before any tuning).  A fused dot keeps its tile
// whatever the tuner finds, so batches of it count all their tiles.
template <typename R>
static int wilson_default_variant(int Lx, int Lt, int nrhs, bool dot) {
  const bool f64 = sizeof(R) == 8;
  if (!dot && (f64 ? streamed64(Lx, Lt) : streamed32(Lx, Lt, nrhs))) return WV_STREAM;
  const long long tiles = (long long)((Lx + 31) / 32) * ((Lt + (f64 ? 7 : 15)) / (f64 ? 8 : 16));
  const bool big = tiles * (dot ? nrhs : 1) >= 2 * 152;
  if (!big) return WV_16x8;
  return f64 ? WV_32x8 : WV_32x8x2;
}

// FP64 vectors whose operator the integer kernel takes (wilson_A_fx_ok): its tiles
// by the number of sites in the launch.  Measured (us, 16 x 8 / 32 x 8 / 32 x 16):
// 128^2 6.2 / 6.3 / 8.3, 256^2 8.2 / 8.2 / 8.3, 512^2 18.2 / 16.4 / 16.5, 256^2 x 64
// 237 / 191 / 172; with the fused dot 256^2 12.4 / 11.3 / 12.4, 210 x 90 x 12
// 25.0 / 21.7 / 22.5, 256^2 x 64 325 / 251 / 207.  Small tiles spread few sites over
// the SMs, large ones repeat less of the halo.  The fused dot takes at most 608 tiles.
static int wilson_fx_variant(int Lx, int Lt, int nrhs, bool dot) {
  const long long sites = (long long)Lx * Lt * nrhs;
  int v = sites < (1 << 16) ? WV_16x8 : sites < (1 << 18) ? WV_32x8 : WV_32x8x2;
  auto tiles = [&](int k) {
    const int ty = WV_SHAPE[k][1] * WV_SHAPE[k][2];
    return ((Lx + WV_SHAPE[k][0] - 1) / WV_SHAPE[k][0]) * ((Lt + ty - 1) / ty);
  };
  while (dot && tiles(v) > 608 && v != WV_32x8x2) v = v == WV_16x8 ? WV_32x8 : WV_32x8x2;
  return v;
}

bool wilson_A_dot_fits(int Lx, int Lt, bool f64, double diag) {
  if (f64 && fixed_diag_ok(diag)) return ((Lx + 31) / 32) * ((Lt + 15) / 16) <= 608;
  return wilson_A_ctas(Lx, Lt, f64) <= 608;
}

template <typename R>
static bool wilson_variant_ok(int v, int Lx, int Lt, int nrhs, bool fx) {
  if (fx) return v == WV_16x8 || v == WV_32x8 || v == WV_32x8x2;
  if (v == WV_STREAM) return sizeof(R) == 8 ? streamed64(Lx, Lt) : streamed32(Lx, Lt, nrhs);
  if (sizeof(R) == 8 && (v == WV_32x8x2 || v == WV_64x4x2)) return false;   // shared memory
  return true;
}

// W: FP64, the fixed-point links when the integer kernel runs the launch, else null; FP32, the
// links times -1/2.
template <typename R>
static cudaError_t launch_variant(int v, const void* in, void* out, const void* U, const void* W,
                                  double diag, int Lx, int Lt, int nrhs, const Epilogue& ep,
                                  cudaStream_t s) {
  if (sizeof(R) == 8 && W)
    return wilson_A_fx(WV_SHAPE[v][0], WV_SHAPE[v][1] * WV_SHAPE[v][2], in, out, U, W, diag, Lx, Lt,
                       nrhs, ep, s);
  switch (v) {
    case WV_STREAM: {
      if constexpr (sizeof(R) == 4) {
        const int rows = stream32_rows(Lx, Lt, nrhs);
        const long long warps = stream32_warps(Lx, Lt, 1, rows);
        launch_after(k_wilson_A_stream2, dim3((unsigned)((warps + 3) / 4), nrhs), 128, 0, s,
                     (const float2*)in, (float2*)out, (const float2*)W, (float)diag, Lx, Lt, rows, ep);
      } else {
        const long long warps = (long long)((Lx + SOUT - 1) / SOUT) * ((Lt + SROWS - 1) / SROWS);
        launch_after(k_wilson_A_stream, dim3((unsigned)((warps + 3) / 4), nrhs), 128, 0, s,
                     (const double2*)in, (double2*)out, (const double2*)U, diag, Lx, Lt, ep);
      }
      break;
    }
    case WV_16x8: launch_wilson_A<R, 16, 8, 1>(in, out, U, diag, Lx, Lt, nrhs, ep, s); break;
    case WV_32x8: launch_wilson_A<R, 32, 8, 1>(in, out, U, diag, Lx, Lt, nrhs, ep, s); break;
    case WV_16x16: launch_wilson_A<R, 16, 16, 1>(in, out, U, diag, Lx, Lt, nrhs, ep, s); break;
    case WV_64x4: launch_wilson_A<R, 64, 4, 1>(in, out, U, diag, Lx, Lt, nrhs, ep, s); break;
    default:
      if constexpr (sizeof(R) == 4) {
        if (v == WV_32x8x2) launch_wilson_A<R, 32, 8, 2>(in, out, U, diag, Lx, Lt, nrhs, ep, s);
        else launch_wilson_A<R, 64, 4, 2>(in, out, U, diag, Lx, Lt, nrhs, ep, s);
      }
      break;
  }
  return cudaGetLastError();
}

struct TuneKey {
  int prec, Lx, Lt, nrhs;
  bool fx;
  bool operator<(const TuneKey& o) const {
    return std::tie(prec, Lx, Lt, nrhs, fx) < std::tie(o.prec, o.Lx, o.Lt, o.nrhs, o.fx);
  }
};
static std::mutex g_tune_mu;
static std::map<TuneKey, StencilTuning> g_tune;

template <typename R>
static int tuned_variant(int Lx, int Lt, int nrhs, bool fx) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  auto it = g_tune.find({(int)sizeof(R), Lx, Lt, nrhs, fx});
  return it == g_tune.end() ? -1 : it->second.variant;
}

__global__ void k_count_diff(const unsigned long long* __restrict__ a,
                             const unsigned long long* __restrict__ b, long long n, int* diff, int dependent) {
  pdl_wait(dependent, a, b, diff);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    if (a[i] != b[i]) atomicAdd(diff, 1);
}

template <typename R>
cudaError_t wilson_A_tune(const void* in, void* out, void* ref, const void* U, const void* W,
                          double diag, int Lx, int Lt, int nrhs, int* dflag, cudaStream_t s) {
  const Epilogue none{};
  const bool fx = sizeof(R) == 8 && wilson_A_fx_ok(W, diag, none);
  if (sizeof(R) == 8 && !fx) W = nullptr;
  const TuneKey key{(int)sizeof(R), Lx, Lt, nrhs, fx};
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    if (g_tune.count(key)) return cudaSuccess;
  }
  const int def = fx ? wilson_fx_variant(Lx, Lt, nrhs, false) : wilson_default_variant<R>(Lx, Lt, nrhs, false);
  const long long words = (long long)Lx * Lt * nrhs * 2 * sizeof(cplx_t<R>) / 8;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  StencilTuning t{};
  t.precision = sizeof(R) == 8 ? 0 : 1;
  t.Lx = Lx; t.Lt = Lt; t.nrhs = nrhs;
  t.variant = def;
  float best = 0.f;
  launch_variant<R>(def, in, ref, U, W, diag, Lx, Lt, nrhs, none, s);
  for (int v = 0; v < WV_COUNT; ++v) {
    if (!wilson_variant_ok<R>(v, Lx, Lt, nrhs, fx)) continue;
    ++t.tried;
    launch_variant<R>(v, in, out, U, W, diag, Lx, Lt, nrhs, none, s);
    int diff = 0;
    cudaMemsetAsync(dflag, 0, sizeof(int), s);
    launch_after(k_count_diff, 152, 256, 0, s, (const unsigned long long*)out, (const unsigned long long*)ref,
                 words, dflag);
    cudaMemcpyAsync(&diff, dflag, sizeof(int), cudaMemcpyDeviceToHost, s);
    cudaError_t err = cudaStreamSynchronize(s);
    if (err != cudaSuccess) {
      cudaEventDestroy(e0);
      cudaEventDestroy(e1);
      return err;
    }
    if (diff) continue;                                    // not bit-identical: never used
    ++t.admitted;
    // the best of three rounds of 20: one round of 10 is off by up to 40% on launches of 5 us
    // (32 CTAs of 64 x 4 x 2 were once chosen for 128^2, 7.6 us against 5.7 in the solve)
    constexpr int REPS = 20;
    for (int w = 0; w < 2; ++w) launch_variant<R>(v, in, out, U, W, diag, Lx, Lt, nrhs, none, s);
    float ms = 0.f;
    for (int round = 0; round < 3; ++round) {
      cudaEventRecord(e0, s);
      for (int w = 0; w < REPS; ++w) launch_variant<R>(v, in, out, U, W, diag, Lx, Lt, nrhs, none, s);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float one = 0.f;
      cudaEventElapsedTime(&one, e0, e1);
      if (round == 0 || one < ms) ms = one;
    }
    const double us = 1000.0 * ms / REPS;
    if (v == def) t.us_default = us;
    if (t.admitted == 1 || ms < best) {
      best = ms;
      t.variant = v;
      t.us_best = us;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  // a timing difference inside the noise of isolated launches does not carry
  // over to launches inside a solve: keep the default unless 3% faster
  if (t.variant != def && !(t.us_best < 0.97 * t.us_default)) {
    t.variant = def;
    t.us_best = t.us_default;
  }
  t.tx = WV_SHAPE[t.variant][0];
  t.ty = WV_SHAPE[t.variant][1];
  t.rpt = WV_SHAPE[t.variant][2];
  {
    std::lock_guard<std::mutex> g(g_tune_mu);
    g_tune[key] = t;
  }
  return cudaGetLastError();
}

int stencil_tunings(StencilTuning* out, int max) {
  std::lock_guard<std::mutex> g(g_tune_mu);
  int k = 0;
  for (const auto& kv : g_tune) {
    if (k < max && out) out[k] = kv.second;
    ++k;
  }
  return k;
}

template <typename R>
cudaError_t wilson_A(const void* in, void* out, const void* U, const void* W, double diag, int Lx,
                     int Lt, int nrhs, const Epilogue& ep, cudaStream_t s) {
  const bool dot = ep.dot_out != nullptr;
  const bool fx = sizeof(R) == 8 && wilson_A_fx_ok(W, diag, ep);
  if (sizeof(R) == 8 && !fx) W = nullptr;
  if (sizeof(R) == 4 && !W && !dot) return cudaErrorInvalidValue;
  if (dot && (nrhs > 64 || !wilson_A_dot_fits(Lx, Lt, sizeof(R) == 8, fx ? diag : 0.0)))
    return cudaErrorInvalidValue;
  int v = dot ? -1 : tuned_variant<R>(Lx, Lt, nrhs, fx);
  if (v < 0) v = fx ? wilson_fx_variant(Lx, Lt, nrhs, dot) : wilson_default_variant<R>(Lx, Lt, nrhs, dot);
  const cudaError_t e = launch_variant<R>(v, in, out, U, W, diag, Lx, Lt, nrhs, ep, s);
  count_launch();
  return e;
}

// out = sigma_3 in on V two-spinors (FP64): spin component 1 negated.
__global__ void k_sigma3(const double2* __restrict__ in, double2* out, long long V, int dependent) {
  pdl_wait(dependent, in, out);
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= V) return;
  const double2 a = in[2 * i], b = in[2 * i + 1];
  out[2 * i] = a;
  out[2 * i + 1] = make_double2(-b.x, -b.y);
}

cudaError_t sigma3_mul(const void* in, void* out, long long V, cudaStream_t s) {
  launch_after(k_sigma3, (unsigned)((V + 255) / 256), 256, 0, s, (const double2*)in, (double2*)out, V);
  count_launch();
  return cudaGetLastError();
}

template <typename R>
__global__ void k_fold_links(const double2* __restrict__ g, cplx_t<R>* __restrict__ U, int Lx,
                             int Lt, double factor, int dependent) {
  pdl_wait(dependent, g, U);
  const int V = Lx * Lt;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * V) return;
  const int mu = i / V, site = i % V;
  const double sg = (mu == 1 && site / Lx == Lt - 1) ? -factor : factor;
  double2 u = g[i];
  U[i] = mk((R)(sg * u.x), (R)(sg * u.y));
}

template <typename R>
cudaError_t fold_links(const void* gauge, void* U, int Lx, int Lt, cudaStream_t s, double factor) {
  const int n = 2 * Lx * Lt;
  launch_after(k_fold_links<R>, (n + 255) / 256, 256, 0, s, (const double2*)gauge, (cplx_t<R>*)U, Lx, Lt,
               factor);
  count_launch();
  return cudaGetLastError();
}

// Non-negative doubles (and NaN above them) order like their bit patterns.
__global__ void __launch_bounds__(256) k_link_unitarity(const double2* __restrict__ g, long long count,
                                                        unsigned long long* out, int dependent) {
  pdl_wait(dependent, g, out);
  unsigned long long m = 0;
  for (long long i = (long long)blockIdx.x * 256 + threadIdx.x; i < count; i += 256LL * gridDim.x) {
    const double2 u = g[i];
    const double d = fabs(sqrt(u.x * u.x + u.y * u.y) - 1.0);
    m = max(m, (unsigned long long)__double_as_longlong(d));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

cudaError_t link_unitarity(const void* gauge, long long count, double* out, cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), s);
  if (e != cudaSuccess) return e;
  const long long g = (count + 255) / 256;
  launch_after(k_link_unitarity, (unsigned)(g < 1216 ? g : 1216), 256, 0, s, (const double2*)gauge, count,
               (unsigned long long*)out);
  count_launch();
  return cudaGetLastError();
}

#define INST(R)                                                                               \
  template cudaError_t wilson_D<R>(const void*, void*, const void*, double, int, int, int,    \
                                   bool, cudaStream_t);                                       \
  template cudaError_t wilson_A<R>(const void*, void*, const void*, const void*, double, int,   \
                                   int, int, const Epilogue&, cudaStream_t);                  \
  template cudaError_t wilson_A_tune<R>(const void*, void*, void*, const void*, const void*,   \
                                        double, int, int, int, int*, cudaStream_t);           \
  template cudaError_t fold_links<R>(const void*, void*, int, int, cudaStream_t, double);
INST(double)
INST(float)
#undef INST

}  // namespace mgk
