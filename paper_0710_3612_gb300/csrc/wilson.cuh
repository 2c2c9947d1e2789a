// Device helpers shared by the fine-lattice stencil kernels: the per-site Wilson
// stencil on global memory, whole-spinor loads and stores, asynchronous copies.
#pragma once

#include "common.cuh"

namespace mgk {

template <typename R, bool DAG>
__device__ __forceinline__ void wilson_site(const cplx_t<R>* __restrict__ in,
                                            const cplx_t<R>* __restrict__ U, R diag, int x, int t,
                                            int Lx, int Lt, cplx_t<R>& o0, cplx_t<R>& o1) {
  using C = cplx_t<R>;
  const int V = Lx * Lt;
  const int site = x + Lx * t;
  const int xp = (x + 1 == Lx) ? site - x : site + 1;
  const int xm = (x == 0) ? site + Lx - 1 : site - 1;
  const int tp = (t + 1 == Lt) ? x : site + Lx;
  const int tm = (t == 0) ? site + (Lt - 1) * Lx : site - Lx;
  const R sf = DAG ? (R)-1 : (R)1;   // projector sign of the forward hop
  C a0 = mk((R)0, (R)0), a1 = mk((R)0, (R)0);
  hop_x<R>(a0, a1, U[site], in[2 * xp], in[2 * xp + 1], sf);
  hop_x<R>(a0, a1, cconj(U[xm]), in[2 * xm], in[2 * xm + 1], -sf);
  hop_t<R>(a0, a1, U[V + site], in[2 * tp], in[2 * tp + 1], sf);
  hop_t<R>(a0, a1, cconj(U[V + tm]), in[2 * tm], in[2 * tm + 1], -sf);
  C p0 = in[2 * site], p1 = in[2 * site + 1];
  o0 = mk(diag * p0.x - (R)0.5 * a0.x, diag * p0.y - (R)0.5 * a0.y);
  o1 = mk(diag * p1.x - (R)0.5 * a1.x, diag * p1.y - (R)0.5 * a1.y);
}

template <typename R> struct spinor_t;              // both spin components of a site
template <> struct spinor_t<float> { using type = float4; };
template <> struct spinor_t<double> { using type = double4_32a; };

__device__ __forceinline__ void split(const float4& v, float2& a, float2& b) {
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void split(const double4_32a& v, double2& a, double2& b) {
  a = make_double2(v.x, v.y);
  b = make_double2(v.z, v.w);
}
__device__ __forceinline__ float4 join(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ double4_32a join(double2 a, double2 b) {
  double4_32a r;
  r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
  return r;
}
__device__ __forceinline__ float4 ld_spinor(const float2* p) { return *(const float4*)p; }
__device__ __forceinline__ double4_32a ld_spinor(const double2* p) {
  const double2 a = p[0], b = p[1];
  return join(a, b);
}
__device__ __forceinline__ void st_spinor(float2* p, float4 v) { *(float4*)p = v; }
__device__ __forceinline__ void st_spinor(double2* p, double4_32a v) {
  p[0] = make_double2(v.x, v.y);
  p[1] = make_double2(v.z, v.w);
}

// Periodic coordinate for -L <= g < 2L.
__device__ __forceinline__ int wrap(int g, int L) { return g < 0 ? g + L : (g >= L ? g - L : g); }
// The same for tiles that may be wider than the lattice: their unused halo is clamped
// into range.
__device__ __forceinline__ int wrap_tile(int g, int L) { return min(wrap(g, L), L - 1); }

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

}  // namespace mgk
