// Device helpers shared by the kernels: complex arithmetic on float2/double2,
// precision traits, and the lattice index functions (site = x + Lx * t).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

namespace mgk {

// Number of kernel launches made by this library (all threads), for reporting.
void count_launch();
unsigned long long launch_count();

// Launches on a stream follow one another by programmatic dependence: a kernel is set up
// while its predecessor drains, and waits in pdl_wait, its first statement, until all of
// that one's work is complete and visible.  As every kernel launched so waits there, a
// chain keeps its order; other launches and copies wait for whole kernels as ever.
// Dependent kernels of 64 to 1024 CTAs back to back in a stream took 4.1 us each with plain
// launches and 1.5 to 1.8 us so (V-cycle on 144 x 96: 106 -> 63 us).  Grids of many waves
// gain nothing and keep plain launches, and so do captured loops, whose gaps are short
// already: with the wait in every kernel the 64-source solve on 256^2 took 2% longer.
static constexpr long long PDL_MAX_CTAS = 152 * 16;

// A pointer whose loads may not be moved ahead of this.  A kernel's `const T* __restrict__`
// argument and __ldg promise data that nobody writes while the kernel runs, which lets a
// compiler move loads over the wait's memory clobber; behind a wait that promise holds only
// from here on.  The pointer that comes out carries no such promise of its own; it is made
// from a global address again, or its loads would be generic ones, which may meet the stores
// to shared memory around them (one-source solve on 128^2 11.2 ms against 10.8 to 11.1).
template <typename T>
__device__ __forceinline__ void pdl_ordered(T& p) {
  size_t g = __cvta_generic_to_global((const void*)p);
  asm volatile("" : "+l"(g)::"memory");
  p = (T)__cvta_global_to_generic(g);
}
// p: every pointer argument of the kernel.  (Pointers inside structure arguments are not
// declared restrict: their loads stay behind the clobber.)
template <typename... T>
__device__ __forceinline__ void pdl_wait(int dependent, T&... p) {
  if (dependent) asm volatile("griddepcontrol.wait;" ::: "memory");
  (pdl_ordered(p), ...);
}

// Launches kernel(args..., dependent).
template <typename... P, typename... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                cudaStream_t stream, A&&... args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(stream, &capture);
  const int dependent = capture == cudaStreamCaptureStatusNone &&
                        (long long)grid.x * grid.y * grid.z <= PDL_MAX_CTAS;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &at;
  cfg.numAttrs = dependent;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)..., dependent);
}

// A kernel's dynamic shared-memory limit belongs to a device: raised on its first launch on
// each (a static of the launcher, one for every kernel; a failure is tried again).
class SmemLimit {
  std::atomic<unsigned long long> done_{0};            // bit per device
 public:
  template <typename K>
  cudaError_t raise(K* kernel, int bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
    if (done_.load() & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done_.fetch_or(bit);
    return e;
  }
};

template <typename R> struct cplx_of;
template <> struct cplx_of<double> { using type = double2; };
template <> struct cplx_of<float> { using type = float2; };
template <typename R> using cplx_t = typename cplx_of<R>::type;

__host__ __device__ __forceinline__ double2 mk(double a, double b) { return make_double2(a, b); }
__host__ __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }

template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return {a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return {a.x - b.x, a.y - b.y}; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// conj(a) * b
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) {
  return {a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x};
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return {a.x, -a.y}; }
// acc += a * b
template <typename C> __device__ __forceinline__ void cfma(C& acc, C a, C b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}
// acc += conj(a) * b
template <typename C> __device__ __forceinline__ void cfmac(C& acc, C a, C b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(-a.y, b.x, acc.y);
}

// One hop of the Wilson stencil in direction x (sigma_1) or t (sigma_2):
//   (1 - s sigma_1) phi = (phi0 - s phi1) (1, -s)^T
//   (1 - s sigma_2) phi = (phi0 + i s phi1) (1, -i s)^T
// accumulated as a += u * projection (both components).
template <typename R>
__device__ __forceinline__ void hop_x(cplx_t<R>& a0, cplx_t<R>& a1, cplx_t<R> u, cplx_t<R> f0,
                                      cplx_t<R> f1, R s) {
  // h = u * (f0 - s f1); a0 += h; a1 += -s h
  cplx_t<R> p = mk(f0.x - s * f1.x, f0.y - s * f1.y);
  cplx_t<R> h = cmul(u, p);
  a0 = cadd(a0, h);
  a1 = mk(a1.x - s * h.x, a1.y - s * h.y);
}

template <typename R>
__device__ __forceinline__ void hop_t(cplx_t<R>& a0, cplx_t<R>& a1, cplx_t<R> u, cplx_t<R> f0,
                                      cplx_t<R> f1, R s) {
  // h = u * (f0 + i s f1); a0 += h; a1 += -i s h
  cplx_t<R> p = mk(f0.x - s * f1.y, f0.y + s * f1.x);
  cplx_t<R> h = cmul(u, p);
  a0 = cadd(a0, h);
  a1 = mk(a1.x + s * h.y, a1.y - s * h.x);   // -i s h = s (h.y, -h.x)
}

__device__ __forceinline__ float2 bf2_to_f2(__nv_bfloat162 v) { return __bfloat1622float2(v); }

// Fixed-order block sums of one double per thread (N = 1) or two (N = 2), returned in
// thread 0.  sh holds N * blockDim doubles.  Each lane of warp 0 (and of warp 1 for the
// second number) first adds the entries of its column, so a 256-thread block issues 12
// FP64 additions per number where shuffles in every warp would issue 45: the FP64 pipe
// takes 16 clocks for each, and small reductions were bound by it.
template <int N>
__device__ __forceinline__ void block_sum(double& a, double& b, double* sh) {
  const int n = blockDim.x, w = threadIdx.x >> 5, l = threadIdx.x & 31;
  sh[threadIdx.x] = a;
  if (N == 2) sh[n + threadIdx.x] = b;
  __syncthreads();
  if (w < N && (N == 1 || n > 32)) {
    double v = 0.0;
    for (int i = l; i < n; i += 32) v += sh[w * n + i];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncwarp();
    if (l == 0) sh[w * n] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = sh[0];
    if (N == 2) b = sh[n];
  }
  __syncthreads();
}

// Single-pass deterministic reduction.  Every block writes its partial sum;
// the last block to finish (found with an atomic ticket) adds the partials in
// a fixed order and resets the ticket.  ws = [64 tickets (as doubles)][partials].
// rhs selects the output and ticket; blk in [0, G) is this block's slot; sh holds
// N * blockDim doubles (at least 64 threads for N = 2).  N = 1: the real part alone,
// the imaginary sum is written as zero.
// Returns true in the block that wrote the sum (all its threads).
template <int N>
__device__ __forceinline__ bool finish_reduction_g(double re, double im, double* ws, double* out,
                                                   double* sh, int rhs, int blk, int G) {
  unsigned* tickets = (unsigned*)ws;
  double* partials = ws + 64;
  __shared__ bool last;
  block_sum<N>(re, im, sh);
  if (threadIdx.x == 0) {
    partials[2 * ((long long)rhs * G + blk)] = re;
    if (N == 2) partials[2 * ((long long)rhs * G + blk) + 1] = im;
    __threadfence();
    last = atomicAdd(&tickets[rhs], 1u) == (unsigned)(G - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  re = 0.0;
  im = 0.0;
  for (int i = threadIdx.x; i < G; i += blockDim.x) {
    re += __ldcg(&partials[2 * ((long long)rhs * G + i)]);
    if (N == 2) im += __ldcg(&partials[2 * ((long long)rhs * G + i) + 1]);
  }
  block_sum<N>(re, im, sh);
  if (threadIdx.x == 0) {
    out[2 * rhs] = re;
    out[2 * rhs + 1] = N == 2 ? im : 0.0;
    tickets[rhs] = 0u;
  }
  return true;
}

template <int N>
__device__ __forceinline__ bool finish_reduction(double re, double im, double* ws, double* out,
                                                 double* sh) {
  return finish_reduction_g<N>(re, im, ws, out, sh, blockIdx.y, blockIdx.x, gridDim.x);
}

// Block map of the geometric blocking S_j: coarse site and in-block offset.
__host__ __device__ __forceinline__ int coarse_site(int x, int t, int Lx, int bx, int bt) {
  return (t / bt) * (Lx / bx) + x / bx;
}
__host__ __device__ __forceinline__ int block_offset(int x, int t, int bx, int bt) {
  return (t % bt) * bx + x % bx;
}

}  // namespace mgk
