// y = B x for 16 to 64 right-hand sides with the packed Hermitian inverse of the coarsest
// operator (k_pack_hermitian), on the 5th-generation tensor cores (tcgen05 kind::tf32,
// accumulators in tensor memory).
//
// A CTA owns 128 rows (two 64-row blocks) and a share of the columns.  Column block J of
// row block I is the stored tile (I, J) or, above the diagonal, the Hermitian image of
// tile (J, I); so every tile is read twice, the second time mostly from L2, and a row's
// sum stays in one CTA.  Reading each tile once for both products (mma.sync) left a
// partial product per tile and side, 136 MB written and read again for 4096 unknowns and
// 64 right-hand sides.
//
// MMA: M = 128 rows, K = a tile's columns with (re, im) side by side, as stored, N = the
// right-hand sides twice: rows (xr, -xi) of the X operand give the real part, rows
// (xi, xr) the imaginary part.  Both operands are split into TF32 hi + lo words; three
// products (lo hi, hi lo, hi hi) make up an FP32-accurate one.  A column block is staged
// in four stages of 16 complex columns.
//
// Roles, synchronised through mbarriers: warps 0-3 and 4-7 take the stages in turn, load
// theirs ahead (cp.async), split and store the operands (K-major core matrices, 8 rows x 16 bytes, every store of
// a warp 512 consecutive bytes), warp 16 issues the MMAs, warps 8-15 add the finished
// column blocks in FP32 registers (the accumulator is used for one block at a time, so
// that no long sum runs in the tensor cores).  Each wait is bounded and reports through
// gemv_tc_take_error.
//
// Bound by shared memory: 1860 wavefronts per stage, half of them cp.async, and 96 KB of
// operand reads by the MMAs, against 900 clocks of TF32 issue; 2300 clocks are taken.
// 4096 unknowns, 64 right-hand sides, with the copy of x and the last sum: 226 us with
// mma.sync; here 130 us with the next stage in registers, 96 us with cp.async three stages
// ahead, 91 us with two producer groups.  The error against 64 bits is the same (9.0e-7 on a
// random Hermitian matrix); the 64-source solve on 256^2 goes from 294 to 247 ms.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "mma_tf32.cuh"
#include "tcgen05.cuh"

namespace mgk {

namespace {

__device__ int g_gemv_tc_err;

constexpr int GT_T = 64;                                 // rows and columns of a stored tile
constexpr int GT_M = 128, GT_KS = 32;                    // rows of a CTA, floats of a stage along K
constexpr int GT_SLOTS = 2;                              // operand buffers
constexpr int GT_OP = GT_M * GT_KS * 4;                  // bytes of one operand word (A, or X at N = 128)
constexpr int GT_GROUP = 128;                            // a producer group, one for each operand buffer
constexpr int GT_PRODUCERS = GT_SLOTS * GT_GROUP, GT_READERS = 256;
constexpr int GT_THREADS = GT_PRODUCERS + GT_READERS + 32;
constexpr int GT_ITEMS = 12;                             // 16-byte chunks of a thread and stage: 8 of A, 4 of X
constexpr int GT_SMEM = GT_SLOTS * 4 * GT_OP + 2 * GT_ITEMS * GT_PRODUCERS * 16 + 1024;

// Byte offset of 16-byte chunk `chunk` (4 floats of K) of operand row `row`.
__device__ __forceinline__ int gt_byte(int row, int chunk) {
  return ((row >> 3) * (GT_KS / 4) + chunk) * 128 + (row & 7) * 16;
}

__device__ __forceinline__ void gt_store(unsigned char* hi, unsigned char* lo, int at, float4 v) {
  uint4 h, l;
  split_tf32(v.x, h.x, l.x);
  split_tf32(v.y, h.y, l.y);
  split_tf32(v.z, h.z, l.z);
  split_tf32(v.w, h.w, l.w);
  *(uint4*)(hi + at) = h;
  *(uint4*)(lo + at) = l;
}

__device__ __forceinline__ void gt_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
      :: "r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void gt_arrive(uint64_t* m) {
  asm volatile("{\n.reg .b64 st;\nmbarrier.arrive.shared::cta.b64 st, [%0];\n}\n"
               :: "r"(tc::saddr(m)) : "memory");
}

__device__ __forceinline__ void gt_copy16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void gt_copy8(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(src) : "memory");
}

__global__ void __launch_bounds__(GT_THREADS, 1)
    k_hgemv_tc(const float2* __restrict__ P, const float2* __restrict__ xs, int ld, int nt, int nrhs,
               float* __restrict__ part, int dependent) {
  pdl_wait(dependent, P, xs, part);
  extern __shared__ __align__(16) unsigned char gt_dyn[];
  __shared__ __align__(8) uint64_t full[GT_SLOTS], empty[GT_SLOTS], done[2], accfree[2];
  __shared__ uint32_t tmem_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.x;
  const int J0 = nt * (int)blockIdx.y / (int)gridDim.y, J1 = nt * ((int)blockIdx.y + 1) / (int)gridDim.y;
  const int stages = 4 * (J1 - J0);
  const int NR = (nrhs + 7) & ~7;                        // operand rows per part (re, im) of X
  unsigned char* ops = gt_dyn + ((1024u - (tc::saddr(gt_dyn) & 1023u)) & 1023u);
  if (warp == 0) tc::tmem_alloc(&tmem_sh, 256);
  if (tid == 0) {
    for (int q = 0; q < GT_SLOTS; ++q) {
      tc::mbar_init(&full[q], GT_GROUP);
      tc::mbar_init(&empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&done[q], 1);
      tc::mbar_init(&accfree[q], GT_READERS);
    }
    tc::fence_mbar_init();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_sh;
  bool ok = true;

  if (warp < 8) {
    // ---- producers: group w takes the stages s = w, w + 2, .. into operand buffer w.
    // Chunk i of a stage (0-7 of A, four for each row block; 8-11 of X) passes through
    // this thread's own 16 bytes of two raw buffers, so that its cp.async groups are the
    // only synchronisation.  Chunks of a missing row block or right-hand side stay zero.
    const int w = tid / GT_GROUP, gt = tid % GT_GROUP;
    float4* raw = (float4*)(ops + GT_SLOTS * 4 * GT_OP) + tid;
    unsigned char* ah = ops + w * 4 * GT_OP;
    unsigned char *al = ah + GT_OP, *xh = al + GT_OP, *xl = xh + GT_OP;
    auto at = [&](int s, int i) { return raw + (((s >> 1) & 1) * GT_ITEMS + i) * GT_PRODUCERS; };
    auto xrow = [&](int i) { return (gt & 7) + 8 * ((gt + GT_GROUP * (i & 3)) >> 6); };
    for (int i = 0; i < GT_ITEMS; ++i)
      if (!(i < 8 ? 2 * b + (i >> 2) < nt : xrow(i) < nrhs))
        *at(0, i) = *at(2, i) = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load = [&](int s) {
      const int J = J0 + (s >> 2), c0 = 16 * (s & 3);    // complex columns c0 .. c0 + 15 of block J
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int I = 2 * b + (i >> 2), e = gt + GT_GROUP * (i & 3);   // 512 chunks per row block
        const uint32_t dst = tc::saddr(at(s, i));
        if (I >= nt) continue;
        if (J <= I) {                                    // as stored: lane = (chunk, row % 8)
          const int row = (e & 7) + 8 * (e >> 6), ch = (e >> 3) & 7;
          gt_copy16(dst, P + ((long long)I * (I + 1) / 2 + J) * GT_T * GT_T + row * GT_T + c0 + 2 * ch);
        } else {                                         // image of tile (J, I): lane = row
          const int row = e & 63, ch = e >> 6;
          const float2* p = P + ((long long)J * (J + 1) / 2 + I) * GT_T * GT_T + (c0 + 2 * ch) * GT_T + row;
          gt_copy8(dst, p);
          gt_copy8(dst + 8, p + GT_T);
        }
      }
#pragma unroll
      for (int i = 8; i < 12; ++i) {
        const int r = xrow(i), ch = ((gt + GT_GROUP * (i & 3)) >> 3) & 7;
        if (r < nrhs) gt_copy16(tc::saddr(at(s, i)), xs + (long long)r * ld + J * GT_T + c0 + 2 * ch);
      }
    };
    auto store = [&](int s) {
      const int J = J0 + (s >> 2);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int e = gt + GT_GROUP * (i & 3);
        const bool direct = J <= 2 * b + (i >> 2);
        const int row = direct ? (e & 7) + 8 * (e >> 6) : e & 63, ch = direct ? (e >> 3) & 7 : e >> 6;
        float4 v = *at(s, i);
        if (!direct) v = make_float4(v.x, -v.y, v.z, -v.w);
        gt_store(ah, al, gt_byte(64 * (i >> 2) + row, ch), v);
      }
#pragma unroll
      for (int i = 8; i < 12; ++i) {
        const int r = xrow(i), ch = ((gt + GT_GROUP * (i & 3)) >> 3) & 7;
        if (r < NR) {
          const float4 v = *at(s, i);
          gt_store(xh, xl, gt_byte(r, ch), make_float4(v.x, -v.y, v.z, -v.w));
          gt_store(xh, xl, gt_byte(NR + r, ch), make_float4(v.y, v.x, v.w, v.z));
        }
      }
    };
    load(w);                                             // stages is a multiple of 4
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int s = w; s < stages; s += 2) {
      // stage s + 2 goes where stage s - 2 was, which has been split and stored
      if (s + 2 < stages) load(s + 2);
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      if (s >= 2)                                        // the MMAs have read the buffer's last stage
        ok = tc::mbar_wait(&empty[w], (uint32_t)((s / 2 - 1) & 1), &g_gemv_tc_err);
      if (!ok) break;
      store(s);
      tc::fence_proxy_async();
      gt_arrive(&full[w]);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  } else if (warp == 16) {
    // ---- MMA warp
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(NR >> 2) << 17) |
                           ((uint32_t)(GT_M >> 4) << 24);   // D FP32, A and B TF32, N = 2 NR
    for (int s = 0; s < stages && ok; ++s) {
      const int g = s >> 2;
      ok = tc::mbar_wait(&full[s % GT_SLOTS], (uint32_t)((s / GT_SLOTS) & 1), &g_gemv_tc_err);
      if (ok && (s & 3) == 0 && g >= 2)                  // block g - 2 has been read
        ok = tc::mbar_wait(&accfree[g & 1], (uint32_t)((g / 2 - 1) & 1), &g_gemv_tc_err);
      if (!ok) break;
      if (lane == 0) {
        tc::fence_after_sync();
        const uint32_t ah = tc::saddr(ops + (s % GT_SLOTS) * 4 * GT_OP);
        const uint32_t d = tmem + (uint32_t)((g & 1) * 128);
#pragma unroll
        for (int kk = 0; kk < GT_KS / 8; ++kk) {
          const uint32_t o = ah + 256 * kk;
          const uint64_t dah = tc::desc(o, 128, GT_KS / 4 * 128), dal = tc::desc(o + GT_OP, 128, GT_KS / 4 * 128);
          const uint64_t dxh = tc::desc(o + 2 * GT_OP, 128, GT_KS / 4 * 128),
                         dxl = tc::desc(o + 3 * GT_OP, 128, GT_KS / 4 * 128);
          gt_mma(d, dal, dxh, idesc, (s & 3) | kk ? 1u : 0u);
          gt_mma(d, dah, dxl, idesc, 1u);
          gt_mma(d, dah, dxh, idesc, 1u);
        }
        tc::commit(&empty[s % GT_SLOTS]);
        if ((s & 3) == 3) tc::commit(&done[g & 1]);
      }
      __syncwarp();
    }
  } else {
    // ---- readers: warp w takes rows 32 (w % 4) .. + 31, warps 8-11 the real parts
    const int qd = warp & 3, p = (warp - 8) >> 2;
    float acc[64];
#pragma unroll
    for (int q = 0; q < 64; ++q) acc[q] = 0.f;
    for (int g = 0; g < J1 - J0; ++g) {
      ok = tc::mbar_wait(&done[g & 1], (uint32_t)((g >> 1) & 1), &g_gemv_tc_err);
      if (!ok) break;
      tc::fence_after_sync();
      const uint32_t t = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)((g & 1) * 128 + p * NR);
#pragma unroll
      for (int q0 = 0; q0 < 64; q0 += 16) {
        if (q0 >= NR) break;
        float v[16];
        tc::tmem_ld8(t + q0, v);
        if (q0 + 8 < NR) tc::tmem_ld8(t + q0 + 8, v + 8);
        tc::tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[q0 + q] += v[q];
        if (q0 + 8 < NR) {
#pragma unroll
          for (int q = 8; q < 16; ++q) acc[q0 + q] += v[q];
        }
      }
      tc::fence_before_sync();
      gt_arrive(&accfree[g & 1]);
    }
    const int row = GT_M * b + 32 * qd + lane;
    if (ok && row < ld) {
      float* o = part + ((long long)blockIdx.y * 2 + p) * nrhs * ld + row;
#pragma unroll
      for (int r = 0; r < 64; ++r)
        if (r < nrhs) o[(long long)r * ld] = acc[r];
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// The column shares of a row added in order.
__global__ void __launch_bounds__(128) k_hgemv_tc_sum(const float* __restrict__ part, double2* __restrict__ y,
                                                      int N, int ld, int splits, bool accumulate,
                                                      float2* __restrict__ y32, int dependent) {
  pdl_wait(dependent, part, y, y32);
  const int row = blockIdx.x * 128 + threadIdx.x, r = blockIdx.y, nrhs = gridDim.y;
  if (row >= N) return;
  float2 a = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int s = 0; s < splits; ++s) {
    const float* p = part + ((long long)s * 2 * nrhs + r) * ld + row;
    a.x += p[0];
    a.y += p[(long long)nrhs * ld];
  }
  const long long i = (long long)r * N + row;
  double2 v = make_double2(a.x, a.y);
  if (accumulate) {
    const double2 w = y[i];
    v = make_double2(v.x + w.x, v.y + w.y);
  }
  y[i] = v;
  if (y32) y32[i] = make_float2((float)v.x, (float)v.y);
}

// Column shares per row block: as many as fill the SMs once (one CTA each).
int gt_splits(int nt) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return std::max(1, std::min(nt, sms / ((nt + 1) / 2)));
}

}  // namespace

// The MMAs pad 16 right-hand sides no less than the mma.sync kernel, but a CTA has some
// 10 us of its own (tensor memory, barriers, first loads), so the line is at 64 right-hand
// sides for 16 tile rows and at 16 for 64: the whole product at 1000 unknowns takes 28.7 us
// both ways at 64 right-hand sides (26.7 against 18.5 us at 16), at 4096 unknowns 78
// against 91 us at 16, 81 against 146 at 32, 91 against 226 at 64.
bool hermitian_gemv_tc_ok(int ld, int nrhs) {
  return nrhs >= 16 && nrhs <= 64 && ld / GT_T * nrhs >= 1024;
}

cudaError_t hermitian_gemv_tc(const void* P, const void* x, void* y, int N, int ld, int nrhs, void* xscratch,
                              void* part, bool accumulate, void* y32, cudaStream_t s) {
  if (ld % GT_T || ld < N || nrhs < 1 || nrhs > 64) return cudaErrorInvalidValue;
  static SmemLimit limit;
  const cudaError_t e = limit.raise(k_hgemv_tc, GT_SMEM);
  if (e != cudaSuccess) return e;
  const cudaError_t ex = to_f32_padded(x, xscratch, N, ld, nrhs, s);
  if (ex != cudaSuccess) return ex;
  const int nt = ld / GT_T, splits = gt_splits(nt);
  launch_after(k_hgemv_tc, dim3((nt + 1) / 2, splits), GT_THREADS, GT_SMEM, s, (const float2*)P,
               (const float2*)xscratch, ld, nt, nrhs, (float*)part);
  launch_after(k_hgemv_tc_sum, dim3((N + 127) / 128, nrhs), 128, 0, s, (const float*)part, (double2*)y, N, ld,
               splits, accumulate, (float2*)y32);
  count_launch();
  count_launch();
  return cudaGetLastError();
}

cudaError_t gemv_tc_take_error(int* flag) {
  int v = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_gemv_tc_err, sizeof(int));
  if (e != cudaSuccess) return e;
  if (v) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_gemv_tc_err, &zero, sizeof(int));
  }
  *flag = v;
  return e;
}

}  // namespace mgk
