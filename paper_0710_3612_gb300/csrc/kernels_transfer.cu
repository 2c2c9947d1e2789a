// FP32 restriction P^dagger and prolongation P with the block vectors in registers.
//
// A warp covers 32 / (2 H2) neighbouring sites of a row (H2 = h rounded up to a power of
// two): lane = (site, chirality, component), which is the order of the fine vector, so every
// load and store of it is one contiguous run.  A lane keeps the Nv vector entries of its
// component for the ROWS sites it owns in its block (the bt rows, and bx / BXW sites of a
// row when a warp holds fewer than bx) and uses them for a chunk of right-hand sides, which
// stream past with the next one's loads in flight.  Restriction sums over the lanes of a
// block by a transposing butterfly (each step halves the outputs a lane holds).
//
// Bound by HBM and latency: per right-hand side a fine entry is 8 bytes and 4 Nv FMAs.  The
// shared-memory kernels (k_restrict_multi, k_prolong_multi) read two shared operands
// for every complex product and keep one site per CTA in flight: 256^2, 64 right-hand
// sides, 84 and 101 us against 37 and 37 us here (109 MB each, 3.0 TB/s).
//
// Rounding: sums run in short chains added pairwise (two halves of the rows, four or
// six chains of the vectors), since one chain of Nv products was further from the exact result than
// the shared-memory kernels' trees at one right-hand side (Nv = 12: 9.3e-8 against 6.5e-8).
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace mgk {

namespace {

template <int ROWS, int NV, int H2, int BXW>
struct Geo {
  static constexpr int SXW = 32 / (2 * H2);            // sites per warp along x
  static constexpr int ABITS = H2 == 1 ? 0 : H2 == 2 ? 1 : H2 == 4 ? 2 : H2 == 8 ? 3 : 4;
  static constexpr int XBITS = BXW == 1 ? 0 : BXW == 2 ? 1 : BXW == 4 ? 2 : 3;
  static constexpr int BITS = ABITS + XBITS;           // lane bits a block's sum runs over
  static constexpr int mask(int i) { return i < ABITS ? 1 << i : 2 * H2 << (i - ABITS); }
};

struct TransferArgs {
  const float2* in;
  float2* out;
  const float2* Vst;
  int Lx, Lt, bx, bt, h, nrhs, chunk, runs;            // runs: warps along x
};

// The warp's lane: site and component, and its vector entries.
template <int ROWS, int NV, int H2, int BXW>
struct Lane {
  using G = Geo<ROWS, NV, H2, BXW>;
  int a, c, j;                                         // component, chirality, coarse site
  long long off[ROWS];                                 // fine entry of each owned site
  bool on;
  __device__ __forceinline__ Lane(const TransferArgs& t, int run, int jt, float2 (&v)[ROWS][NV]) {
    const int lane = threadIdx.x & 31, XL = t.bx / BXW, n = 2 * t.h;
    a = lane & (H2 - 1);
    c = (lane / H2) & 1;
    const int x0 = run * G::SXW * XL + lane / (2 * H2);
    on = a < t.h && x0 < t.Lx;
    j = x0 / t.bx + (t.Lx / t.bx) * jt;
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      const long long i = x0 + (q % XL) * G::SXW + (long long)t.Lx * (jt * t.bt + q / XL);
      off[q] = i * n + c * t.h + a;
#pragma unroll
      for (int k = 0; k < NV; ++k)
        v[q][k] = on ? t.Vst[((i * 2 + c) * NV + k) * t.h + a] : make_float2(0.f, 0.f);
    }
  }
};

template <int ROWS, int NV, int H2, int BXW>
__global__ void __launch_bounds__(128) k_restrict_reg(const TransferArgs t, int dependent) {
  pdl_wait(dependent);
  using G = Geo<ROWS, NV, H2, BXW>;
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int run = w % t.runs, jt = w / t.runs;
  if (jt >= t.Lt / t.bt) return;
  float2 v[ROWS][NV];
  const Lane<ROWS, NV, H2, BXW> l(t, run, jt, v);
  const long long nf = (long long)t.Lx * t.Lt * 2 * t.h;
  const long long nc = (long long)(t.Lx / t.bx) * (t.Lt / t.bt) * 2 * NV;
  const int r0 = blockIdx.y * t.chunk, r1 = min(r0 + t.chunk, t.nrhs);
  float2 r[ROWS];
#pragma unroll
  for (int q = 0; q < ROWS; ++q) r[q] = l.on ? t.in[r0 * nf + l.off[q]] : make_float2(0.f, 0.f);
  for (int rhs = r0; rhs < r1; ++rhs) {
    float2 nx[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q)
      nx[q] = l.on && rhs + 1 < r1 ? t.in[(rhs + 1) * nf + l.off[q]] : make_float2(0.f, 0.f);
    float2 acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      float2 hi = make_float2(0.f, 0.f);               // the rows in two halves
      acc[k] = hi;
#pragma unroll
      for (int q = 0; q < ROWS; ++q) cfmac(q < ROWS / 2 ? acc[k] : hi, v[q][k], r[q]);
      acc[k] = cadd(acc[k], hi);
    }
    int k0 = 0;
    bool writer = l.on || l.a >= t.h;                  // lanes past h hold sums of others too
    constexpr int B = G::BITS;
    // cnt: outputs a lane still holds after each step
    auto step = [&](auto cnt_c, int m) {
      constexpr int cnt = decltype(cnt_c)::value;
      const bool up = (lane & m) != 0;
      if constexpr (cnt % 2 == 0) {
        constexpr int half = cnt / 2;
#pragma unroll
        for (int i = 0; i < half; ++i) {
          const float2 send = up ? acc[i] : acc[i + half], keep = up ? acc[i + half] : acc[i];
          acc[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, send.x, m),
                               keep.y + __shfl_xor_sync(0xffffffffu, send.y, m));
        }
        k0 += up ? half : 0;
      } else {
#pragma unroll
        for (int i = 0; i < cnt; ++i) {
          acc[i].x += __shfl_xor_sync(0xffffffffu, acc[i].x, m);
          acc[i].y += __shfl_xor_sync(0xffffffffu, acc[i].y, m);
        }
        writer = writer && !up;
      }
    };
    constexpr int C1 = NV, C2 = C1 % 2 ? C1 : C1 / 2, C3 = C2 % 2 ? C2 : C2 / 2, C4 = C3 % 2 ? C3 : C3 / 2,
                  C5 = C4 % 2 ? C4 : C4 / 2;
    if constexpr (B > 0) step(std::integral_constant<int, C1>(), G::mask(0));
    if constexpr (B > 1) step(std::integral_constant<int, C2>(), G::mask(1));
    if constexpr (B > 2) step(std::integral_constant<int, C3>(), G::mask(2));
    if constexpr (B > 3) step(std::integral_constant<int, C4>(), G::mask(3));
    constexpr int CN = B == 0 ? C1 : B == 1 ? C2 : B == 2 ? C3 : B == 3 ? C4 : C5;
    if (writer && l.j < (int)(nc / (2 * NV)) && (run * G::SXW * (t.bx / BXW) + lane / (2 * H2)) < t.Lx) {
      float2* o = t.out + rhs * nc + (long long)l.j * 2 * NV + l.c * NV + k0;
      if constexpr (CN % 2 == 0) {
#pragma unroll
        for (int i = 0; i < CN; i += 2)
          *(float4*)(o + i) = make_float4(acc[i].x, acc[i].y, acc[i + 1].x, acc[i + 1].y);
      } else {
#pragma unroll
        for (int i = 0; i < CN; ++i) o[i] = acc[i];
      }
    }
#pragma unroll
    for (int q = 0; q < ROWS; ++q) r[q] = nx[q];
  }
}

template <int ROWS, int NV, int H2, int BXW, bool ACC>
__global__ void __launch_bounds__(128) k_prolong_reg(const TransferArgs t, int dependent) {
  pdl_wait(dependent);
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5);
  const int run = w % t.runs, jt = w / t.runs;
  if (jt >= t.Lt / t.bt) return;
  float2 v[ROWS][NV];
  const Lane<ROWS, NV, H2, BXW> l(t, run, jt, v);
  if (!l.on) return;
  const long long nf = (long long)t.Lx * t.Lt * 2 * t.h;
  const long long nc = (long long)(t.Lx / t.bx) * (t.Lt / t.bt) * 2 * NV;
  const int r0 = blockIdx.y * t.chunk, r1 = min(r0 + t.chunk, t.nrhs);
  const float2* e0 = t.in + (long long)l.j * 2 * NV + l.c * NV;
  float4 e[NV / 2];
#pragma unroll
  for (int k = 0; k < NV / 2; ++k) e[k] = ((const float4*)(e0 + r0 * nc))[k];
  for (int rhs = r0; rhs < r1; ++rhs) {
    float2 f[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) f[q] = ACC ? t.out[rhs * nf + l.off[q]] : make_float2(0.f, 0.f);
    float4 nx[NV / 2];
    const float4* en = (const float4*)(e0 + min(rhs + 1, r1 - 1) * nc);
#pragma unroll
    for (int k = 0; k < NV / 2; ++k) nx[k] = en[k];
    float2 s[ROWS];
#pragma unroll
    for (int q = 0; q < ROWS; ++q) {
      constexpr int CH = NV == 12 ? 6 : 4;             // chains: see the rounding above
      float2 p[CH] = {};
#pragma unroll
      for (int k = 0; k < NV / 2; ++k) {
        cfma(p[2 * k % CH], v[q][2 * k], make_float2(e[k].x, e[k].y));
        cfma(p[2 * k % CH + 1], v[q][2 * k + 1], make_float2(e[k].z, e[k].w));
      }
      s[q] = cadd(cadd(p[0], p[1]), cadd(p[2], p[3]));
      if constexpr (CH == 6) s[q] = cadd(s[q], cadd(p[4], p[5]));
    }
#pragma unroll
    for (int q = 0; q < ROWS; ++q) t.out[rhs * nf + l.off[q]] = ACC ? cadd(f[q], s[q]) : s[q];
#pragma unroll
    for (int k = 0; k < NV / 2; ++k) e[k] = nx[k];
  }
}

// Right-hand sides per warp: enough chunks for 16 warps on every SM.  256^2 x 64, restriction
// and prolongation together: 74 us; half as many right-hand sides per warp 84, a quarter 103
// (the vectors are read again for each chunk), twice as many 68 but the solve 1% slower.
int chunk_of(long long warps, int nrhs) {
  int chunk = nrhs;
  while (chunk > 1 && warps * ((nrhs + chunk - 1) / chunk) < 1LL * 152 * 16) chunk = (chunk + 1) / 2;
  return chunk;
}

template <int ROWS, int NV, int H2, int BXW>
cudaError_t launch(TransferArgs t, bool prolong, bool acc, cudaStream_t s) {
  using G = Geo<ROWS, NV, H2, BXW>;
  const int sx = G::SXW * (t.bx / BXW);
  t.runs = (t.Lx + sx - 1) / sx;
  const long long warps = (long long)t.runs * (t.Lt / t.bt);
  t.chunk = chunk_of(warps, t.nrhs);
  const dim3 grid((unsigned)((warps + 3) / 4), (t.nrhs + t.chunk - 1) / t.chunk);
  if (!prolong)
    launch_after(k_restrict_reg<ROWS, NV, H2, BXW>, grid, 128, 0, s, t);
  else if (acc)
    launch_after(k_prolong_reg<ROWS, NV, H2, BXW, true>, grid, 128, 0, s, t);
  else
    launch_after(k_prolong_reg<ROWS, NV, H2, BXW, false>, grid, 128, 0, s, t);
  return cudaGetLastError();
}

}  // namespace

// The blockings with a register kernel: 4 x 4 blocks of the fine lattice (h = 1) and 2 x 2
// blocks of levels whose dof per chirality is the Nv of the next one (4, 8 or 12).
// The coarse vectors are read and written 16 bytes at a time.
bool transfer_reg_ok(const void* coarse, int bx, int bt, int h, int Nv) {
  if ((uintptr_t)coarse % 16) return false;
  if (h == 1) return bx == 4 && bt == 4 && (Nv == 4 || Nv == 8 || Nv == 12);
  return bx == 2 && bt == 2 && h == Nv && (Nv == 4 || Nv == 8 || Nv == 12);
}

cudaError_t transfer_reg(const void* in, void* out, const void* Vst, int Lx, int Lt, int bx, int bt,
                         int h, int Nv, int nrhs, bool prolong, bool acc, cudaStream_t s) {
  if (!transfer_reg_ok(prolong ? in : out, bx, bt, h, Nv)) return cudaErrorInvalidValue;
  const TransferArgs t{(const float2*)in, (float2*)out, (const float2*)Vst, Lx, Lt, bx, bt, h, nrhs, 0, 0};
  cudaError_t e;
  if (h == 1)
    e = Nv == 4 ? launch<4, 4, 1, 4>(t, prolong, acc, s)
        : Nv == 8 ? launch<4, 8, 1, 4>(t, prolong, acc, s) : launch<4, 12, 1, 4>(t, prolong, acc, s);
  else
    e = Nv == 4 ? launch<2, 4, 4, 2>(t, prolong, acc, s)
        : Nv == 8 ? launch<2, 8, 8, 2>(t, prolong, acc, s) : launch<4, 12, 16, 1>(t, prolong, acc, s);
  count_launch();
  return e;
}

}  // namespace mgk
