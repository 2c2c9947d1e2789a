// Dense inverse of the coarsest operator: Gauss-Jordan sweeps of 64 x 64 pivot
// blocks on the lower tiles of a Hermitian positive definite complex64 matrix,
// ordered and restricted by the sparsity of the 9-point stencil it comes from.
//
// Sweeping pivot block k with P = M_kk^{-1}: M_ij -= M_ik P M_kj (i, j != k);
// M_kj <- P M_kj; M_ik <- -M_ik P; M_kk <- P.  The pivots may be swept in any order
// (each is a Schur complement of a positive definite matrix), and the swept form
// stays Hermitian up to sign: S_ij = S_ji^H when i and j are both swept or both not,
// S_ij = -S_ji^H otherwise.  So with C_b = M_bk (b != k) and N_b = C_b P the row panel
// is M_kb -> s_b N_b^H, s_b = +1 for unswept and -1 for swept b, and every stored
// tile is updated as M_IJ -= s_J C_I N_J^H.
//
// Block row b takes part in the sweep of k only if M_bk is not zero.  The coarsest
// stencil couples a block to few others, and swept blocks only to what has grown
// together around them, so the plan (made on the host from the block graph) sweeps
// the block with the fewest couplings next, which orders separators last, and sweeps
// blocks without a common coupling in one pair of launches.  At 16 x 16 sites of 16
// dof (64 blocks) 25,840 tile products in 28 groups are left of 129,024 in 64 steps,
// at 32 x 32 sites a tenth.  Skipped products are with zero blocks: the arithmetic on
// the rest is unchanged.  4096 unknowns: 8.0 -> 1.85 ms (the update of every tile in order
// took 64 x 101 us, its panels 64 x 24 us).
#include <algorithm>
#include <numeric>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "mma_tf32.cuh"

namespace mgk {

namespace {

static constexpr int B = 64;                     // block size
static constexpr int LA = B + 1;                 // row stride of a block being inverted
static constexpr int LD = 66;                    // row stride (float2) of staged tiles: the
                                                 // fragment loads of a warp hit 32 banks
static constexpr int TILE = B * B;
static constexpr int GMAX = 8;                   // pivots per group

// In-place inversion of the Hermitian positive definite 64 x 64 block a[][LA] in shared
// memory by 256 threads: four 16 x 16 sub-pivots K, each swept with one entry per thread (in
// a register; the rows and columns others need go through two alternating buffers, one barrier
// a step), then the row panel T = P a_Kx and the rank-16 update of the other 48 x 48 entries,
// 3 x 3 per thread; the column panel follows from T by the sign rule.  The diagonal of a
// Hermitian block is real, so a pivot is inverted by one division.  tmp: [16][48] complex.
// With its launch 28 us (36 with the sub-pivot in one warp's registers: 16 unrolled steps of
// cold instructions; 42 with two barriers and a complex division a step).
__device__ void invert64(float2* a, float2* tmp) {
  const int tid = threadIdx.x, ti = tid >> 4, tj = tid & 15;
#pragma unroll 1
  for (int K = 0; K < 4; ++K) {
    const int k0 = 16 * K;
    float2 v = a[(k0 + ti) * LA + k0 + tj];
    tmp[ti * 17 + tj] = v;
    __syncthreads();
#pragma unroll 2
    for (int p = 0; p < 16; ++p) {
      const float2* s = tmp + (p & 1) * 16 * 17;
      const float inv = 1.f / s[p * 17 + p].x;
      const float2 rp = s[p * 17 + tj], cp = s[ti * 17 + p];
      const float2 f = make_float2(inv * rp.x, inv * rp.y);
      if (tj == p)
        v = ti == p ? make_float2(inv, 0.f) : make_float2(-inv * cp.x, -inv * cp.y);
      else
        v = ti == p ? f : csub(v, cmul(cp, f));
      tmp[((p + 1) & 1) * 16 * 17 + ti * 17 + tj] = v;
      __syncthreads();
    }
    a[(k0 + ti) * LA + k0 + tj] = v;
    __syncthreads();
    {                                              // T[q][x], q = ti, x = tj + 16 u
      float2 acc[3] = {};
#pragma unroll 4
      for (int s = 0; s < 16; ++s) {
        const float2 p = a[(k0 + ti) * LA + k0 + s];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const int x = tj + 16 * u, col = x < k0 ? x : x + 16;
          cfma(acc[u], p, a[(k0 + s) * LA + col]);
        }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) tmp[ti * 48 + tj + 16 * u] = acc[u];
    }
    __syncthreads();
    float2 nv[3][3];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        const int xi = ti + 16 * u, xj = tj + 16 * w;
        nv[u][w] = a[(xi < k0 ? xi : xi + 16) * LA + (xj < k0 ? xj : xj + 16)];
      }
#pragma unroll 2
    for (int s = 0; s < 16; ++s) {
      float2 cv[3], rv[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int xi = ti + 16 * u;
        cv[u] = a[(xi < k0 ? xi : xi + 16) * LA + k0 + s];
        rv[u] = tmp[s * 48 + tj + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < 3; ++u)
#pragma unroll
        for (int w = 0; w < 3; ++w) cfma(nv[u][w], make_float2(-cv[u].x, -cv[u].y), rv[w]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 3; ++u) {
#pragma unroll
      for (int w = 0; w < 3; ++w) {
        const int xi = ti + 16 * u, xj = tj + 16 * w;
        a[(xi < k0 ? xi : xi + 16) * LA + (xj < k0 ? xj : xj + 16)] = nv[u][w];
      }
      // row panel a_Kx = T and column panel a_xK = -s T^H, s = +1 for unswept x, else -1
      const int x = tj + 16 * u, col = x < k0 ? x : x + 16;
      const float2 t = tmp[ti * 48 + x];
      a[(k0 + ti) * LA + col] = t;
      a[col * LA + k0 + ti] = x < k0 ? make_float2(t.x, -t.y) : make_float2(-t.x, t.y);
    }
    __syncthreads();
  }
}

// One group of pivots on the device (offsets into the plan's int array):
//   panels: {block b, pivot index, swept flag of b} per coupled block and pivot, then
//   one entry per pivot with b = the pivot block itself;
//   piv: the pivot blocks; next: the pivot blocks of the next group;
//   act: the blocks coupled to any pivot, act_mask: the pivots they couple to (bit i),
//   bit 30 swept, bit 31 pivot of the next group; slot[u * GMAX + i]: panel slot.
struct GroupArgs {
  const int3* panels;
  const int *piv, *next, *act, *act_mask, *slot;
  int npiv, nnext, nact;
  const float2* P;                               // inverted pivots of this group
  float2* Pnext;
  float2 *C, *N;                                 // panel tiles per slot
};

__global__ void __launch_bounds__(256) k_gji_first(const float2* __restrict__ M, int ld, GroupArgs g, int dependent) {
  pdl_wait(dependent, M);
  __shared__ float2 a[B * LA], tmp[16 * 48];
  const long long k = g.next[blockIdx.x];
  for (int q = threadIdx.x; q < TILE; q += 256) a[(q / B) * LA + q % B] = M[(k * B + q / B) * ld + k * B + q % B];
  __syncthreads();
  invert64(a, tmp);
  for (int q = threadIdx.x; q < TILE; q += 256) g.Pnext[blockIdx.x * TILE + q] = a[(q / B) * LA + q % B];
}

// Panels of a group: C_b = M_bk from the stored lower tile, N_b = C_b P, and the swept tile
// written back in place (M_bk <- -N_b, or M_kb <- s_b N_b^H when the stored tile is (k, b));
// the pivot tile itself becomes P.  Four CTAs per (block, pivot), 16 rows of C_b each: they
// read and write only their own rows (or columns) of the stored tile.  A group has 20 to 72
// panels, too few to fill the GPU with one CTA each (12 us; four 7 to 10 us).
__global__ void __launch_bounds__(256) k_gji_panel(float2* __restrict__ M, int ld, GroupArgs g, int dependent) {
  pdl_wait(dependent, M);
  __shared__ __align__(16) float2 sP[B * B];
  __shared__ __align__(16) float2 sX[16 * (B + 1)];
  const int3 e = g.panels[blockIdx.x];
  const int b = e.x, k = g.piv[e.y], tid = threadIdx.x, r0 = 16 * blockIdx.y;
  const float2* P = g.P + e.y * TILE;
  if (b == k) {
    for (int q = tid; q < 16 * B; q += 256)
      M[((long long)k * B + r0 + q / B) * ld + k * B + q % B] = P[r0 * B + q];
    return;
  }
  const bool lower = b > k;                      // the stored tile is (b, k)
  float2* tile = M + (long long)(lower ? b : k) * B * ld + (long long)(lower ? k : b) * B;
  const float sg = e.z ? -1.f : 1.f;
  float4 p[8];
  float2 v[4];
#pragma unroll
  for (int u = 0; u < 8; ++u) p[u] = ((const float4*)P)[tid + 256 * u];
#pragma unroll
  for (int u = 0; u < 4; ++u) {                  // lower: row r0 + q / 64; else column r0 + q % 16
    const int q = tid + 256 * u;
    v[u] = lower ? tile[(long long)(r0 + q / B) * ld + q % B] : tile[(long long)(q / 16) * ld + r0 + q % 16];
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) ((float4*)sP)[tid + 256 * u] = p[u];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int q = tid + 256 * u;
    if (lower)
      sX[(q / B) * (B + 1) + q % B] = v[u];
    else                                         // M_bk = s_b M_kb^H
      sX[(q % 16) * (B + 1) + q / 16] = make_float2(sg * v[u].x, -sg * v[u].y);
  }
  __syncthreads();
  const int r = tid >> 4, c0 = tid & 15;         // row r0 + r, columns c0 + 16 u
  float2 acc[4] = {};
#pragma unroll 8
  for (int q = 0; q < B; ++q) {
    const float2 x = sX[r * (B + 1) + q];
#pragma unroll
    for (int u = 0; u < 4; ++u) cfma(acc[u], x, sP[q * B + c0 + 16 * u]);
  }
  float2* C = g.C + (long long)blockIdx.x * TILE + (r0 + r) * B;
  float2* N = g.N + (long long)blockIdx.x * TILE + (r0 + r) * B;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = c0 + 16 * u;
    const float2 w = acc[u];
    C[c] = sX[r * (B + 1) + c];
    N[c] = w;
    if (lower) tile[(long long)(r0 + r) * ld + c] = make_float2(-w.x, -w.y);
  }
  if (!lower) {                                  // s_b N_b^H, transposed through shared memory
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
      sX[r * (B + 1) + c0 + 16 * u] = make_float2(sg * acc[u].x, -sg * acc[u].y);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = tid + 256 * u;
      tile[(long long)(q / 16) * ld + r0 + q % 16] = sX[(q % 16) * (B + 1) + q / 16];
    }
  }
}

// Tiles of a group: M_IJ -= s_J sum over its pivots of C_I N_J^H for every pair I >= J of
// coupled blocks (pairs without a common pivot return).  The leading CTAs take the diagonal
// tiles of the next group's pivots and invert them, so that this overlaps with the other tiles.
//
// The complex product runs on the tensor cores as a real GEMM: A = C_I with (re, im)
// interleaved along K (64 x 128), B[2q + c][2j + d] from N_J row j: (re, im) for d = 0,
// (-im, re) for d = 1; m16n8k8 TF32 with three products per FP32-accurate product.  8 warps
// in a 2 x 4 grid, 32 x 32 real outputs each; lane (g, t) holds complex outputs (row g or
// g + 8, column t) of each 16 x 4 complex sub-tile.
__global__ void __launch_bounds__(256, 3) k_gji_update(float2* __restrict__ M, int ld, GroupArgs g, int dependent) {
  pdl_wait(dependent, M);
  extern __shared__ float2 usm[];
  float2* sC = usm;                              // C_I [64][LD]
  float2* sN = usm + B * LD;                     // N_J [64][LD]
  const int tid = threadIdx.x;
  int I, J, ui = -1, uj = -1;
  const bool invert = blockIdx.x < g.nnext;
  if (invert) {
    I = J = g.next[blockIdx.x];
    for (int u = 0; u < g.nact; ++u)
      if (g.act[u] == I) ui = uj = u;
  } else {
    const int t = blockIdx.x - g.nnext;
    ui = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((ui + 1) * (ui + 2) / 2 <= t) ++ui;
    while (ui * (ui + 1) / 2 > t) --ui;
    uj = t - ui * (ui + 1) / 2;
    I = g.act[ui];                               // act is ascending: I >= J
    J = g.act[uj];
    if (ui == uj && g.act_mask[ui] < 0) return;  // a next pivot: taken by its own CTA
  }
  unsigned mask = ui < 0 ? 0u : (unsigned)(g.act_mask[ui] & g.act_mask[uj]) & 0xffu;
  if (!mask && !invert) return;
  const float sg = uj >= 0 && (g.act_mask[uj] >> 30 & 1) ? -1.f : 1.f;
  float2* tile = M + (long long)I * B * ld + (long long)J * B;
  const int warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
  const int wm = warp >> 2, wn = warp & 3;       // rows 32 wm.., complex columns 16 wn..
  float acc[2][4][4];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[mt][n][e] = 0.f;
  bool first = true;
  for (; mask; mask &= mask - 1) {
    const int i = __ffs(mask) - 1;
    const float4* c = (const float4*)(g.C + (long long)g.slot[ui * GMAX + i] * TILE);
    const float4* n = (const float4*)(g.N + (long long)g.slot[uj * GMAX + i] * TILE);
    float4 vc[8], vn[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      vc[u] = c[tid + 256 * u];
      vn[u] = n[tid + 256 * u];
    }
    if (!first) __syncthreads();
    first = false;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int q = 2 * (tid + 256 * u), r = q / B, cc = q % B;
      *(float4*)&sC[r * LD + cc] = vc[u];
      *(float4*)&sN[r * LD + cc] = vn[u];
    }
    __syncthreads();
    const float *fC = (const float*)sC, *fN = (const float*)sN;
#pragma unroll 2
    for (int kk = 0; kk < 2 * B / 8; ++kk) {     // 16 real k-steps of 8
      uint32_t ah[2][4], al[2][4], bh[4][2], bl[4][2];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        const float* r0 = fC + (32 * wm + 16 * mt + gq) * 2 * LD + 8 * kk + tq;
        const float* r8 = r0 + 8 * 2 * LD;
        split_tf32(r0[0], ah[mt][0], al[mt][0]);
        split_tf32(r8[0], ah[mt][1], al[mt][1]);
        split_tf32(r0[4], ah[mt][2], al[mt][2]);
        split_tf32(r8[4], ah[mt][3], al[mt][3]);
      }
#pragma unroll
      for (int nn = 0; nn < 4; ++nn) {
        // B[8 kk + tq (+ 4)][8 n' + gq]: column j = 4 n' + gq / 2, d = gq % 2
        const int j = 16 * wn + 4 * nn + (gq >> 1), d = gq & 1;
        const float* r = fN + j * 2 * LD + 8 * kk + (tq ^ d);
        const float s = d && !(tq & 1) ? -1.f : 1.f;
        split_tf32(s * r[0], bh[nn][0], bl[nn][0]);
        split_tf32(s * r[4], bh[nn][1], bl[nn][1]);
      }
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nn = 0; nn < 4; ++nn) {
          mma_tf32(acc[mt][nn], al[mt], bh[nn]);
          mma_tf32(acc[mt][nn], ah[mt], bl[nn]);
          mma_tf32(acc[mt][nn], ah[mt], bh[nn]);
        }
    }
  }
  if (invert) __syncthreads();                   // sC is reused for the new tile
  float2 old[2][4][2];                           // all tile loads before the stores
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        old[mt][n][h] = tile[(long long)(32 * wm + 16 * mt + gq + 8 * h) * ld + 16 * wn + 4 * n + tq];
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int n = 0; n < 4; ++n)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 32 * wm + 16 * mt + gq + 8 * h, c = 16 * wn + 4 * n + tq;
        const float2 o = old[mt][n][h];
        const float2 nv = make_float2(o.x - sg * acc[mt][n][2 * h], o.y - sg * acc[mt][n][2 * h + 1]);
        tile[(long long)r * ld + c] = nv;
        if (invert) sC[r * LA + c] = nv;
      }
  if (invert) {
    __syncthreads();
    invert64(sC, sN);
    for (int q = tid; q < TILE; q += 256) g.Pnext[blockIdx.x * TILE + q] = sC[(q / B) * LA + q % B];
  }
}

}  // namespace

// Plan from the stencil: blocks a, b are coupled when a site of a neighbours a site of b.
InversePlan inverse_plan(int Lx, int Lt, int n, int ld) {
  InversePlan plan;
  const int nt = ld / B, words = (nt + 63) / 64;
  std::vector<uint64_t> adj((size_t)nt * words, 0);
  auto set = [&](int a, int b) { adj[(size_t)a * words + b / 64] |= 1ull << (b % 64); };
  auto has = [&](int a, int b) { return adj[(size_t)a * words + b / 64] >> (b % 64) & 1; };
  for (int b = 0; b < nt; ++b) set(b, b);
  for (int j = 0; j < Lx * Lt; ++j)
    for (int d = 0; d < 9; ++d) {
      const int x = (j % Lx + d % 3 - 1 + Lx) % Lx, t = (j / Lx + d / 3 - 1 + Lt) % Lt, k = x + Lx * t;
      for (int a = j * n / B; a <= (j * n + n - 1) / B; ++a)
        for (int b = k * n / B; b <= (k * n + n - 1) / B; ++b) set(a, b);
    }
  std::vector<char> swept(nt, 0);
  std::vector<std::vector<int>> groups;
  std::vector<std::vector<std::vector<int>>> coupled;    // per group and pivot
  std::vector<std::vector<char>> status;                 // swept flags before each group
  int left = nt;
  while (left > 0) {
    std::vector<int> deg(nt, 0), order;
    for (int k = 0; k < nt; ++k) {
      if (swept[k]) continue;
      for (int w = 0; w < words; ++w) deg[k] += __builtin_popcountll(adj[(size_t)k * words + w]);
      deg[k] -= 1;
      order.push_back(k);
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return deg[a] < deg[b]; });
    const double limit = 1.6 * deg[order[0]] + 4.0;
    std::vector<int> grp;
    int total = 0;
    for (int k : order) {
      if (deg[k] > limit || (int)grp.size() == GMAX) break;
      bool apart = grp.empty() || total + deg[k] <= nt;   // panel tiles of a group: at most nt
      for (int p : grp) apart = apart && !has(k, p);
      if (!apart) continue;
      grp.push_back(k);
      total += deg[k];
    }
    std::vector<std::vector<int>> nb;
    for (int k : grp) {
      std::vector<int> c;
      for (int b = 0; b < nt; ++b)
        if (b != k && has(k, b)) c.push_back(b);
      nb.push_back(c);
    }
    status.push_back(swept);
    for (size_t i = 0; i < grp.size(); ++i) {
      for (int a : nb[i])
        for (int w = 0; w < words; ++w) adj[(size_t)a * words + w] |= adj[(size_t)grp[i] * words + w];
      swept[grp[i]] = 1;
      --left;
    }
    groups.push_back(grp);
    coupled.push_back(nb);
  }
  std::vector<int>& v = plan.data;
  for (size_t q = 0; q < groups.size(); ++q) {
    InversePlan::Group G;
    G.npiv = (int)groups[q].size();
    G.nnext = q + 1 < groups.size() ? (int)groups[q + 1].size() : 0;
    std::vector<int> slot((size_t)nt * GMAX, -1), mask(nt, 0);
    G.panels = (int)v.size();
    int s = 0;
    for (int i = 0; i < G.npiv; ++i)
      for (int b : coupled[q][i]) {
        v.insert(v.end(), {b, i, (int)status[q][b]});
        slot[(size_t)b * GMAX + i] = s++;
        mask[b] |= 1 << i;
      }
    for (int i = 0; i < G.npiv; ++i) v.insert(v.end(), {groups[q][i], i, 0});
    G.npanels = s + G.npiv;
    G.piv = (int)v.size();
    v.insert(v.end(), groups[q].begin(), groups[q].end());
    G.next = (int)v.size();
    if (G.nnext) v.insert(v.end(), groups[q + 1].begin(), groups[q + 1].end());
    std::vector<char> isnext(nt, 0);
    for (int i = 0; i < G.nnext; ++i) isnext[groups[q + 1][i]] = 1;
    std::vector<int> act;
    for (int b = 0; b < nt; ++b)
      if (mask[b]) act.push_back(b);
    G.nact = (int)act.size();
    G.act = (int)v.size();
    v.insert(v.end(), act.begin(), act.end());
    G.mask = (int)v.size();
    for (int b : act) v.push_back(mask[b] | (status[q][b] ? 1 << 30 : 0) | (isnext[b] ? (int)0x80000000u : 0));
    G.slot = (int)v.size();
    for (int b : act) v.insert(v.end(), slot.begin() + (size_t)b * GMAX, slot.begin() + (size_t)(b + 1) * GMAX);
    plan.groups.push_back(G);
  }
  plan.first = plan.groups.empty() ? 0 : plan.groups[0].piv;
  return plan;
}

// Work (complex64 entries): the C and N tiles of a group's panels, the inverted pivots of
// this and of the next group.
size_t inverse_work_entries(int ld) { return (size_t)2 * ld * B + (size_t)2 * GMAX * TILE; }

cudaError_t inverse_first(void* M, int ld, const InversePlan& plan, const int* data, void* work,
                          cudaStream_t s) {
  static SmemLimit limit;
  const cudaError_t e0 = limit.raise(k_gji_update, (int)(2 * B * LD * sizeof(float2)));
  if (e0 != cudaSuccess) return e0;
  GroupArgs g{};
  g.next = data + plan.first;
  g.Pnext = (float2*)work + (size_t)2 * ld * B;
  launch_after(k_gji_first, plan.groups[0].npiv, 256, 0, s, (const float2*)M, ld, g);
  count_launch();
  return cudaGetLastError();
}

cudaError_t inverse_group(void* M, int ld, const InversePlan& plan, const int* data, int q, void* work,
                          bool update, cudaStream_t s) {
  const InversePlan::Group& G = plan.groups[q];
  float2* P = (float2*)work + (size_t)2 * ld * B;
  GroupArgs g{(const int3*)(data + G.panels), data + G.piv, data + G.next, data + G.act,
              data + G.mask, data + G.slot, G.npiv, G.nnext, G.nact,
              P + (size_t)(q & 1) * GMAX * TILE, P + (size_t)((q + 1) & 1) * GMAX * TILE,
              (float2*)work, (float2*)work + (size_t)ld * B};
  const size_t smem = 2 * B * LD * sizeof(float2);
  if (!update) {
    launch_after(k_gji_panel, dim3(G.npanels, B / 16), 256, 0, s, (float2*)M, ld, g);
  } else {
    const int grid = G.nnext + G.nact * (G.nact + 1) / 2;
    if (grid == 0) return cudaSuccess;
    launch_after(k_gji_update, grid, 256, smem, s, (float2*)M, ld, g);
  }
  count_launch();
  return cudaGetLastError();
}

}  // namespace mgk
