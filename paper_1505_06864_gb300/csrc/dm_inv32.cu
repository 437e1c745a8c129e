// Float32 block inverse G_t = D_t^{-1}: blocked Gauss-Jordan with implicit
// partial pivoting (rows keep their place, as in dm_gj.cu), one CTA per block
// with the block in shared memory, panels of eight columns.
//
// Per panel four warps run the pivots, a row (or two) per lane, the panel's
// eight columns in registers: float32 multiply-adds are cheap, so each pivot
// is the exchange alone (two warp reductions, one CTA barrier, the winner's
// row from shared memory, one reciprocal).  Then all eight warps apply the
// rank-8 update to the other columns, a lane per column with the eight pivot
// rows' entries in registers, a row per warp at a time (its eight multipliers
// by broadcast).  An inverse that updates the whole block per pivot pays that
// exchange with 1024 threads at a barrier: 163 us for 97 blocks of m = 128,
// this one 85 us (per panel about 4000 cycles for the eight pivots and 5000 for
// the update, of which the multiply-adds are 1000 and the block's trip through
// shared memory the rest).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dm_internal.cuh"

namespace dm {
namespace inv32 {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kChain = 4;
constexpr int SW = 8;
constexpr int kMaxRows = 256;

struct Shared {
  float4 row[2][kChain][2];         // the warps' candidate rows
  uint32_t key[2][kChain];          // 0: no eligible row; else the bits of |value| + 1
  int idx[2][kChain];
  float U[kMaxRows][SW];            // the eliminated panel
  int order[kMaxRows], place[kMaxRows];  // pivot row of every column; column of every pivot row
  uint32_t used[kMaxRows / 32], panel[kMaxRows / 32];  // pivot rows so far; of this panel
  int bad;
};

// The pivots of the columns c0 .. c0 + w - 1 on warps 0 .. nw - 1: lane holds
// rows 32 warp + lane + 128 i.  Register c holds column (j - 1 + c) mod 8
// before pivot j; the pivot's own row takes part as zeros plus the reciprocal
// times itself.  While a pivot is left some row is eligible, with a key of at
// least 1; were none, the pivot would count as unusable, and the row stays
// inside the block.
template <int RPL>
__device__ __forceinline__ void chain(float* M, int ld, int m, int c0, int w, int nw, Shared& sh, int warp, int lane) {
  float a[RPL][SW], fn[RPL], s[SW];
  bool dead[RPL];
#pragma unroll
  for (int c = 0; c < SW; ++c) s[c] = 0.f;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int row = 32 * warp + lane + 128 * i;
    dead[i] = row >= m || ((sh.used[row >> 5] >> (row & 31)) & 1u) != 0;
    fn[i] = 0.f;
#pragma unroll
    for (int c = 0; c < SW; ++c) {
      const int col = c0 + ((c + 7) & 7);
      a[i][c] = row < m && col < m ? M[row * ld + col] : 0.f;
    }
  }
#pragma unroll 2
  for (int j = 0; j < w; ++j) {
    uint32_t key = 0;
    int bi = 0;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const float last = fmaf(fn[i], s[0], a[i][0]);
#pragma unroll
      for (int c = 1; c < SW; ++c) a[i][c - 1] = fmaf(fn[i], s[c], a[i][c]);
      a[i][SW - 1] = last;
      const uint32_t b = __float_as_uint(a[i][0]) & 0x7fffffffu;
      const uint32_t ki = dead[i] ? 0u : (b > 0x7f800000u ? 0u : b) + 1u;  // NaN counts as zero
      if (i == 0 || ki > key) key = ki, bi = i;
    }
    const uint32_t wkey = __reduce_max_sync(0xffffffffu, key);
    const int src = (int)__reduce_min_sync(0xffffffffu, key == wkey ? (uint32_t)lane : 32u);
    const int buf = j & 1;
    if (lane == src) {
#pragma unroll
      for (int i = 0; i < RPL; ++i)
        if (bi == i) {
          sh.row[buf][warp][0] = make_float4(a[i][0], a[i][1], a[i][2], a[i][3]);
          sh.row[buf][warp][1] = make_float4(a[i][4], a[i][5], a[i][6], a[i][7]);
        }
      sh.key[buf][warp] = wkey;
      sh.idx[buf][warp] = 32 * warp + lane + 128 * bi;
    }
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nw) : "memory");
    int best = 0;
    uint32_t kb = sh.key[buf][0];
#pragma unroll
    for (int q = 1; q < kChain; ++q)
      if (q < nw && sh.key[buf][q] > kb) kb = sh.key[buf][q], best = q;
    const float4 lo = sh.row[buf][best][0], hi = sh.row[buf][best][1];
    const int prow = min(sh.idx[buf][best], m - 1);
    float inv = __frcp_rn(lo.x);
    const bool unusable = kb == 0 || !(fabsf(lo.x) > 0.f) || !isfinite(inv);
    if (unusable) inv = 0.f;
    s[0] = 1.f;
    s[1] = lo.y, s[2] = lo.z, s[3] = lo.w, s[4] = hi.x, s[5] = hi.y, s[6] = hi.z, s[7] = hi.w;
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
      const bool isp = 32 * warp + lane + 128 * i == prow;
      fn[i] = isp ? inv : -a[i][0] * inv;
      a[i][0] = 0.f;
      if (isp) {
        dead[i] = true;
#pragma unroll
        for (int c = 1; c < SW; ++c) a[i][c] = 0.f;
      }
    }
    if (warp == 0 && lane == 0) {
      sh.order[c0 + j] = prow;
      sh.place[prow] = c0 + j;
      if (unusable) sh.bad = 1;
    }
  }
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int row = 32 * warp + lane + 128 * i;
    if (row < m)
#pragma unroll
      for (int c = 0; c < SW; ++c) {
        const int cc = (w - 1 + c) & 7;
        const float v = fmaf(fn[i], s[c], a[i][c]);
        sh.U[row][cc] = v;
        if (c0 + cc < m) M[row * ld + c0 + cc] = v;
      }
  }
}

template <int RPL>
__global__ void __launch_bounds__(kThreads) k_inv_f32(const PartDesc* __restrict__ parts, int t,
                                                      const double* __restrict__ B, float* __restrict__ G,
                                                      int* __restrict__ status) {
  extern __shared__ __align__(16) float M[];
  __shared__ Shared sh;
  constexpr int CC = 4 * RPL;  // columns per lane
  const PartDesc p = parts[blockIdx.x];
  if (t >= p.L) return;
  const int m = p.m, ld = m | 1, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nw = min(kChain, (m + 31) / 32);
  const long long o = p.blk + (long long)t * m * m;
  float* g = G + o;
  if (tid < kMaxRows / 32) sh.used[tid] = 0;
  if (tid == 0) sh.bad = 0;
  if (t == 0)
#pragma unroll 16
    for (int e = tid; e < m * m; e += kThreads) M[(e / m) * ld + e % m] = (float)B[o + e];
  else
#pragma unroll 16
    for (int e = tid; e < m * m; e += kThreads) M[(e / m) * ld + e % m] = g[e];
  __syncthreads();
#pragma unroll 1
  for (int c0 = 0; c0 < m; c0 += SW) {
    const int w = min(SW, m - c0);
    if (warp < nw) chain<RPL>(M, ld, m, c0, w, nw, sh, warp, lane);
    else if (warp == kWarps - 1 && lane < kMaxRows / 32) sh.panel[lane] = 0;
    __syncthreads();
    // the panel's pivot rows in this lane's columns
    float v[SW][CC];
#pragma unroll
    for (int j = 0; j < SW; ++j) {
      const int row = sh.order[c0 + min(j, w - 1)];
#pragma unroll
      for (int q = 0; q < CC; ++q) v[j][q] = j < w && lane + 32 * q < m ? M[row * ld + lane + 32 * q] : 0.f;
    }
    if (tid < w) {
      const int row = sh.order[c0 + tid];
      atomicOr(&sh.used[row >> 5], 1u << (row & 31));
      atomicOr(&sh.panel[row >> 5], 1u << (row & 31));
    }
    __syncthreads();
    constexpr int RR = 4;  // rows at once: their loads before the first multiply-add
    for (int r0 = warp; r0 < m; r0 += kWarps * RR) {
      float x[RR][CC];
      float4 u[RR][2];
#pragma unroll
      for (int h = 0; h < RR; ++h) {
        const int row = min(r0 + kWarps * h, m - 1);
        const bool z = ((sh.panel[row >> 5] >> (row & 31)) & 1u) != 0;
        u[h][0] = *reinterpret_cast<const float4*>(&sh.U[row][0]);
        u[h][1] = *reinterpret_cast<const float4*>(&sh.U[row][4]);
#pragma unroll
        for (int q = 0; q < CC; ++q) x[h][q] = z || lane + 32 * q >= m ? 0.f : M[row * ld + lane + 32 * q];
      }
#pragma unroll
      for (int h = 0; h < RR; ++h)
#pragma unroll
        for (int q = 0; q < CC; ++q) {
          x[h][q] = fmaf(u[h][0].x, v[0][q], x[h][q]);
          x[h][q] = fmaf(u[h][0].y, v[1][q], x[h][q]);
          x[h][q] = fmaf(u[h][0].z, v[2][q], x[h][q]);
          x[h][q] = fmaf(u[h][0].w, v[3][q], x[h][q]);
          x[h][q] = fmaf(u[h][1].x, v[4][q], x[h][q]);
          x[h][q] = fmaf(u[h][1].y, v[5][q], x[h][q]);
          x[h][q] = fmaf(u[h][1].z, v[6][q], x[h][q]);
          x[h][q] = fmaf(u[h][1].w, v[7][q], x[h][q]);
        }
#pragma unroll
      for (int h = 0; h < RR; ++h)
#pragma unroll
        for (int q = 0; q < CC; ++q) {
          const int c = lane + 32 * q, row = r0 + kWarps * h;
          if (row < m && c < m && (c < c0 || c >= c0 + w)) M[row * ld + c] = x[h][q];
        }
    }
    __syncthreads();
  }
  // D^{-1}[k][p_j] = M[p_k][j]
  for (int k = warp; k < m; k += kWarps) {
    const float* src = M + sh.order[k] * ld;
#pragma unroll
    for (int q = 0; q < CC; ++q) {
      const int c = lane + 32 * q;
      if (c < m) g[(long long)k * m + c] = src[sh.place[c]];
    }
  }
  if (tid == 0 && sh.bad) atomicMin(status + p.sys, p.row0 + t + 1);
}

}  // namespace inv32

// Blocks of up to this size fit with the rest in a CTA's shared memory.
int inv_f32_max_m() { return 224; }

void launch_inv_f32(const PartDesc* parts, int nparts, int t, const double* B, float* G, int* status, int max_m,
                    cudaStream_t st) {
  if (nparts <= 0) return;
  const size_t smem = (size_t)max_m * (max_m | 1) * sizeof(float);
  auto go = [&](auto kernel) {
    allow_smem(kernel, smem);
    kernel<<<nparts, inv32::kThreads, smem, st>>>(parts, t, B, G, status);
  };
  if (max_m <= 128) go(inv32::k_inv_f32<1>);
  else go(inv32::k_inv_f32<2>);
}

}  // namespace dm
