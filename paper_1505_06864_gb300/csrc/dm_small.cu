// Factor sweeps of float64 levels with small blocks (m <= 32), one CTA per
// subsystem and one launch per level: the forward sweep (inverse, Acal, the
// next Schur block, the left spike; Section 3 applied to Eq. e231) and the
// backward spike sweep, with every block of the current row in shared memory.
// Per row the step kernels of the larger levels take about a dozen dependent
// launches of 4 to 15 us each, whatever the size; here a row costs the float64
// work itself: at m = 16 about 2 us per two products (the float64 unit of one
// SM: two multiply-adds per clock) and 4 us for the sixteen pivots.
//
// The inverse is Gauss-Jordan with implicit partial pivoting (rows keep their
// place, as in dm_gj.cu): four warps, a row per lane, ceil(m / 4) columns per
// warp in registers; the warp that owns the next pivot column updates it
// first, searches it (largest high word of |value|, candidates that agree to
// 2^-20 counting as equal) and publishes its multipliers before it updates its
// other columns.  The other four warps fetch the next row's blocks meanwhile.
//
// Factor + solve against the step kernels (us): m = 4 N = 64 342 / 627, m = 8
// 420 / 908, m = 16 798 / 1354, m = 32 1391 / 1774; N = 4096 (97 subsystems) m =
// 16 2471 / 4939, m = 32 4653 / 6632; 400 systems of N = 200, m = 32 (8800
// subsystems) 39.0 / 55.3 ms: faster for every m <= 32 and any number of
// subsystems.  (Above, a product's m^3 / 2 cycles on one SM outgrow the launches.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dm_internal.cuh"
#include "dm_recip.cuh"

namespace dm {
namespace small {

constexpr int kThreads = 256;
constexpr int kInvWarps = 4;
constexpr int MS = kSmallM;      // largest block
constexpr int LD = MS + 1;       // row stride in shared memory
constexpr int BLK = MS * LD;     // one block
constexpr int kBlocks = 7;       // D, G, X (Acal), Y, Z (ZL), A, C; B is added to D on the way

struct Pivot {
  double inv;
  int row, pad;
};

struct Shared {
  double f[2][32];  // the pivot column, double-buffered by the pivot's parity
  Pivot pv[2];
  int order[MS];    // pivot row of every column
};

// Gauss-Jordan on warps 0 .. 3; CPW columns per warp.  D in `D`, the inverse
// to `G`.
template <int CPW>
__device__ __forceinline__ void invert(const double* D, double* G, int m, Shared& sh, int warp, int lane, bool& bad) {
  double a[CPW];
  const int c0 = warp * CPW;
#pragma unroll
  for (int c = 0; c < CPW; ++c) a[c] = lane < m && c0 + c < m ? D[lane * LD + c0 + c] : 0.0;
  bool dead = lane >= m;
  int step = 0;  // the column this lane's row is the pivot of
  // the search of column j on its owner warp, values v (the row is a lane's
  // number, so it stays inside the 32 rows of every shared array)
  auto publish = [&](double v, int j) {
    const uint32_t key = dead ? 0u : abs_hi(v) + 1u;
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
    const int src = (int)__reduce_min_sync(0xffffffffu, key == kmax ? (uint32_t)lane : 32u);
    double inv = pivot_unusable(v) ? 0.0 : pivot_recip(v);
    sh.f[j & 1][lane] = v;
    if (lane == src) {
      // near the ends of the range the division (the blocks are not equilibrated here)
      if (__double_as_longlong(inv) == 0) inv = pivot_recip_any(v);
      sh.pv[j & 1] = Pivot{inv, lane, 0};
      sh.order[j] = lane;
      if (__double_as_longlong(inv) == 0) bad = true;
    }
  };
  if (warp == 0) publish(a[0], 0);
#pragma unroll 1
  for (int w = 0; w < kInvWarps; ++w) {
#pragma unroll
    for (int c = 0; c < CPW; ++c) {
      const int j = w * CPW + c;
      if (j >= m) break;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      const Pivot pv = sh.pv[j & 1];
      const double f = sh.f[j & 1][lane];
      const bool isp = lane == pv.row;
      // this row minus its multiplier times the pivot row; the pivot's own row
      // as zeros plus the reciprocal times itself
      const double fn = isp ? pv.inv : -f * pv.inv;
      if (isp) dead = true, step = j;
      auto update = [&](int cc) {
        const double u = __shfl_sync(0xffffffffu, a[cc], pv.row);
        a[cc] = warp == w && cc == c ? fn : fma(fn, u, isp ? 0.0 : a[cc]);
      };
      constexpr int last = CPW - 1;
      const int nx = c == last ? 0 : c + 1;  // the next pivot's column in its owner
      update(nx);
      if (j + 1 < m && warp == (c == last ? w + 1 : w)) publish(a[nx], j + 1);
#pragma unroll
      for (int cc = 0; cc < CPW; ++cc)
        if (cc != nx) update(cc);
    }
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");
  if (lane < m)
#pragma unroll
    for (int c = 0; c < CPW; ++c)
      if (c0 + c < m) G[step * LD + sh.order[c0 + c]] = a[c];
}

// epi(row, column, sum_k L[row][k] R[k][column]): four rows per thread where
// the block has that many.
template <typename Epi>
__device__ __forceinline__ void product(const double* L, const double* R, int m, int tid, Epi epi) {
  const int per = max(1, kThreads / m), c = tid % m, r0 = tid / m;  // `per` rows at once
  if (r0 >= per) return;
  for (int r = r0; r < m; r += 4 * per) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    const int n = min(4, (m - r + per - 1) / per);
    for (int k = 0; k < m; ++k) {
      const double b = R[k * LD + c];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < n) acc[q] = fma(L[(r + q * per) * LD + k], b, acc[q]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < n) epi(r + q * per, c, acc[q]);
  }
}

// The same where R has its nonzeros within w of the diagonal (LEFT: L has):
// 2w + 1 terms per entry, the others are exact zeros.
template <bool LEFT, typename Epi>
__device__ __forceinline__ void band_product(const double* L, const double* R, int m, int w, int tid, Epi epi) {
  for (int e = tid; e < m * m; e += kThreads) {
    const int r = e / m, c = e - r * m, mid = LEFT ? r : c;
    double acc = 0.0;
    for (int k = max(0, mid - w); k <= min(m - 1, mid + w); ++k) acc = fma(L[r * LD + k], R[k * LD + c], acc);
    epi(r, c, acc);
  }
}

__device__ __forceinline__ void load(double* S, const double* __restrict__ g, int m, int tid, int n) {
  for (int e = tid; e < m * m; e += n) S[(e / m) * LD + e % m] = g[e];
}

__global__ void __launch_bounds__(kThreads) k_small_factor(const PartDesc* __restrict__ parts,
                                                           const double* __restrict__ A, const double* __restrict__ B,
                                                           const double* __restrict__ C, double* __restrict__ G,
                                                           double* __restrict__ Acal, double* __restrict__ ZL,
                                                           double* __restrict__ ZR, int* __restrict__ status,
                                                           const int* __restrict__ band) {
  extern __shared__ __align__(16) double sm[];
  __shared__ Shared sh;
  double *D = sm, *Gs = sm + BLK, *X = sm + 2 * BLK, *Y = sm + 3 * BLK, *Z = sm + 4 * BLK, *As = sm + 5 * BLK,
         *Cs = sm + 6 * BLK;
  const PartDesc p = parts[blockIdx.x];
  const int m = p.m, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long mm = (long long)m * m;
  const int wb = band ? *band : kBandMax + 1;  // half-bandwidth of the level's A and C
  const bool banded = wb <= kBandMax;
  const bool hl = (p.flags & HAS_LEFT) != 0, hr = (p.flags & HAS_RIGHT) != 0;
  load(D, B + p.blk, m, tid, kThreads);
  if (hl) load(Y, A + p.blk, m, tid, kThreads);
  __syncthreads();
  for (int t = 0; t < p.L; ++t) {
    const long long o = p.blk + (long long)t * mm;
    const bool last = t == p.L - 1, gc = !last || hr;
    if (warp < kInvWarps) {
      bool bad = false;
      if (m <= 8) invert<2>(D, Gs, m, sh, warp, lane, bad);
      else if (m <= 16) invert<4>(D, Gs, m, sh, warp, lane, bad);
      else invert<8>(D, Gs, m, sh, warp, lane, bad);
      if (bad) atomicMin(status + p.sys, p.row0 + t + 1);
    } else {
      if (gc) load(Cs, C + o, m, tid - 32 * kInvWarps, kThreads - 32 * kInvWarps);
      if (!last) load(As, A + o + mm, m, tid - 32 * kInvWarps, kThreads - 32 * kInvWarps);
    }
    __syncthreads();
    for (int e = tid; e < m * m; e += kThreads) G[o + e] = Gs[(e / m) * LD + e % m];
    // Acal_t = G_t C_t (the right spike's seed in the last row), Bcal_t = G_t Y_t
    auto to_x = [&](int r, int c, double v) {
      X[r * LD + c] = v;
      (last ? ZR : Acal)[o + r * m + c] = v;
    };
    if (gc && banded) band_product<false>(Gs, Cs, m, wb, tid, to_x);
    else if (gc) product(Gs, Cs, m, tid, to_x);
    if (hl)
      product(Gs, Y, m, tid, [&](int r, int c, double v) {
        Z[r * LD + c] = v;
        ZL[o + r * m + c] = v;
      });
    __syncthreads();
    if (last) break;
    // D_{t+1} = B_{t+1} - A_{t+1} Acal_t, Y_{t+1} = -A_{t+1} Bcal_t
    auto to_d = [&](int r, int c, double v) { D[r * LD + c] = B[o + mm + r * m + c] - v; };
    auto to_y = [&](int r, int c, double v) { Y[r * LD + c] = -v; };
    if (banded) {
      band_product<true>(As, X, m, wb, tid, to_d);
      if (hl) band_product<true>(As, Z, m, wb, tid, to_y);
    } else {
      product(As, X, m, tid, to_d);
      if (hl) product(As, Z, m, tid, to_y);
    }
    __syncthreads();
  }
  // backward: ZL_t -= Acal_t ZL_{t+1}, ZR_t = -Acal_t ZR_{t+1}; ZL_{t+1} in Z
  // (then Y, in turn), ZR_{t+1} in X (then D)
  if (!hl && !hr) return;
  double *zl = Z, *zln = Y, *zr = X, *zrn = D;
  load(As, Acal + p.blk + max(0, p.L - 2) * mm, m, tid, kThreads);
  __syncthreads();
  for (int t = p.L - 2; t >= 0; --t) {
    const long long o = p.blk + (long long)t * mm;
    if (t > 0) load(Cs, Acal + o - mm, m, tid, kThreads);
    if (hl)
      product(As, zl, m, tid, [&](int r, int c, double v) {
        const double n = ZL[o + r * m + c] - v;
        zln[r * LD + c] = n;
        ZL[o + r * m + c] = n;
      });
    if (hr)
      product(As, zr, m, tid, [&](int r, int c, double v) {
        zrn[r * LD + c] = -v;
        ZR[o + r * m + c] = -v;
      });
    __syncthreads();
    double* x = zl; zl = zln; zln = x;
    x = zr; zr = zrn; zrn = x;
    x = As; As = Cs; Cs = x;
  }
}

}  // namespace small

void launch_small_factor(const PartDesc* parts, int nparts, const double* A, const double* B, const double* C, double* G,
                         double* Acal, double* ZL, double* ZR, int* status, const int* band, cudaStream_t st) {
  if (nparts <= 0) return;
  constexpr int smem = small::kBlocks * small::BLK * (int)sizeof(double);
  allow_smem(small::k_small_factor, smem);
  small::k_small_factor<<<nparts, small::kThreads, smem, st>>>(parts, A, B, C, G, Acal, ZL, ZR, status,
                                                                  band);
}

}  // namespace dm
