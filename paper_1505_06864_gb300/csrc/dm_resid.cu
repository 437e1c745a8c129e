// Residual r = b - T x with float64 accuracy on the bf16 tensor cores (an
// exact splitting in the manner of Ozaki's error-free matrix products).  Block
// row i of a system is L = [A_i B_i C_i] (m x 3m) times X = [x_{i-1}; x_i;
// x_{i+1}] (3m x r).  Every row of L gets a scale e (the exponent of the row's
// largest magnitude) and every column of X a scale f, every value seven
// balanced base-256 digits (dm_slices.cuh: rounded at 2^-56 of its scale), and
//   L X = 2^(e+f+2) sum_{d=2..9} 2^(-8d) acc_d,  acc_d = sum_{s+t=d} Ldigit_s Xdigit_t.
// Each acc_d sums at most seven products over K <= 128 (one of the three
// blocks) of magnitude <= 2^14: integers below 2^24, exact in float32; after
// each block they are added up in 64-bit integers.  Operand rounding and the
// dropped pairs bound the error of an entry by 3m 2^-55 times its scales 2^(e+f).
//
// A float64 dot product's bound is 3m 2^-53 sum |row| |column|, far below that
// where the row weights small entries of x only (unknowns of different scale, a
// solution that decays within three block rows).  So every entry is certified: one
// more product, of |L| and |x| rounded to bf16 (down, so from below), gives the
// sum, and an entry with less than 2^-6 of its scales is computed again by
// float64 multiply-adds, a warp per entry.  Dense and banded blocks with
// solutions of one scale have 2^-4.5 of them and more (none is recomputed: the
// magnitudes cost 60 us of a residual of N = 4096, m = 128, r = 8).  The error of
// an entry is then at most 3m 2^-49 sum |row| |column|.
//
// Bound by the digit extraction (about 40 instructions per entry of L, once
// per residual) beside reading L: so the digits stay in registers.  A warp
// takes 16 point rows of one block row; the mma.sync fragment of a 16 x 16
// tile is what each lane loads itself (16-byte loads, 64 bytes per row), no
// staging through shared memory and no barrier but for the digits of X, which
// the CTA prepares per block (a tenth of the work).  tcgen05 would need every
// digit of L in shared memory first: that version (one 169 KB CTA per SM, a
// barrier and a wait per 64 columns) read 4096 blocks of m = 128 with r = 8 in
// 2.9 ms, and the float64 pipe needs 3.2 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "dm_internal.cuh"
#include "dm_slices.cuh"

namespace dm {
namespace resid {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int S = kBalSlices;
constexpr int NACC = S + 1;  // d = 2 .. 9
constexpr int SX = S + 1;    // an entry of x in shared memory: its digits and its magnitude
constexpr float kCertified = 0x1p-6f;
constexpr int kMaxMRow = 128, kMaxCols = 16;
static_assert(kMaxMRow <= 16 * kWarps, "a block row's 16-row tiles in one CTA");

__device__ __forceinline__ uint32_t abs_hi(unsigned long long bits) { return (uint32_t)(bits >> 32) & 0x7fffffffu; }

// Largest high word (sign cleared) of every point row of [A_i B_i C_i] of the
// sliced systems: a warp per point row, one CTA per block row.
__global__ void __launch_bounds__(kThreads) k_row_scales(const SysDesc* __restrict__ sys, int nsys,
                                                         const double* __restrict__ A, const double* __restrict__ B,
                                                         const double* __restrict__ C, unsigned* __restrict__ rowhi) {
  const int si = find_sys(sys, nsys, blockIdx.x);
  const SysDesc sd = sys[si];
  if (!sd.sliced) return;
  const int i = blockIdx.x - sd.row0, m = sd.m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long o = sd.blk + (long long)i * m * m;
  const bool hasA = i > 0, hasC = i < sd.N - 1;
  const unsigned long long* a = reinterpret_cast<const unsigned long long*>(A + o);
  const unsigned long long* bb = reinterpret_cast<const unsigned long long*>(B + o);
  const unsigned long long* c = reinterpret_cast<const unsigned long long*>(C + o);
  for (int rr = warp; rr < m; rr += kWarps) {
    uint32_t mx = 0;
    for (int k = lane; k < m; k += 32) {
      const long long e = (long long)rr * m + k;
      mx = max(mx, abs_hi(__ldg(bb + e)));
      if (hasA) mx = max(mx, abs_hi(__ldg(a + e)));
      if (hasC) mx = max(mx, abs_hi(__ldg(c + e)));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) rowhi[sd.eoff + (long long)i * m + rr] = mx;
  }
}

// Largest high word of every column of every block x_i of the sliced systems
// ([global block row][16]): a warp per block row, lane = column + 16 * parity
// of the point row.
__global__ void __launch_bounds__(kThreads) k_col_scales(const SysDesc* __restrict__ sys, int nsys, int nrows,
                                                         const double* __restrict__ x, unsigned* __restrict__ colhi) {
  const int row = blockIdx.x * kWarps + (threadIdx.x >> 5);
  if (row >= nrows) return;
  const int lane = threadIdx.x & 31;
  const SysDesc sd = sys[find_sys(sys, nsys, row)];
  if (!sd.sliced) return;
  const int i = row - sd.row0, m = sd.m, r = sd.r;
  const int c = lane & 15, par = lane >> 4;
  const unsigned long long* xi = reinterpret_cast<const unsigned long long*>(x + sd.vec + (long long)i * m * r);
  uint32_t mx = 0;
  if (c < r)
#pragma unroll 4
    for (int k = par; k < m; k += 2) mx = max(mx, abs_hi(__ldg(xi + (long long)k * r + c)));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  if (lane < 16) colhi[(long long)row * kMaxCols + c] = mx;
}

__device__ __forceinline__ void mma_k16(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// The lane's eight entries of a 16 x 16 tile of L, in fragment order: rows r0
// and r0 + 8, columns k, k + 1 and k + 8, k + 9 (zero past m).
template <bool V2>
__device__ __forceinline__ void load_tile(const double* __restrict__ L, int m, int r0, int k,
                                          unsigned long long (&v)[8]) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int row = r0 + 8 * (h & 1), kk = k + 8 * (h >> 1);
    const double* p = L + (long long)row * m + kk;
    v[2 * h] = v[2 * h + 1] = 0ull;
    if (V2) {  // m even: both columns inside or both outside
      if (row < m && kk < m) {
        const ulonglong2 q = __ldg(reinterpret_cast<const ulonglong2*>(p));
        v[2 * h] = q.x;
        v[2 * h + 1] = q.y;
      }
    } else {
      if (row < m && kk < m) v[2 * h] = __ldg(reinterpret_cast<const unsigned long long*>(p));
      if (row < m && kk + 1 < m) v[2 * h + 1] = __ldg(reinterpret_cast<const unsigned long long*>(p + 1));
    }
  }
}

// |v| 2^-e, |v| < 2^e, as bf16 rounded down (in the high half of the word); for
// e below -896 less than that.
__device__ __forceinline__ uint32_t magnitude(unsigned long long bits, int e) {
  const int h = (int)(bits >> 32) & 0x7fffffff;
  return (uint32_t)max((h >> 13) - ((max(e, -896) + 896) << 7), 0) << 16;
}

// acc += the 16 rows of L (one block, m columns) times the digits xd of x, sum
// += the product of the magnitudes.
template <int NT, bool V2>
__device__ __forceinline__ void tile_products(const double* __restrict__ L, int m, int r0, int tg, const int (&er)[2],
                                              const uint2* xd, int lane, float (&acc)[NACC][NT][4],
                                              float (&sum)[NT][4]) {
  const int nks = (m + 15) / 16;
  unsigned long long v[8];
  load_tile<V2>(L, m, r0, 2 * tg, v);
#pragma unroll 1
  for (int ks = 0; ks < nks; ++ks) {
    uint32_t a[S][4], am[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      am[h] = pack_hi(magnitude(v[2 * h], er[h & 1]), magnitude(v[2 * h + 1], er[h & 1]));
      uint32_t d0[S], d1[S];
      digits<S>(v[2 * h], er[h & 1], d0);
      digits<S>(v[2 * h + 1], er[h & 1], d1);
#pragma unroll
      for (int s = 0; s < S; ++s) a[s][h] = pack_hi(d0[s], d1[s]);
    }
    if (ks + 1 < nks) load_tile<V2>(L, m, r0, 16 * (ks + 1) + 2 * tg, v);  // in flight beside the products
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      uint2 b[S];
      mma_k16(sum[nt], am, xd[((ks * SX + S) * NT + nt) * 32 + lane]);
#pragma unroll
      for (int t = 0; t < S; ++t) b[t] = xd[((ks * SX + t) * NT + nt) * 32 + lane];
#pragma unroll
      for (int s = 1; s <= S; ++s)
#pragma unroll
        for (int t = 1; t <= S; ++t)
          if (s + t <= S + 2) mma_k16(acc[s + t - 2][nt], a[s - 1], b[t - 1]);
    }
  }
}

// sum_k L[k] x[k r] over the m entries of one point row of a block (lanes
// together; this lane's part).
__device__ __forceinline__ double row_part(const double* __restrict__ L, const double* __restrict__ x, int m, int r,
                                           int lane) {
  double acc = 0.0;
#pragma unroll 4
  for (int k = lane; k < m; k += 32) acc = fma(__ldg(L + k), __ldg(x + (long long)k * r), acc);
  return acc;
}

// One entry of L X in float64 by a warp: o the row in A, B, C, xi its column in
// x_i (mr entries from one x_i to the next).
__device__ __noinline__ double float64_entry(const double* __restrict__ A, const double* __restrict__ B,
                                             const double* __restrict__ C, long long o, const double* __restrict__ xi,
                                             long long mr, int m, int r, bool hasA, bool hasC, int lane) {
  double acc = row_part(B + o, xi, m, r, lane);
  if (hasA) acc += row_part(A + o, xi - mr, m, r, lane);
  if (hasC) acc += row_part(C + o, xi + mr, m, r, lane);
#pragma unroll
  for (int w = 16; w; w >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, w);
  return acc;
}

// One CTA per group of block rows of a sliced system with 8 (NT - 1) < r <= 8
// NT: a warp per 16 point rows.
template <int NT>
__global__ void __launch_bounds__(kThreads, NT == 1 ? 2 : 1)
    k_residual_digits(const SysDesc* __restrict__ sys, int nsys, const double* __restrict__ A,
                      const double* __restrict__ B, const double* __restrict__ C, const double* __restrict__ x,
                      const double* __restrict__ b, double* __restrict__ rout, double* __restrict__ nrm,
                      const unsigned* __restrict__ rowhi, const unsigned* __restrict__ colhi) {
  extern __shared__ __align__(16) uint2 xd[];  // [block row of the group][k16 step][digit, magnitude][NT][lane]
  __shared__ double red[2 * kMaxCols];
  __shared__ int fcol[kWarps][kMaxCols];
  int lo = 0, hi = nsys - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sys[mid].cta0[NT - 1] <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const SysDesc sd = sys[lo];
  const int m = sd.m, r = sd.r, mt = (m + 15) / 16, nb = kWarps / mt;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tg = lane & 3;
  const int i0 = (blockIdx.x - sd.cta0[NT - 1]) * nb, rows = min(nb, sd.N - i0);  // the group's block rows
  const int sub = warp / mt, i = i0 + sub, r0 = 16 * (warp - sub * mt) + g;
  const bool active = sub < rows;
  const long long mm = (long long)m * m, mr = (long long)m * r;
  const int xw = mt * SX * NT * 32;  // words of one block row's digits
  if (tid < 2 * kMaxCols) red[tid] = 0.0;
  if (tid < kMaxCols * rows) {
    const int q = tid / kMaxCols, c = tid - q * kMaxCols, ii = i0 + q;
    const long long row = (long long)(sd.row0 + ii) * kMaxCols + c;
    uint32_t h = colhi[row];
    if (ii > 0) h = max(h, colhi[row - kMaxCols]);
    if (ii < sd.N - 1) h = max(h, colhi[row + kMaxCols]);
    fcol[q][c] = scale_exponent(h);
  }
  int er[2] = {0, 0};
  if (active) {
    const unsigned* eh = rowhi + sd.eoff + (long long)i * m;
    if (r0 < m) er[0] = scale_exponent(eh[r0]);
    if (r0 + 8 < m) er[1] = scale_exponent(eh[r0 + 8]);
  }
  const long long o = sd.blk + (long long)(active ? i : 0) * mm;
  const bool v2 = (m & 1) == 0 && (((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) |
                                     reinterpret_cast<uintptr_t>(C)) & 15) | (sd.blk & 1)) == 0;
  long long T[NT][4];  // (L X) 2^(54 - e - f)
  float sum[NT][4];  // sum |L| |X| 2^(-e - f), from below
  uint32_t nan = 0;
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int q = 0; q < 4; ++q) T[nt][q] = 0, sum[nt][q] = 0.f;
#pragma unroll 1
  for (int part = 0; part < 3; ++part) {  // A_i x_{i-1}, B_i x_i, C_i x_{i+1}
    __syncthreads();
    // the digits of x_{i - 1 + part}, in the order of the fragments
    for (int e = tid; e < rows * mt * NT * 32; e += kThreads) {
      const int ln = e & 31, q1 = e >> 5, nt = q1 % NT, q2 = q1 / NT, ks = q2 % mt, q = q2 / mt;
      const int ii = i0 + q - 1 + part, c = 8 * nt + (ln >> 2), k = 16 * ks + 2 * (ln & 3);
      const double* xp = x + sd.vec + (long long)ii * mr + c;
      const bool in = ii >= 0 && ii < sd.N && c < r;
      uint32_t d[4][S], mg[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int kk = k + (u & 1) + 8 * (u >> 1);
        const double val = in && kk < m ? xp[(long long)kk * r] : 0.0;
        digits<S>((unsigned long long)__double_as_longlong(val), fcol[q][c], d[u]);
        mg[u] = magnitude((unsigned long long)__double_as_longlong(val), fcol[q][c]);
      }
#pragma unroll
      for (int t = 0; t < S; ++t)
        xd[q * xw + ((ks * SX + t) * NT + nt) * 32 + ln] = make_uint2(pack_hi(d[0][t], d[1][t]), pack_hi(d[2][t], d[3][t]));
      xd[q * xw + ((ks * SX + S) * NT + nt) * 32 + ln] = make_uint2(pack_hi(mg[0], mg[1]), pack_hi(mg[2], mg[3]));
    }
    __syncthreads();
    if (!active || (part == 0 && i == 0) || (part == 2 && i == sd.N - 1)) continue;
    const double* L = (part == 0 ? A : part == 1 ? B : C) + o;
    float acc[NACC][NT][4];
#pragma unroll
    for (int d = 0; d < NACC; ++d)
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[d][nt][q] = 0.f;
    if (v2)
      tile_products<NT, true>(L, m, r0, tg, er, xd + sub * xw, lane, acc, sum);
    else
      tile_products<NT, false>(L, m, r0, tg, er, xd + sub * xw, lane, acc, sum);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        int a[NACC];
#pragma unroll
        for (int d = 0; d < NACC; ++d) a[d] = __float2int_rn(acc[d][nt][q]);
        if (acc[0][nt][q] != acc[0][nt][q]) nan |= 1u << (4 * nt + q);  // a NaN or an infinity
        const long long h = (long long)a[0] * 65536 + (a[1] * 256 + a[2]);
        const long long l = (((long long)a[3] * 256 + a[4]) * 256 + a[5]) * 65536 + ((long long)a[6] * 256 + a[7]);
        T[nt][q] += h * (1 << 24) + ((l + 32768) >> 16);  // three times below 2^61.1
      }
  }
  if (active) {
    const double* bi = b + sd.vec + (long long)i * mr;
    double* ri = rout + sd.vec + (long long)i * mr;
    double val[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = r0 + 8 * (q >> 1), c = 8 * nt + 2 * tg + (q & 1);
        const int s = er[q >> 1] + fcol[sub][c] - 54;
        bool odd = false;
        double v = round_scaled(T[nt][q], s, odd);
        if (odd) v = ldexp((double)T[nt][q], s);
        if ((nan >> (4 * nt + q)) & 1u) v = __longlong_as_double(0x7ff8000000000000ll);
        // a sum of 0: no term above 2^-126 of the scales
        uint32_t left = __ballot_sync(0xffffffffu, row < m && c < r && sum[nt][q] != 0.f && !(sum[nt][q] >= kCertified));
        while (left) {
          const int src = __ffs(left) - 1;
          left &= left - 1;
          const int lrow = r0 - g + (src >> 2) + 8 * (q >> 1), lc = 8 * nt + 2 * (src & 3) + (q & 1);
          const double w = float64_entry(A, B, C, o + (long long)lrow * m, x + sd.vec + (long long)i * mr + lc, mr, m, r,
                                         i > 0, i < sd.N - 1, lane);
          if (lane == src) v = w;
        }
        val[nt][q] = v;
      }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int cc = 0; cc < 2; ++cc) {
        const int c = 8 * nt + 2 * tg + cc;
        double sr = 0.0, sb = 0.0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = r0 + 8 * h, q = 2 * h + cc;
          if (row < m && c < r) {
            const long long e = (long long)row * r + c;
            const double bb = bi[e], rv = bb - val[nt][q];
            ri[e] = rv;
            sr = fma(rv, rv, sr);
            sb = fma(bb, bb, sb);
          }
        }
#pragma unroll
        for (int w = 4; w < 32; w <<= 1) {
          sr += __shfl_xor_sync(0xffffffffu, sr, w);
          sb += __shfl_xor_sync(0xffffffffu, sb, w);
        }
        if (g == 0 && c < r) {
          atomicAdd(&red[c], sr);
          atomicAdd(&red[kMaxCols + c], sb);
        }
      }
  }
  __syncthreads();
  if (tid < r) {
    atomicAdd(&nrm[(long long)lo * 4 * kMaxR + tid], red[tid]);
    atomicAdd(&nrm[(long long)lo * 4 * kMaxR + kMaxR + tid], red[kMaxCols + tid]);
  }
}

}  // namespace resid

bool residual_sliced_fits(int m, int r) {
  return m >= 1 && m <= resid::kMaxMRow && r >= 1 && r <= resid::kMaxCols;
}

int residual_sliced_class(int r) { return (r - 1) / 8; }

int residual_sliced_ctas(int N, int m) {
  const int nb = resid::kWarps / ((m + 15) / 16);
  return (N + nb - 1) / nb;
}

void launch_row_scales(const SysDesc* sys, int nsys, int nrows, const double* A, const double* B,
                       const double* C, unsigned* rowhi, cudaStream_t st) {
  if (nsys <= 0 || nrows <= 0) return;
  resid::k_row_scales<<<nrows, resid::kThreads, 0, st>>>(sys, nsys, A, B, C, rowhi);
}

void launch_col_scales(const SysDesc* sys, int nsys, int nrows, const double* x, unsigned* colhi, cudaStream_t st) {
  if (nsys <= 0 || nrows <= 0) return;
  resid::k_col_scales<<<(nrows + resid::kWarps - 1) / resid::kWarps, resid::kThreads, 0, st>>>(sys, nsys, nrows, x,
                                                                                              colhi);
}

void launch_residual_sliced(const SysDesc* sys, int nsys, const int (&ctas)[2], const double* A, const double* B,
                            const double* C, const double* x, const double* b, double* r, double* nrm,
                            const unsigned* rowhi, const unsigned* colhi, cudaStream_t st) {
  // the group's block rows have at most 16 kWarps = 128 point rows together
  constexpr int smem1 = resid::kWarps * resid::SX * 32 * (int)sizeof(uint2);
  if (ctas[0] > 0)
    resid::k_residual_digits<1><<<ctas[0], resid::kThreads, smem1, st>>>(sys, nsys, A, B, C, x, b, r, nrm, rowhi, colhi);
  if (ctas[1] > 0)
    resid::k_residual_digits<2><<<ctas[1], resid::kThreads, 2 * smem1, st>>>(sys, nsys, A, B, C, x, b, r, nrm, rowhi,
                                                                             colhi);
}

}  // namespace dm
