// Float64 block inverse G_t = D_t^{-1} of the digit-sliced levels: blocked
// Gauss-Jordan with partial pivoting (the paper's inversion, Section 4;
// Gauss-Jordan as in the library's other inverses), panels of 32 columns, the
// rank-32 trailing updates as digit-sliced tensor-core products (dm_oz.cu,
// k_oz_step<3>).
//
// The pivoting is implicit: rows stay where they are, and the pivot of column
// k is the row p_k of largest magnitude in column k among the rows that were
// no pivot before.  For a panel K = [k0, k0 + 32) with pivot rows p_K:
//   1. k_gj_panel: in-place Gauss-Jordan restricted to the panel's columns
//      (row p_k scaled by 1/M[p_k][k] with 1/M[p_k][k] in column k, every
//      other row i minus M[i][k] times row p_k with -M[i][k]/M[p_k][k] in
//      column k); the panel then holds U = [W in the rows p_K; -M_RK W
//      elsewhere] (W = M[p_K, K]^{-1}).  It also writes U's row slices and the
//      column slices of V = M[p_K, J], J the columns outside K.
//   2. k_oz_step<3>: M[:, J] = (M[:, J], rows p_K zeroed) + U V.
// After the last panel the working matrix W satisfies D^{-1}[k][p_j] =
// W[p_k][j]; k_gj_finish moves the entries there and writes the row slices of
// the inverse.  The working matrix is a buffer per subsystem (rolling), so it
// stays in L2 from step to step.  It holds D_t equilibrated, 2^-rho D 2^-gam with
// the level's exponents per equation and unknown (dm_oz.cu), so that its digits
// and its pivots see entries of one scale; k_gj_finish takes the exponents back.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "dm_internal.cuh"
#include "dm_recip.cuh"
#include "dm_slices.cuh"

namespace dm {
namespace gj {

constexpr int S = kBalSlices;           // digit slices of U and V (K = 32)
constexpr int PW = 32;                 // panel width
constexpr int SW = 8;                  // subpanel width
constexpr int PS = PW + 1;             // row stride of the panel in shared memory (float64)
constexpr int kMaxChain = 8;           // most warps that run the pivot chain
constexpr int kHelpers = 8;            // more warps for the rank-8 updates, beside the chain's

__global__ void __launch_bounds__(256) k_gj_copy_b0(const PartDesc* __restrict__ parts, int m,
                                                    const double* __restrict__ B, double* __restrict__ W,
                                                    const int* __restrict__ gam, const int* __restrict__ rho) {
  const PartDesc p = parts[blockIdx.x];
  const long long mm = (long long)m * m;
  double* w = W + (long long)blockIdx.x * mm;
  const double* b = B + p.blk;
  const int *gb = gam + p.blk / m, *rb = rho + p.blk / m;
  for (long long e = threadIdx.x + (long long)blockIdx.y * blockDim.x; e < mm; e += (long long)blockDim.x * gridDim.y)
    w[e] = scale_pow2(b[e], -(rb[e / m] + gb[e % m]));
}

// What the chain's warps exchange per pivot (double-buffered by its parity).
struct __align__(16) GjCand {  // a warp's best row for the next pivot
  double v;       // its element of the pivot column
  uint32_t key;   // 0: no eligible row; else the high word of |v| + 1
  int idx;        // the row
};
struct __align__(16) GjPivot {  // the pivot
  double inv;  // its reciprocal (0 when unusable)
  int idx;     // its row
  int warp;    // the warp that holds it
};
struct GjShared {
  GjCand cand[2][kMaxChain];
  GjPivot piv[2];
  double row[2][kMaxChain][SW];  // every candidate row after the pending pivot's update
};

// The pivot chain of one subpanel (columns c0 .. c0 + w - 1 of the panel), run
// by warps 0 .. nw - 1: lane `lane` of warp `warp` holds rows 32 warp + lane +
// 32 CW i, i < RPL, eight columns each, in registers.
//
// A float64 instruction holds its warp for 64 cycles on GB300 (measured; one
// warp per SM sub-partition, dependent or not), and other instructions of the
// same warp do not overlap it.  So the chain's warps do the multiply-adds (9
// RPL float64 instructions per pivot) and the search among their own rows, and a control warp
// picks the pivot among the warps' candidates and takes its reciprocal in
// integer arithmetic while they run.  Per pivot: every row updates its next
// pivot column first and the warps publish their best candidates (largest
// high word of |value|: candidates that agree to 2^-20 count as equal, the
// first one is taken); then they update the other seven columns and publish
// the candidate rows; after one barrier with the control warp every row takes
// its multiplier.  The pivot's own row takes part as zeros plus the
// reciprocal times itself, so that no result is selected after a
// multiply-add.
//
// The registers rotate by one column per pivot (register c of `a` holds
// column (j - 1 + c) mod 8 before pivot j, of `b` column (j + c) mod 8 after
// it), from one set to the other: rotated in place, every multiply-add would
// wait until the one before has read its operands.
template <int RPL>
struct GjRows {
  double a[RPL][SW], fn[RPL];  // fn: minus the multiplier of the pending pivot
  bool dead[RPL];              // past the block's end, or a pivot row already
};

template <int CW, int RPL>
__device__ __forceinline__ void gj_pivot(const GjRows<RPL>& in, GjRows<RPL>& out, double (&s)[SW], int buf, int nw,
                                         GjShared& sh, int warp, int lane) {
  uint32_t key = 0;
  double bnv = 0.0;
  int bi = 0;
#pragma unroll
  for (int i = 0; i < RPL; ++i) out.a[i][0] = fma(in.fn[i], s[1], in.a[i][1]);
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const uint32_t ki = in.dead[i] ? 0u : abs_hi(out.a[i][0]) + 1u;
    if (i == 0 || ki > key) key = ki, bnv = out.a[i][0], bi = i;
  }
  const uint32_t wkey = __reduce_max_sync(0xffffffffu, key);
  const int src = (int)__reduce_min_sync(0xffffffffu, key == wkey ? (uint32_t)lane : 32u);
  if (lane == src) {
    GjCand& cd = sh.cand[buf][warp];
    cd.v = bnv;
    cd.key = wkey;
    cd.idx = 32 * warp + lane + 32 * CW * bi;
  }
  asm volatile("bar.arrive 1, %0;" ::"r"(32 * nw + 32) : "memory");
  // src < 32: adds nothing, but keeps the multiply-adds below after the search
  const int z = src & 64;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const double f = __hiloint2double(__double2hiint(in.fn[i]) + z, __double2loint(in.fn[i]));
#pragma unroll
    for (int c = 2; c < SW; ++c) out.a[i][c - 1] = fma(f, s[c], in.a[i][c]);
    out.a[i][SW - 1] = fma(f, s[0], in.a[i][0]);
  }
  if (lane == src) {
#pragma unroll
    for (int i = 0; i < RPL; ++i)
      if (bi == i) {
#pragma unroll
        for (int c = 0; c < SW; c += 2)
          *reinterpret_cast<double2*>(&sh.row[buf][warp][c]) = make_double2(out.a[i][c], out.a[i][c + 1]);
      }
  }
  asm volatile("bar.sync 2, %0;" ::"r"(32 * nw + 32) : "memory");
  const GjPivot pv = sh.piv[buf];
  const double* u = sh.row[buf][pv.warp];
#pragma unroll
  for (int c = 0; c < SW; c += 2) {
    const double2 u2 = *reinterpret_cast<const double2*>(u + c);
    s[c] = u2.x;
    s[c + 1] = u2.y;
  }
  s[0] = 1.0;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    out.fn[i] = -out.a[i][0] * pv.inv;
    out.a[i][0] = 0.0;
    out.dead[i] = in.dead[i];
    if (32 * warp + lane + 32 * CW * i == pv.idx) {
      out.dead[i] = true;
      out.fn[i] = pv.inv;
#pragma unroll
      for (int c = 1; c < SW; ++c) out.a[i][c] = 0.0;
    }
  }
}

template <int CW, int RPL>
__device__ __forceinline__ void gj_chain(double* P, int m, int c0, int w, int nw, const uint32_t* used, GjShared& sh,
                                         int warp, int lane) {
  GjRows<RPL> x, y;
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int row = 32 * warp + lane + 32 * CW * i;
    x.dead[i] = row >= m || ((used[row >> 5] >> (row & 31)) & 1u) != 0;
    x.fn[i] = 0.0;
#pragma unroll
    for (int c = 0; c < SW; ++c) x.a[i][c] = row < m ? P[row * PS + c0 + ((c + 7) & 7)] : 0.0;
  }
  double s[SW];  // the pending pivot's row (1 in its own column)
#pragma unroll
  for (int c = 0; c < SW; ++c) s[c] = 0.0;
#pragma unroll 1
  for (int j = 0; j < w; j += 2) {
    gj_pivot<CW, RPL>(x, y, s, 0, nw, sh, warp, lane);
    if (j + 1 < w)
      gj_pivot<CW, RPL>(y, x, s, 1, nw, sh, warp, lane);
    else
      x = y;
  }
  // the last pivot's update
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int row = 32 * warp + lane + 32 * CW * i;
#pragma unroll
    for (int c = 0; c < SW; ++c) y.a[i][c] = fma(x.fn[i], s[c], x.a[i][c]);
    if (row < m)
#pragma unroll
      for (int c = 0; c < SW; ++c) P[row * PS + c0 + ((w - 1 + c) & 7)] = y.a[i][c];
  }
}

// The control warp's side of gj_chain.  Before the last pivot some row is
// eligible, and an eligible row's key is at least 1, so a pivot is always
// found; were none (key 0), it would count as singular, and the row stays
// inside the block whatever a warp published.
__device__ __forceinline__ void gj_control(int m, int c0, int w, int nw, GjShared& sh, int* piv_s, int lane, bool& bad) {
#pragma unroll 1
  for (int j = 0; j < w; ++j) {
    asm volatile("bar.sync 1, %0;" ::"r"(32 * nw + 32) : "memory");
    const GjCand c = sh.cand[j & 1][min(lane, nw - 1)];
    const uint32_t kmax = __reduce_max_sync(0xffffffffu, c.key);
    const int best = (int)__reduce_min_sync(0xffffffffu, c.key == kmax ? (uint32_t)lane : 32u);
    const double inv = kmax == 0 || pivot_unusable(c.v) ? 0.0 : pivot_recip(c.v);
    if (lane == best) {
      const int row = min(c.idx, m - 1);
      sh.piv[j & 1] = GjPivot{inv, row, best};
      piv_s[c0 + j] = row;
      if (__double_as_longlong(inv) == 0) bad = true;
    }
    asm volatile("bar.sync 2, %0;" ::"r"(32 * nw + 32) : "memory");
  }
}

// c += the product of two digit pairs (K = 16) or of one (K = 8): no side
// effects, so the compiler may order the products of independent sums.
__device__ __forceinline__ void mma_k16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_k8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

constexpr int kNotFinite = 1 << 14;  // scale of a row or column with a NaN or an infinity

__device__ __forceinline__ int bal_exponent(uint32_t hmax) {
  return hmax >= 0x7ff00000u ? kNotFinite : scale_exponent(hmax);
}

// The digits of a subpanel's pivot rows V (seven bf16 per value: [digit][column][row]) and
// their columns' scales; the digits of its columns U by 16-row tile, in the
// order in which gj_rank8's lanes hold them (two words more: a row's scale and
// whether it is a pivot row).
struct GjDigits {
  uint32_t v[kBalSlices][PW][SW / 2];
  int vexp[PW];
  uint32_t pivots[kMaxM / 32];  // the subpanel's pivot rows
};
constexpr int kTileWords = 2 * kBalSlices + 2;

// The digits of V = the rows piv[0 .. w - 1] of the panel; threads 0 .. 255, a value each.
__device__ __forceinline__ void gj_digits_v(const double* P, const int* piv, int w, GjDigits& dg, int tid) {
  const int c = tid >> 3, j = tid & 7;
  const double v = j < w ? P[piv[min(j, w - 1)] * PS + c] : 0.0;
  uint32_t h = abs_hi(v);
  h = max(h, __shfl_xor_sync(0xffffffffu, h, 1));
  h = max(h, __shfl_xor_sync(0xffffffffu, h, 2));
  h = max(h, __shfl_xor_sync(0xffffffffu, h, 4));
  const int e = bal_exponent(h);
  uint32_t d[kBalSlices];
  digits<7>((unsigned long long)__double_as_longlong(v), e, d);
  unsigned short* dst = reinterpret_cast<unsigned short*>(dg.v);
#pragma unroll
  for (int k = 0; k < kBalSlices; ++k) dst[(k * PW + c) * SW + j] = (unsigned short)(d[k] >> 16);
  if (j == 0) dg.vexp[c] = e;
}

// Rank-8 update of nq of the panel's 8-column groups (from column n0 on, wrapping) after
// a subpanel's pivots: P[i][c] = (i a pivot row of the subpanel ? 0 : P[i][c])
// + sum_j U[i][j] V[j][c], U the subpanel's columns, V its pivot rows before
// the update; warp wi of nwk takes a run of the 16 x 8 tiles, row tile by row tile.
// In float64 instructions it would cost twice the pivot chain itself, so it
// runs on the tensor cores: seven balanced base-256 digits per operand (row
// scales for U, column scales for V), the 28 digit products with s + t <= 8
// in 16 mma.sync per 16 x 8 tile (two digit pairs share a K = 16
// instruction), sums below 8 * 7 * 2^14 < 2^22, exact on top of the float
// 1.5 2^23 they start from, whose bits then hold the integer; one integer rounding
// and one float64 add per entry.  (tcgen05 has no use here: K = 8 and the
// operands are in registers.)  A tile is a chain of dependent integer
// instructions (3500 cycles when every warp made its digits of U and V
// itself), so V's digits come from gj_digits_v, and U's are kept for the
// helpers (keep: written to Ud; else read from there when `kept`).
__device__ __noinline__ void gj_rank8(double* P, uint32_t* Ud, const GjDigits& dg, int mt, int c0, int n0, int nq,
                                      bool keep, bool kept, int wi, int nwk) {
  const int lane = threadIdx.x & 31, g = lane >> 2, tg = lane & 3;
  const int per = (mt * nq + nwk - 1) / nwk, i1 = min(mt * nq, (wi + 1) * per);
  uint32_t a[2][kBalSlices];
  int re[2];
  bool z[2];
  int rb = -1;
#pragma unroll 1
  for (int i = wi * per; i < i1; ++i) {
    __syncwarp();  // mma.sync below takes whole warps
    const int rt = nq == 1 ? i : i / nq, nc = (n0 + SW * (i - rt * nq)) & (PW - 1);
    uint32_t* ud = Ud + rt * (kTileWords * 32) + lane;
    if (rt != rb) {
      rb = rt;
      if (kept) {
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
#pragma unroll
          for (int k = 0; k < kBalSlices; ++k) a[h2][k] = ud[32 * (h2 * kBalSlices + k)];
          const int x = (int)ud[32 * (2 * kBalSlices + h2)];
          re[h2] = x >> 1;
          z[h2] = (x & 1) != 0;
        }
      } else {
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const int row = 16 * rt + 8 * h2 + g;
          const double v0 = P[row * PS + c0 + 2 * tg], v1 = P[row * PS + c0 + 2 * tg + 1];
          uint32_t h = max(abs_hi(v0), abs_hi(v1));
          h = max(h, __shfl_xor_sync(0xffffffffu, h, 1));
          h = max(h, __shfl_xor_sync(0xffffffffu, h, 2));
          re[h2] = bal_exponent(h);
          uint32_t d0[kBalSlices], d1[kBalSlices];
          digits<7>((unsigned long long)__double_as_longlong(v0), re[h2], d0);
          digits<7>((unsigned long long)__double_as_longlong(v1), re[h2], d1);
#pragma unroll
          for (int k = 0; k < kBalSlices; ++k) a[h2][k] = pack_hi(d0[k], d1[k]);
          z[h2] = ((dg.pivots[row >> 5] >> (row & 31)) & 1u) != 0;
          if (keep) {
#pragma unroll
            for (int k = 0; k < kBalSlices; ++k) ud[32 * (h2 * kBalSlices + k)] = a[h2][k];
            ud[32 * (2 * kBalSlices + h2)] = (uint32_t)(re[h2] * 2 + (z[h2] ? 1 : 0));
          }
        }
      }
    }
    uint32_t b[kBalSlices];
#pragma unroll
    for (int k = 0; k < kBalSlices; ++k) b[k] = dg.v[k][nc + g][tg];
    const int fe[2] = {dg.vexp[nc + 2 * tg], dg.vexp[nc + 2 * tg + 1]};
    float c[kBalSlices][4];  // acc_d + 1.5 2^23, d = 2 .. 8
#pragma unroll
    for (int k = 0; k < kBalSlices; ++k)
#pragma unroll
      for (int o = 0; o < 4; ++o) c[k][o] = 12582912.0f;
#pragma unroll
    for (int s = 1; s <= kBalSlices; s += 2)
#pragma unroll
      for (int d = s + 1; d <= 8; ++d) {
        if (s + 1 <= d - 1)
          mma_k16(c[d - 2], a[0][s - 1], a[1][s - 1], a[0][s], a[1][s], b[d - s - 1], b[d - s - 2]);
        else
          mma_k8(c[d - 2], a[0][s - 1], a[1][s - 1], b[d - s - 1]);
      }
    // units 2^(e_r + f_c + 2 - 60): the last accumulator's low four bits are
    // dropped; kBias is what the start leaves in 256 x + y
    constexpr uint32_t kBias1 = 0x4B400000u, kBias = kBias1 * 257u;
    auto total = [&](const uint32_t (&t)[kBalSlices]) {
      return (long long)(int)(t[0] * 256u + t[1] - kBias) * (1ll << 36) +
             (long long)(int)(t[2] * 256u + t[3] - kBias) * (1ll << 20) +
             (long long)(int)(t[4] * 256u + t[5] - kBias) * 16 + ((int)(t[6] - kBias1) >> 4);
    };
    double v[4];
    bool odd = re[0] == kNotFinite || re[1] == kNotFinite || fe[0] == kNotFinite || fe[1] == kNotFinite;
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      uint32_t t[kBalSlices];
#pragma unroll
      for (int k = 0; k < kBalSlices; ++k) t[k] = __float_as_uint(c[k][o]);
      v[o] = round_scaled(total(t), re[o >> 1] + fe[o & 1] - 58, odd);
    }
    if (odd) {  // results outside the normal range, NaN and infinite operands
#pragma unroll 1
      for (int o = 0; o < 4; ++o) {
        uint32_t t[kBalSlices];
#pragma unroll
        for (int k = 0; k < kBalSlices; ++k)
          t[k] = __float_as_uint(o == 0 ? c[k][0] : o == 1 ? c[k][1] : o == 2 ? c[k][2] : c[k][3]);
        const int er = o < 2 ? re[0] : re[1], ec = (o & 1) ? fe[1] : fe[0];
        const double x = er == kNotFinite || ec == kNotFinite ? __longlong_as_double(0x7ff8000000000000ll)
                                                              : ldexp((double)total(t), er + ec - 58);
        if (o == 0) v[0] = x;
        if (o == 1) v[1] = x;
        if (o == 2) v[2] = x;
        if (o == 3) v[3] = x;
      }
    }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      double* d = P + (16 * rt + 8 * (o >> 1) + g) * PS + nc + 2 * tg + (o & 1);
      *d = (z[o >> 1] ? 0.0 : *d) + v[o];
    }
  }
}

// Shared memory of k_gj_panel for mt 16-row tiles.
constexpr size_t smem_bytes(int mt) { return (size_t)mt * (16 * PS * sizeof(double) + kTileWords * 32 * sizeof(uint32_t)); }

// Eight values' digits to a slice array: slice sl at dst + sl * stride.
__device__ __noinline__ void gj_slice8(double v0, double v1, double v2, double v3, double v4, double v5, double v6, double v7,
                                       int e, __nv_bfloat16* dst, int stride) {
  const double v[8] = {v0, v1, v2, v3, v4, v5, v6, v7};
  uint32_t d[8][S];
#pragma unroll
  for (int c = 0; c < 8; ++c) digits<S>((unsigned long long)__double_as_longlong(v[c]), e, d[c]);
#pragma unroll
  for (int sl = 0; sl < S; ++sl)
    *reinterpret_cast<uint4*>(dst + (long long)sl * stride) =
        make_uint4(pack_hi(d[0][sl], d[1][sl]), pack_hi(d[2][sl], d[3][sl]), pack_hi(d[4][sl], d[5][sl]),
                   pack_hi(d[6][sl], d[7][sl]));
}

// One panel of every active subsystem's working matrix, a CTA per block: up to
// eight chain warps (a row per lane; two rows above m = 256), the control
// warp, and eight helpers.  Bound by the chain's float64 instructions and
// barriers: about 1150 cycles per pivot at m = 64, 1290 at 128 (one warp per SM
// sub-partition) and 1880 at m = 256 (two), half of the kernel's time; the updates that the
// chain waits for take a sixth, the slices at the end an eighth.  A cluster of CTAs with the rows
// split and a cluster barrier per pivot took 83 / 90 / 98 us per panel at m =
// 64 / 128 / 256, this one with every warp making its own digits of U and V 40 / 48 / 74 us, and
// 37 / 43 / 63 us (115 to 102 at m = 400) with the digits shared (34, 97, 64 blocks).  The loops
// stay rolled: the code runs once per launch, and unrolled it waited for its
// instructions.
template <int CW, int RPL>
__global__ void __launch_bounds__(32 * (CW + kHelpers + 1), 1)
    k_gj_panel(const PartDesc* __restrict__ parts, int t, int m, int panel, double* __restrict__ W,
               int* __restrict__ piv, __nv_bfloat16* __restrict__ Us, int* __restrict__ Uexp,
               __nv_bfloat16* __restrict__ Vs, int* __restrict__ Vexp, int* __restrict__ status) {
  extern __shared__ __align__(16) double P[];  // [16 ceil(m / 16)][PS], then U's digits by tile
  __shared__ GjShared sh;
  constexpr int kWorkers = CW + kHelpers, kWarps = kWorkers + 1, kThreads = 32 * kWarps;  // the last: control
  __shared__ GjDigits dg;
  __shared__ int piv_s[PW];
  __shared__ uint32_t used[kMaxM / 32];
  const int q = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const PartDesc p = parts[q];
  if (t >= p.L) return;
  double* M = W + (long long)q * m * m;
  const int k0 = PW * panel, kw = min(PW, m - k0), mt = (m + 15) / 16;
  const int nw = min(CW, (m + 31) / 32);
  uint32_t* Ud = reinterpret_cast<uint32_t*>(P + 16 * mt * PS);
  if (tid < kMaxM / 32) used[tid] = 0;
  __syncthreads();
  for (int k = tid; k < k0; k += kThreads) {
    const int r = piv[(long long)q * m + k];
    atomicOr(&used[r >> 5], 1u << (r & 31));
  }
#pragma unroll 8
  for (int i = warp; i < 16 * mt; i += kWarps)
    P[i * PS + lane] = (i < m && lane < kw) ? M[(long long)i * m + k0 + lane] : 0.0;
  __syncthreads();
  bool bad = false;
  // Per subpanel: the pivots on the chain's warps and the control warp while the helpers
  // finish the rank-8 update of the subpanel before (its 16 columns that are
  // not next); then all of them but the control warp update the next subpanel's columns (after the
  // last subpanel all other columns), which its chain waits for.
#pragma unroll 1
  for (int c0 = 0; c0 < kw; c0 += SW) {
    const int w = min(SW, kw - c0);
    if (warp < nw)
      gj_chain<CW, RPL>(P, m, c0, w, nw, used, sh, warp, lane);
    else if (warp == kWorkers)
      gj_control(m, c0, w, nw, sh, piv_s, lane, bad);
    else if (warp >= CW && c0 > 0)
      gj_rank8(P, Ud, dg, mt, c0 - SW, c0 + SW, 2, false, true, warp - CW, kHelpers);
    __syncthreads();
    // this subpanel's pivot rows
    if (tid < SW * PW) gj_digits_v(P, piv_s + c0, w, dg, tid);
    if (tid >= SW * PW && tid < SW * PW + kMaxM / 32) {
      uint32_t bits = 0;
      for (int j = 0; j < w; ++j)
        if ((piv_s[c0 + j] >> 5) == tid - SW * PW) bits |= 1u << (piv_s[c0 + j] & 31);
      dg.pivots[tid - SW * PW] = bits;
      used[tid - SW * PW] |= bits;
    }
    __syncthreads();
    if (kw > SW && warp < kWorkers) {
      const bool last = c0 + SW >= kw;
      gj_rank8(P, Ud, dg, mt, c0, c0 + SW, last ? 3 : 1, !last, false, warp, kWorkers);
    }
    __syncthreads();
  }
  if (tid < kw) piv[(long long)q * m + k0 + tid] = piv_s[tid];
  // the eliminated panel and the row slices of U (scale per row over its 32
  // values): four threads per row, eight values each
#pragma unroll 1
  for (int i0 = 0; i0 < m; i0 += kThreads / 4) {
    const int i = i0 + (tid >> 2), cb = (tid & 3) * 8;
    double v[8];
    uint32_t hmax = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      v[c] = i < m ? P[i * PS + cb + c] : 0.0;
      hmax = max(hmax, abs_hi(v[c]));
    }
    hmax = max(hmax, __shfl_xor_sync(0xffffffffu, hmax, 1));
    hmax = max(hmax, __shfl_xor_sync(0xffffffffu, hmax, 2));
    if (i < m) {
      const int e = scale_exponent(hmax);
      if ((tid & 3) == 0) Uexp[(long long)q * m + i] = e;
      gj_slice8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], e, Us + (long long)q * S * m * PW + (long long)i * PW + cb, m * PW);
    }
  }
  for (int i = warp; i < m; i += kWarps)
    if (lane < kw) M[(long long)i * m + k0 + lane] = P[i * PS + lane];
  // the column slices of V = the pivot rows outside the panel (transposed: row
  // j of the copy holds V[0..31][j]; the panel's own columns are never read)
#pragma unroll 1
  for (int j0 = 0; j0 < m; j0 += kThreads / 4) {
    const int j = j0 + (tid >> 2), cb = (tid & 3) * 8;  // four threads per column, eight rows each
    const bool in = j < m && (j < k0 || j >= k0 + kw);
    double v[8];
    uint32_t vmax = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = in && cb + c < kw ? M[(long long)piv_s[cb + c] * m + j] : 0.0;
#pragma unroll
    for (int c = 0; c < 8; ++c) vmax = max(vmax, abs_hi(v[c]));
    vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, 1));
    vmax = max(vmax, __shfl_xor_sync(0xffffffffu, vmax, 2));
    if (in) {
      const int e = scale_exponent(vmax);
      if ((tid & 3) == 0) Vexp[(long long)q * m + j] = e;
      gj_slice8(v[0], v[1], v[2], v[3], v[4], v[5], v[6], v[7], e, Vs + (long long)q * S * m * PW + (long long)j * PW + cb, m * PW);
    }
  }
  if (bad) atomicMin(status + p.sys, p.row0 + t + 1);
}

// After the last panel: X[k][p_j] = W[p_k][j], X = (2^-rho D 2^-gam)^{-1}, moved to its
// place in G as D^{-1} = 2^-gam X 2^-rho
// and the row slices of the block inverse G_t written (the left operand of
// the next products), one pass: a CTA takes 32 rows of one block (blockIdx.x
// = block * groups + group), a warp a row at a time: the row is read once,
// scattered to its final column order in shared memory (its largest magnitude
// does not depend on the order), then written as float64 and as digit slices.
template <int S>
__global__ void __launch_bounds__(256) k_gj_finish(const PartDesc* __restrict__ parts, int t, int m,
                                                   const double* __restrict__ W, double* __restrict__ G,
                                                   const int* __restrict__ piv, __nv_bfloat16* __restrict__ Gs,
                                                   int* __restrict__ eG, const int* __restrict__ gam,
                                                   const int* __restrict__ rho, const int* __restrict__ be) {
  __shared__ int ip[kMaxM], rs[kMaxM], ds[kMaxM];
  __shared__ double rowb[8][kMaxM];
  const int groups = (m + 31) / 32;
  const int q = blockIdx.x / groups, g = blockIdx.x - q * groups;
  const PartDesc p = parts[q];
  if (t >= p.L) return;
  const long long mm = (long long)m * m;
  const int mp = slice_pitch(m);
  const double* M = W + (long long)q * mm;
  double* Gt = G + p.blk + (long long)t * mm;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long vt = p.blk / m + (long long)t * m;  // the block row's exponents
  for (int c = threadIdx.x; c < m; c += blockDim.x) ip[c] = piv[(long long)q * m + c], rs[c] = rho[vt + c], ds[c] = be[vt + c] - rs[c];
  const int gv = 32 * g + lane < m ? gam[vt + 32 * g + lane] : 0;  // of the CTA's rows
  __syncthreads();
  double* rb = rowb[warp];
  const int rend = min(m, 32 * g + 32);
  for (int r = 32 * g + warp; r < rend; r += 8) {
    int key = kNoKey;
    const double* src = M + (long long)ip[r] * m;
    for (int c = lane; c < m; c += 32) {
      const double v = src[c];
      rb[ip[c]] = v;
      key = max(key, scale_key(abs_hi(v), ds[ip[c]]));
    }
    // the slices are of G_t 2^be (dm_oz.cu) = 2^-gam X 2^(be - rho)
    const int e = key_exponent(__reduce_max_sync(0xffffffffu, key));
    const int gr = __shfl_sync(0xffffffffu, gv, r - 32 * g);
    if (lane == 0) eG[(long long)q * m + r] = e - gr;
    __syncwarp();
    for (int c = lane; c < m; c += 32) Gt[(long long)r * m + c] = scale_pow2(rb[c], -(gr + rs[c]));
    for (int c0 = lane * 8; c0 < m; c0 += 256) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = c0 + u < m ? rb[c0 + u] : 0.0;
      uint32_t d[8][S];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        digits<S>((unsigned long long)__double_as_longlong(v[u]), e - (c0 + u < m ? ds[c0 + u] : 0), d[u]);
#pragma unroll
      for (int sl = 0; sl < S; ++sl)
        *reinterpret_cast<uint4*>(Gs + (((long long)q * S + sl) * m + r) * mp + c0) =
            make_uint4(pack_hi(d[0][sl], d[1][sl]), pack_hi(d[2][sl], d[3][sl]), pack_hi(d[4][sl], d[5][sl]),
                       pack_hi(d[6][sl], d[7][sl]));
    }
    __syncwarp();
  }
}

}  // namespace gj

// The blocked Gauss-Jordan inversion of block row t of every active subsystem
// (working matrix W: D_t, written by launch B of the step before), as phases:
// the copy of B_0, per panel of 32 columns the panel and its trailing update
// (dm_oz.cu), and the finishing pass.
void launch_gj_begin(const PartDesc* parts, int nparts, int t, int m, const double* B, double* W, const int* gam,
                     const int* rho, cudaStream_t st) {
  if (nparts > 0 && t == 0)
    gj::k_gj_copy_b0<<<dim3(nparts, std::max(1, m * m / 8192)), 256, 0, st>>>(parts, m, B, W, gam, rho);
}

void launch_gj_panel(const PartDesc* parts, int nparts, int t, int m, int pnl, double* W, int* piv, void* Us,
                     int* Uexp, void* Vs, int* Vexp, int* status, cudaStream_t st) {
  if (nparts <= 0) return;
  const size_t smem = gj::smem_bytes((m + 15) / 16);
#define DM_GJ(C_, R_)                                                                                                   \
  do {                                                                                                              \
    allow_smem(gj::k_gj_panel<C_, R_>, smem);                                                                       \
    gj::k_gj_panel<C_, R_><<<nparts, 32 * (C_ + gj::kHelpers + 1), smem, st>>>(                                     \
        parts, t, m, pnl, W, piv, static_cast<__nv_bfloat16*>(Us), Uexp, static_cast<__nv_bfloat16*>(Vs), Vexp,     \
        status);                                                                                                    \
  } while (0)
  if (m <= 128) DM_GJ(4, 1);
  else if (m <= 256) DM_GJ(8, 1);
  else DM_GJ(8, 2);
#undef DM_GJ
}

void launch_gj_finish(const PartDesc* parts, int nparts, int t, int m, const double* W, double* G, const int* piv,
                      void* Gs, int* eG, const OzScales& sc, cudaStream_t st) {
  if (nparts <= 0) return;
  const int grid = nparts * ((m + 31) / 32);
  auto* g = static_cast<__nv_bfloat16*>(Gs);
  if (oz_slices(m) == 7)
    gj::k_gj_finish<7><<<grid, 256, 0, st>>>(parts, t, m, W, G, piv, g, eG, sc.gam, sc.rho, sc.be);
  else
    gj::k_gj_finish<8><<<grid, 256, 0, st>>>(parts, t, m, W, G, piv, g, eG, sc.gam, sc.rho, sc.be);
}

}  // namespace dm
