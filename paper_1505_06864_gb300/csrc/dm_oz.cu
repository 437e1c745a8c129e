// Float64 block products of the factor sweeps on the bf16 tensor cores by
// exact digit slicing (Ozaki's error-free splitting of matrix products; the
// digit extraction, accumulator grouping and pipeline are this library's).
//
// The products are the ones of the tensor-core step kernels (dm_tc2.cu):
// launch A = G_t [C_t | Y_t], launch B = A_{t+1} [Acal_t | Bcal_t], backward
// Acal_t [ZL_{t+1} | ZR_{t+1}] (Section 3 applied to Eq. e231), here with
// float64 operands and results.  Every operand block is cut into S digit
// slices (dm_slices.cuh): a left operand L with one power-of-two scale per
// row r (|L[r][k]| < 2^e_r), a right operand R with one per column n
// (|R[k][n]| < 2^f_n), stored transposed (row n of the copy is column n of
// R).  Then, with the digits' base b = 2^8 (S = 7) or 2^7 (S = 8),
//
//   (L R)[r][n] = 2^(e_r + f_n + 2) sum_{d=2..S+2} b^(-d) acc_d[r][n],
//   acc_d = sum_{s+t=d} Lslice_s Rslice_t,
//
// The error of an entry is so bounded by the largest entries of the row and
// the column, where a float64 dot product's is by its terms.  Where equations
// or unknowns differ in scale, entry k of the row is large just where entry k
// of the column is small, and one scale per row and column would lose the
// small ones (m = 100, rows scaled over eight decades: solutions to 1e-11
// against 1.5e-13).  So the operands are balanced along k by exact powers of
// two, one per equation (be) or unknown (bu) of a block row, found before
// the sweeps (k_level_scan): L[r][k] 2^(s_k) times 2^(-s_k) R[k][n],
// inside the extraction of the digits.  The products' results, and all that is
// stored in float64, are not scaled.
//
// Kept are the slice pairs with s + t <= S + 2 (34 of 49 and 43 of 64).  The
// digits are balanced (|digit| <= b / 2), so each acc_d is an integer of at most
// S K b^2 / 4 <= 2^24 for K <= 128 (S = 7) and K <= 512 (S = 8), and the
// float32 accumulation in tensor memory is exact.  Operands are rounded at
// 2^-56 of their scale (as far as they are smaller than a quarter of it: the
// others are exact), the dropped pairs are below 2^-61 sqrt(K) max_k |L[r][k]|
// max_k |R[k][n]|.  (Without the last diagonal, 28 and 36 pairs, the dropped
// ones doubled the error of systems with cond(B_i) = 1e4.)
//
// A CTA computes a tile of one product: 128 x 64 (S = 7) or 128 x 48 (S = 8),
// 128 x 32 for KIND 3: S + 1 accumulators in tensor memory (512 or 432 columns;
// KIND 3: two sets of 256), a two-stage ring of 32-wide K slabs, one CTA per
// SM.  Per 16-wide K step one thread issues the MMAs: left slice s against
// right slices t = 1 .. min(S, S + 2 - s) at once (stored consecutively, at
// most N = 256 per instruction), into accumulators d = s + t; s = 1 and the
// pair (2, S) cover all of them, so they initialise them in the first K step.
// The epilogue combines the accumulators in 64-bit integers and scales once in
// float64 (GB300's float64 pipe is narrow).  Operand slices of results are
// made by separate slicing launches, which see whole rows and columns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "dm_internal.cuh"
#include "dm_slices.cuh"
#include "dm_tcgen05.cuh"

namespace dm {
namespace oz {
using namespace ptx;

__host__ __device__ constexpr int epi_warps(int kind, int S) { return kind != 3 && S == 8 ? 12 : 16; }  // epilogue warps from 2 on
__host__ __device__ constexpr int threads_of(int kind, int S) {  // warp 0: TMA producer, warp 1: MMA issuer
  return 64 + 32 * epi_warps(kind, S);
}
constexpr int MT = 128;          // rows per tile
constexpr int NT3 = 32;          // columns per tile of the inverse's trailing updates (KIND 3)
constexpr int KS = 32;           // K elements per stage (64-byte rows, 64-byte swizzle)
constexpr int kStages = 2;
constexpr int ROWB = KS * 2;     // 64 bytes
constexpr int LSL = MT * ROWB;   // one left slice in a stage: 8 KB
constexpr int STG = 32 * 8;                  // an epilogue warp's 32 x 8 float64 staging tile
constexpr uint32_t kCols = 512;
constexpr uint32_t kSbo = 8 * ROWB;  // 512-byte swizzle atoms
constexpr uint64_t kLayout = 4;       // 64-byte swizzle

// columns per tile
constexpr int nt_of(int kind, int S) { return kind == 3 ? NT3 : S == 7 ? 64 : 48; }
// bytes of a stage and of the kernel's shared memory
template <int KIND, int S>
constexpr int stage_bytes() {
  return S * (LSL + nt_of(KIND, S) * ROWB);
}
template <int KIND, int S>
constexpr int smem_bytes() {
  return 1024 + kStages * stage_bytes<KIND, S>() + epi_warps(KIND, S) * STG * 8;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, int w,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
      : "memory");
}

// The integer value of an integer-valued float32 |v| <= 2^22: v + 1.5 2^23
// lies in [2^23, 2^24], where the float's low mantissa bits are v's.
__device__ __forceinline__ int acc_int_small(float v) { return __float_as_int(v + 12582912.0f) - 0x4B400000; }

}  // namespace oz

struct OzMaps {
  CUtensorMap L, R0, R1;
};

namespace oz {

// KIND 0: launch A, 1: launch B (forward step `step`), 2: backward step
// `step`, over the subsystems.  Exponent arrays: [block][m] ints, indexed
// like the slices.
// KIND 3: the trailing update of panel `step` (columns K = [32 step, 32 step
// + 32), pivot rows p_K = piv[K]) of the blocked Gauss-Jordan inversion of
// block row `aux` in the working matrix: M[:, J] = (M[:, J] with the rows p_K
// zeroed) + U V, U the eliminated panel, V = M[p_K, J] before the update
// (both as slices, K = 32), J the other columns.
// KIND 4, 5: the supplementary blocks of a separator (Eq. e2311), left A_q /
// C_q: KIND 4 j = 0: HB = B_q - A_q ZR^j[q-1], j = 1: HA = -A_q ZL^j[q-1];
// KIND 5 j = 0: HB -= C_q ZL^{j+1}[q+1], j = 1: HC = -C_q ZR^{j+1}[q+1]
// (parts unused, out.seps instead).
//
// A tile = (subsystem or separator, product j, 128-row M-tile, N-tile
// of nt_of columns); tile = ((unit * 2 + j) * ntm + M-tile) * ntn + N-tile (KIND 3,
// one product: (unit * ntm + M-tile) * ntn + N-tile).
struct OzTile {
  PartDesc p;
  SepDesc sd;
  int unit, j, tm, tn, t, zl, zr;
  bool act;
};

template <int KIND, int S>
__device__ __forceinline__ OzTile oz_tile(int tile, const PartDesc* __restrict__ parts, const OzOut& out, int step,
                                          int aux, int m, int ntm, int ntn) {
  OzTile w{};
  constexpr int nj = KIND == 3 ? 1 : 2;  // KIND 3 has one product
  const int per = nj * ntm * ntn;
  w.unit = tile / per;
  const int rest = tile - w.unit * per;
  w.tn = rest % ntn;
  // KIND 3: the 32-column tile equal to panel `step` produces nothing and is
  // not enumerated (ntn counts the others)
  if (KIND == 3 && w.tn >= step) ++w.tn;
  const int r2 = rest / ntn;
  w.j = nj == 1 ? 0 : (r2 & 1);
  w.tm = nj == 1 ? r2 : (r2 >> 1);
  if constexpr (KIND >= 4)
    w.sd = out.seps[w.unit];
  else
    w.p = parts[w.unit];
  const PartDesc& p = w.p;
  const int j = w.j, pidx = w.unit;
  bool act;
  if (KIND == 4) {
    act = j == 0 || (w.sd.flags & HAS_HA) != 0;
  } else if (KIND == 5) {
    act = j == 0 || (w.sd.flags & HAS_HC) != 0;
  } else if (KIND == 0) {
    w.t = step;
    act = w.t < p.L && (j == 0 ? (w.t < p.L - 1 || (p.flags & HAS_RIGHT) != 0) : (p.flags & HAS_LEFT) != 0);
  } else if (KIND == 1) {
    w.t = step;
    act = w.t < p.L - 1 && (j == 0 || (p.flags & HAS_LEFT) != 0);
  } else if (KIND == 2) {
    w.t = p.L - 2 - step;
    act = w.t >= 0 && (j == 0 ? (p.flags & HAS_LEFT) != 0 : (p.flags & HAS_RIGHT) != 0);
  } else {
    w.t = aux;
    act = w.t < p.L && j == 0;
  }
  // products with a banded operand run in the banded kernels instead
  const bool banded = out.band && *out.band <= kBandMax;
  if (banded && ((KIND == 0 && j == 0) || KIND == 1 || KIND >= 4)) act = false;
  w.act = act && w.tm * MT < m && w.tn * nt_of(KIND, S) < m;
  const long long mm = (long long)m * m;
  const int b0 = (int)(p.blk / mm), t = w.t;
  if (KIND == 4) {
    w.zl = (int)(w.sd.blk_q / mm);  // A_q (all blocks)
    w.zr = 4 * pidx + j;            // ZR^j[q-1]^T / ZL^j[q-1]^T
  } else if (KIND == 5) {
    w.zl = pidx;                    // C_q (per separator)
    w.zr = 4 * pidx + 2 + j;        // ZL^{j+1}[q+1]^T / ZR^{j+1}[q+1]^T
  } else if (KIND == 3) {
    w.zl = pidx;  // U slices (rolling)
    w.zr = pidx;  // V^T slices (rolling)
  } else if (KIND == 0) {
    w.zl = pidx;                     // G_t slices (rolling)
    w.zr = j == 0 ? b0 + t : pidx;   // C_t^T (all blocks) / Y_t^T (rolling)
  } else if (KIND == 1) {
    w.zl = b0 + t + 1;                          // A_{t+1}
    w.zr = j == 0 ? pidx : 2 * pidx + (t & 1);  // Acal_t^T / Bcal_t^T
  } else {
    w.zl = b0 + t;                    // Acal_t
    w.zr = 2 * pidx + ((t + 1) & 1);  // ZL_{t+1}^T / ZR_{t+1}^T
  }
  return w;
}

// Persistent: a CTA per SM walks the tiles blockIdx.x, blockIdx.x + gridDim.x,
// ...  Warp 0 (one lane) streams every tile's K slabs by TMA into a two-stage
// ring and runs ahead into the next tile; warp 1 (one lane) issues the MMAs
// of a tile once the epilogue has drained the accumulators they go to (KIND 3
// has two sets, so its MMAs run beside the previous tile's epilogue; the
// other kinds' accumulators fill the tensor memory); warps from 2 on run the
// epilogue (KIND 3: two teams of eight, a set of accumulators each), loading
// what it needs besides the accumulators while the MMAs run.  Every wait is bounded; a role that gives up sets `err`, which the
// others see at their next tile.
template <int KIND, int S>
__global__ void __launch_bounds__(threads_of(KIND, S), 1)
    k_oz_step(const PartDesc* __restrict__ parts, int step, int aux, int m, int ntm, int ntn, int ntiles, OzOut out,
              const int* __restrict__ lexp, const int* __restrict__ rexp0, const int* __restrict__ rexp1,
              int* __restrict__ errflag, const __grid_constant__ OzMaps maps) {
  constexpr int kEpi = epi_warps(KIND, S);
  constexpr int NTK = nt_of(KIND, S);   // columns per tile
  constexpr int NACC = S + 1;            // accumulators d = 2 .. S + 2
  constexpr int RSLK = NTK * ROWB;      // one right slice in a stage
  constexpr int LBYTES = S * LSL, STAGE = stage_bytes<KIND, S>();
  constexpr int SETC = NACC * NTK;                         // tensor-memory columns of one set of accumulators
  constexpr int NBUF = 2 * SETC <= (int)kCols ? 2 : 1;  // sets
  constexpr int DB = S == 7 ? 8 : 7;                    // bits per digit
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t full[kStages], empty[kStages], tfull[2], tempty[2], mdone;
  __shared__ uint32_t tmem_slot;
  __shared__ int err, nissued, ncons;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  double* stage_out = reinterpret_cast<double*>(base + kStages * STAGE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* verr = &err;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&tfull[s], 1);
      mbar_init(&tempty[s], kEpi / NBUF);
    }
    mbar_init(&mdone, 1);
    err = 0;
    nissued = 0;
    ncons = 0;
    fence_mbar_init();
  }
  if (warp == 1) tmem_alloc(&tmem_slot, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const long long mm = (long long)m * m;
  const int nslab = KIND == 3 ? 1 : (m + KS - 1) / KS;
  constexpr uint32_t tx = (uint32_t)(S * (MT + NTK) * ROWB);

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      for (int tile = blockIdx.x; tile < ntiles && !*verr; tile += gridDim.x) {
        const OzTile w = oz_tile<KIND, S>(tile, parts, out, step, aux, m, ntm, ntn);
        if (!w.act) continue;
        const CUtensorMap* mr = w.j == 0 ? &maps.R0 : &maps.R1;
        bool ok = true;
        for (int s = 0; s < nslab; ++s, ++it) {
          const int st = it & 1;
          if (it >= kStages && !mbar_wait(&empty[st], (uint32_t)(((it >> 1) - 1) & 1))) {
            ok = false;
            break;
          }
          const uint32_t sb = smem_u32(base + st * STAGE);
          mbar_expect_tx(&full[st], tx);
          tma_load_4d(sb, &maps.L, s * KS, w.tm * MT, 0, w.zl, &full[st]);
          tma_load_4d(sb + LBYTES, mr, s * KS, w.tn * NTK, 0, w.zr, &full[st]);
        }
        if (!ok) {
          *verr = 1;
          break;
        }
      }
      nissued = it;
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      int it = 0, lt = 0;
      for (int tile = blockIdx.x; tile < ntiles && !*verr; tile += gridDim.x) {
        const OzTile w = oz_tile<KIND, S>(tile, parts, out, step, aux, m, ntm, ntn);
        if (!w.act) continue;
        // the accumulators of the tile that used this set before have been read
        const int bf = lt % NBUF, use = lt / NBUF;
        if (use > 0 && !mbar_wait(&tempty[bf], (uint32_t)((use - 1) & 1))) {
          *verr = 1;
          break;
        }
        tc_fence_after();
        bool ok = true;
        for (int s = 0; s < nslab; ++s, ++it) {
          const int st = it & 1;
          if (!mbar_wait(&full[st], (uint32_t)((it >> 1) & 1))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t la = smem_u32(base + st * STAGE), ra = la + LBYTES;
#pragma unroll
          for (int k = 0; k < KS / 16; ++k) {
            const uint32_t off = (uint32_t)(k * 32);
#pragma unroll
            for (int sl = 1; sl <= S; ++sl) {
              constexpr int per = 256 / NTK;  // right slices per instruction
              const int T = min(S, S + 2 - sl);
              const uint64_t ad = kmajor_desc(la + (sl - 1) * LSL + off, kSbo, kLayout);
#pragma unroll
              for (int ta = 1, cnt = 0; ta <= T; ta += cnt) {
                cnt = min(per, T - ta + 1);
                if (sl == 2 && ta < S && ta + cnt > S) cnt = S - ta;  // (2, S) by itself
                const uint64_t bd = kmajor_desc(ra + (ta - 1) * RSLK + off, kSbo, kLayout);
                const uint32_t dcol = (uint32_t)(bf * SETC + (sl + ta - 2) * NTK);
                const uint32_t acc = (s == 0 && k == 0 && (sl == 1 || (sl == 2 && ta == S))) ? 0u : 1u;
                mma<1>(tmem + dcol, ad, bd, make_idesc(1u, MT, NTK * cnt), acc);
              }
            }
          }
          mma_commit(&empty[st]);
        }
        if (!ok) {
          *verr = 1;
          break;
        }
        mma_commit(&tfull[bf]);
        ++lt;
      }
      ncons = it;
      // every MMA issued here is complete before the accumulators are freed
      mma_commit(&mdone);
      mbar_wait(&mdone, 0u);
    }
    __syncwarp();
  } else {
    // a warp reaches tensor-memory lanes 32 (warp % 4) ..; the warps of a team
    // that share a lane quarter share the tile's columns, CW each
    constexpr int CW = NTK / (kEpi / NBUF / 4);
    const int ew = warp - 2, quarter = warp & 3, team = NBUF == 2 ? ew >> 3 : 0, part = NBUF == 2 ? (ew >> 2) & 1 : ew >> 2;
    double* stg = stage_out + ew * STG;
    const int cl = lane & 7, r0 = lane >> 3;
    const int k0 = 32 * step;  // KIND 3: the panel's columns
    int lt = 0;
    for (int tile = blockIdx.x; tile < ntiles && !*verr; tile += gridDim.x) {
      const OzTile w = oz_tile<KIND, S>(tile, parts, out, step, aux, m, ntm, ntn);
      if (!w.act) continue;
      const int bf = lt % NBUF, use = lt / NBUF;
      ++lt;
      if (NBUF == 2 && bf != team) continue;
      const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(bf * SETC);
      const int j = w.j, t = w.t, pidx = w.unit;
      const PartDesc& p = w.p;
      const SepDesc& sd = w.sd;
      const int* rexp = j == 0 ? rexp0 : rexp1;
      // Before the accumulators are ready: the row's scale, the column scales
      // of the warp's columns (one per lane, passed by shuffle) and the
      // values the stores update (they do not depend on the products)
      const int rbase = w.tm * MT + quarter * 32, row = rbase + lane;
      const int cbase = w.tn * NTK + part * CW;  // the warp's columns
      int er = row < m ? lexp[(long long)w.zl * m + row] : 0;
      int fexp = lane < CW && cbase + lane < m ? rexp[(long long)w.zr * m + cbase + lane] : 0;
      const bool rmw = KIND == 2 && j == 0, dnext = KIND == 1 && j == 0, gj = KIND == 3, hb = KIND >= 4 && j == 0;
      const bool upd = rmw || dnext || gj || hb;
      const long long o = p.blk + (long long)t * mm;
      // the working matrix of the blocked inversion (or D_{t+1}'s place in G)
      double* const wk = out.W ? out.W + (long long)pidx * mm : out.G + o + mm;
      const double* src = rmw    ? out.ZL + o
                          : gj   ? wk
                          : hb   ? (KIND == 4 ? out.B + sd.blk_q : out.HB + sd.hblk)
                                 : out.B + o + mm;
      // D_{t+1} goes into the working matrix equilibrated (the exponents as the
      // scales: of the lane's row, and a column of the warp's per lane): the
      // product by its scales, B_{t+1} as it is loaded
      const bool even = KIND == 1 && dnext && out.W != nullptr;
      int rrow = 0, gcol = 0;
      if (even) {
        const long long v1 = (o + mm) / m;  // block row t + 1
        if (row < m) rrow = out.rho[v1 + row];
        if (lane < CW && cbase + lane < m) gcol = out.gam[v1 + cbase + lane];
        er -= rrow;
        fexp -= gcol;
      }
      // where the results go
      double* dst;
      if (KIND >= 4)
        dst = (j == 0 ? out.HB : KIND == 4 ? out.HA : out.HC) + sd.hblk;  // HB = B_q - A_q ZR, then HB -= C_q ZL;
                                                                         // HA = -A_q ZL, HC = -C_q ZR
      else if (KIND == 0)
        dst = (j == 0 ? (t < p.L - 1 ? out.Acal : out.ZR) : out.ZL) + o;
      else if (KIND == 1)
        dst = j == 0 ? wk : out.Y + (long long)pidx * mm;  // D_{t+1} = B_{t+1} - A_{t+1} Acal_t, Y = -A_{t+1} Bcal_t
      else if (KIND == 2)
        dst = (j == 0 ? out.ZL : out.ZR) + o;  // ZL_t -= Acal_t ZL_{t+1}, ZR_t = -Acal_t ZR_{t+1}
      else
        dst = wk;                              // Gauss-Jordan trailing update
      // KIND 3: which of the warp's 32 rows are pivot rows of the panel
      uint32_t zrows = 0;
      if (KIND == 3) {
        const int pv = k0 + lane < m ? out.piv[(long long)pidx * m + k0 + lane] : -1;
        zrows = __reduce_or_sync(0xffffffffu, pv >= 0 && (pv >> 5) == (rbase >> 5) ? 1u << (pv & 31) : 0u);
      }
      // the values chunk ci's stores update, loaded before its accumulators are converted
      auto load_in = [&](int ci, double (&in)[8]) {
        const int n = cbase + 8 * ci + cl;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int rr = rbase + r0 + 4 * i;
          in[i] = (upd && n < m && rr < m && !(gj && ((zrows >> (r0 + 4 * i)) & 1u))) ? src[(long long)rr * m + n]
                                                                                      : 0.0;
        }
        if (even) {
          const int gn = __shfl_sync(0xffffffffu, gcol, 8 * ci + cl);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            in[i] = scale_pow2(in[i], -(__shfl_sync(0xffffffffu, rrow, r0 + 4 * i) + gn));
        }
      };
      double in[8];
      load_in(0, in);
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&tfull[bf], (uint32_t)(use & 1)));
      if (!ok) {
        *verr = 1;
        break;
      }
      tc_fence_after();
      // Accumulators of this thread's row (tensor-memory lane) for 8 columns
      // at a time.  Each acc_d is an integer-valued float of at most 2^24 (its
      // integer by float32 or conversion instructions); with b the digits'
      // base,
      //   S = 7: hi = (acc_2 b + acc_3) b + acc_4, lo the other five (< 2^56),
      //   S = 8: hi = ((acc_2 b + acc_3) b + acc_4) b + acc_5, lo the other five (< 2^53)
      // give the sum exactly as hi b^5 + lo.  It is rounded to a 64-bit integer
      // T (at 2^-57 (S = 7; KIND 3: 2^-59), 2^-55 (S = 8) of 2^(e_r + f_n + 2), below the
      // operands' own rounding) and T to float64, both in integer
      // instructions: a float64 instruction holds its warp for 64 cycles, so
      // only the addition of an updated value is one.  Results are staged
      // through the warp's 32 x 8 float64 tile so that row-major writes are
      // coalesced.  The chunk loop stays rolled: unrolled, a launch of few
      // tiles waited for its instructions.
#pragma unroll 1
      for (int ci = 0; ci < CW / 8; ++ci) {
        const int ch = part * CW + 8 * ci;
        // chunks past the block's last column produce nothing: only the
        // release of the accumulators after the last chunk remains
        const bool dead = cbase + 8 * ci >= m, last = ci == CW / 8 - 1;
        if (dead) {
          if (last) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[bf]);
          }
          continue;
        }
        if (ci > 0) load_in(ci, in);
        uint32_t r[NACC][8];
#pragma unroll
        for (int dd = 0; dd < NACC; ++dd) tmem_ld8_nowait(tl + (uint32_t)(dd * NTK + ch), r[dd]);
        tmem_wait_ld();
#pragma unroll
        for (int dd = 0; dd < NACC; ++dd) tmem_regs_after_wait(r[dd]);
        if (last) {  // the last accumulator read of this tile: the MMAs may go on
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&tempty[bf]);
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int k = er + __shfl_sync(0xffffffffu, fexp, 8 * ci + c) + 2;
          // |acc_d| <= (d - 1) K b^2 / 4, at most 2^22 for K = 32 always, else
          // for the first two
          int a[NACC];
#pragma unroll
          for (int dd = 0; dd < NACC; ++dd)
            a[dd] = KIND == 3 || dd < 2 ? acc_int_small(__uint_as_float(r[dd][c]))
                                        : __float2int_rn(__uint_as_float(r[dd][c]));
          long long hi, lo;
          if (S == 7) {
            hi = (long long)a[0] * 65536 + (a[1] * 256 + a[2]);
            lo = (((long long)a[3] * 256 + a[4]) * 256 + a[5]) * 65536 + ((long long)a[6] * 256 + a[7]);
          } else {
            hi = (long long)(a[0] * 128 + a[1]) * 16384 + (a[2] * 128 + a[3]);
            lo = (long long)(a[4] * 128 + a[5]) * 2097152 + (long long)(a[6] * 128 + a[7]) * 128 + a[NACC - 1];
          }
          // |hi| < 2^35 (KIND 3), 2^38 (S = 7), 2^42 (S = 8): T = (hi b^5 + lo) / 2^drop below 2^63
          constexpr int ulo = DB * (S + 2), drop = KIND == 3 ? 13 : 15, up = 5 * DB - drop;
          const long long T = hi * (1ll << up) + ((lo + (1 << (drop - 1))) >> drop);
          bool odd = false;
          double val = round_scaled(T, k - ulo + drop, odd);
          const float a2 = __uint_as_float(r[0][c]);
          if (odd || a2 != a2)  // outside the normal range; NaN or infinite operand: its first digit is NaN, so acc_2 is
            val = a2 != a2 ? __longlong_as_double(0x7ff8000000000000ll) : ldexp((double)T, k - ulo + drop);
          stg[lane * 8 + (c ^ (lane & 7))] = val;
        }
        __syncwarp();
        // row-major float64 results: lane = (row quarter, column), 8 row quads
        const int n = cbase + 8 * ci + cl;
        if (n < m) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int rl = r0 + 4 * i, rr = rbase + rl;
            if (rr >= m) continue;
            const double v = stg[rl * 8 + (cl ^ (rl & 7))];
            dst[(long long)rr * m + n] = gj ? in[i] + v : upd ? in[i] - v : KIND == 0 ? v : -v;
          }
        }
        __syncwarp();
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0)  // copies still in flight after an error
    for (int s = ncons; s < nissued; ++s) mbar_wait(&full[s & 1], (uint32_t)((s >> 1) & 1));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kCols);
  if (threadIdx.x == 0 && err && errflag) atomicExch(errflag, 1);
}

// ---------------------------------------------------------------- slicing
// A CTA slices one group of 32 rows (left operands) or 32 columns (right
// operands) of one float64 m x m block; a block takes ceil(m / 32) CTAs.  The
// entries of index k (columns of a left operand, rows of a right one) take
// part with 2^(sh.sign sh.kap[k]).  (Read beside the entries: staged in shared
// memory, a load and a barrier ahead of them, they cost a launch of few blocks
// 1 us.)
struct Shift {
  const int* kap;
  int sign;
  __device__ __forceinline__ int operator()(int k) const { return sign * __ldg(kap + k); }
};

// Row slices (left operands): exps[r] = e with |v 2^shift| < 2^e for the row's
// entries v; slice s element (r, k) at ((q * S + s) m + r) pitch + k, the
// pitch m rounded up to 8 (16-byte rows for TMA; the columns past m are zero).
// One warp per row, eight consecutive columns per lane.
template <int S>
__device__ __forceinline__ void slice_rows_group(const double* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                                                 long long qdst, int* __restrict__ exps, int m, int g,
                                                 Shift sh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int mp = slice_pitch(m);
  const unsigned long long* bits = reinterpret_cast<const unsigned long long*>(src);
  const int rend = min(m, 32 * g + 32);
  for (int r = 32 * g + warp; r < rend; r += nw) {
    int key = kNoKey;
    for (int c = lane; c < m; c += 32) key = max(key, scale_key((uint32_t)(bits[(long long)r * m + c] >> 32), sh(c)));
    const int e = key_exponent(__reduce_max_sync(0xffffffffu, key));
    if (lane == 0) exps[qdst * m + r] = e;
    for (int c0 = lane * 8; c0 < m; c0 += 256) {
      uint32_t q[8][S];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const bool in = c0 + u < m;
        digits<S>(in ? bits[(long long)r * m + c0 + u] : 0ull, in ? e - sh(c0 + u) : e, q[u]);
      }
#pragma unroll
      for (int sl = 0; sl < S; ++sl) {
        uint4 w;
        w.x = (q[0][sl] >> 16) | (q[1][sl] & 0xffff0000u);
        w.y = (q[2][sl] >> 16) | (q[3][sl] & 0xffff0000u);
        w.z = (q[4][sl] >> 16) | (q[5][sl] & 0xffff0000u);
        w.w = (q[6][sl] >> 16) | (q[7][sl] & 0xffff0000u);
        *reinterpret_cast<uint4*>(dst + ((qdst * S + sl) * m + r) * mp + c0) = w;
      }
    }
  }
}

// Column slices, transposed (right operands): exps[n] for column n, slice s
// element (n, k) = digit s of src[k][n] at ((q * S + s) m + n) pitch + k.  The
// group's 32 column maxima first (eight warps over the rows), then 32 x 32
// tiles through shared memory; a thread writes four consecutive k of one n
// per slice (8-byte stores).  256 threads.
template <int S>
__device__ __forceinline__ void slice_cols_group(const double* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                                                 long long qdst, int* __restrict__ exps, int m, int g,
                                                 Shift sh, int (*red)[32], int* s_e,
                                                 unsigned long long (*tile)[33]) {
  const int mp = slice_pitch(m);
  const unsigned long long* bits = reinterpret_cast<const unsigned long long*>(src);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = 32 * g + lane;
  int key = kNoKey;
  if (n < m)
    for (int k = warp; k < m; k += 8) key = max(key, scale_key((uint32_t)(bits[(long long)k * m + n] >> 32), sh(k)));
  red[warp][lane] = key;
  __syncthreads();
  if (warp == 0) {
#pragma unroll
    for (int w = 0; w < 8; ++w) key = max(key, red[w][lane]);
    const int e = key_exponent(key);
    s_e[lane] = e;
    if (n < m) exps[qdst * m + n] = e;
  }
  __syncthreads();
  const int nl = threadIdx.x >> 3, kq = (threadIdx.x & 7) * 4;
  for (int k0 = 0; k0 < m; k0 += 32) {
    int sk[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) sk[u] = sh(min(k0 + kq + u, m - 1));
    for (int y = warp; y < 32; y += 8) {
      const int k = k0 + y;
      tile[y][lane] = (k < m && n < m) ? bits[(long long)k * m + n] : 0ull;
    }
    __syncthreads();
    const int nn = 32 * g + nl, k = k0 + kq;
    if (nn < m && k < mp) {  // past m the tile holds zeros
      uint32_t q[4][S];
#pragma unroll
      for (int u = 0; u < 4; ++u) digits<S>(tile[kq + u][nl], s_e[nl] - sk[u], q[u]);
#pragma unroll
      for (int sl = 0; sl < S; ++sl) {
        uint2 w;
        w.x = (q[0][sl] >> 16) | (q[1][sl] & 0xffff0000u);
        w.y = (q[2][sl] >> 16) | (q[3][sl] & 0xffff0000u);
        *reinterpret_cast<uint2*>(dst + ((qdst * S + sl) * m + nn) * mp + k) = w;
      }
    }
    __syncthreads();
  }
}

// Slices of every block of a level's array (A as rows, its columns the
// unknowns of the block row before; C as transposed columns, its rows the
// block row's equations): blockIdx.x = block * groups + group, looping past the grid.
// With `band` set and the level's A and C banded (*band <= kBandMax), nothing
// is done: only the tensor-core tiles the banded kernels replace read these.
template <bool COLS, int S>
__global__ void __launch_bounds__(256) k_oz_slice_all(const double* __restrict__ src, int nblocks, int m,
                                                      __nv_bfloat16* __restrict__ dst, int* __restrict__ exps,
                                                      const int* __restrict__ bu, const int* __restrict__ be,
                                                      const int* __restrict__ band) {
  __shared__ int red[8][32], s_e[32];
  __shared__ unsigned long long tile[32][33];
  if (band && *band <= kBandMax) return;
  const long long mm = (long long)m * m;
  const int groups = (m + 31) / 32;
  for (long long i = blockIdx.x; i < (long long)nblocks * groups; i += gridDim.x) {
    const int q = (int)(i / groups), g = (int)(i - (long long)q * groups);
    if (COLS)
      slice_cols_group<S>(src + q * mm, dst, q, exps, m, g, Shift{be + (long long)q * m, -1}, red, s_e, tile);
    else  // the first block row has no unknowns before it
      slice_rows_group<S>(src + q * mm, dst, q, exps, m, g, Shift{bu + (long long)max(q - 1, 0) * m, q > 0 ? -1 : 0});
    __syncthreads();
  }
}

// Per-subsystem slicing jobs (k_oz_slice_jobs, blockIdx.x = subsystem), kind:
//   0 G_t rows -> rolling (q);            1 Acal_t rows -> all blocks (b0 + t);
//   2 Acal_t columns -> rolling (q);      3 ZL_t columns -> rolling slot (2q + t%2);
//   4 ZR_{L-1} columns (last row, right spike) -> slot;  5 Y_{t+1} columns -> rolling (q);
//   6 ZL_t columns, backward step;        7 ZR_t columns, backward step;
//   8 Y_0 = A_first columns -> rolling (q), at the start of a factorisation.
// Index k runs over the equations of block row t in G_t's columns and C_t's
// and Y_t's rows, over the unknowns of block row t in the columns of A_{t+1}
// and Acal_{t-1} and the rows of Acal_t, ZL_t, ZR_t.
// Several per-subsystem slicing jobs in one launch (blockIdx.y = job).
template <int S>
__global__ void __launch_bounds__(256) k_oz_slice_jobs(const PartDesc* __restrict__ parts, int step, int m,
                                                       OzSliceJobs jobs) {
  __shared__ int red[8][32], s_e[32];
  __shared__ unsigned long long tile[32][33];
  const OzSliceJob& jb = jobs.job[blockIdx.y];
  const int groups = (m + 31) / 32;
  const int q = blockIdx.x / groups, g = blockIdx.x - q * groups;
  const PartDesc p = parts[q];
  const long long mm = (long long)m * m;
  const bool hl = (p.flags & HAS_LEFT) != 0, hr = (p.flags & HAS_RIGHT) != 0;
  int t = step;
  bool act;
  long long sblk, dq;
  switch (jb.kind) {
    case 0: act = t < p.L; sblk = p.blk / mm + t; dq = q; break;
    case 1: act = t < p.L - 1; sblk = p.blk / mm + t; dq = p.blk / mm + t; break;
    case 2: act = t < p.L - 1; sblk = p.blk / mm + t; dq = q; break;
    case 3: act = t < p.L && hl; sblk = p.blk / mm + t; dq = 2 * q + (t & 1); break;
    case 4: act = t == p.L - 1 && hr; sblk = p.blk / mm + t; dq = 2 * q + (t & 1); break;
    case 5: act = t < p.L - 1 && hl; sblk = q; dq = q; break;
    case 6: t = p.L - 2 - step; act = t >= 0 && hl; sblk = p.blk / mm + t; dq = 2 * q + (t & 1); break;
    case 7: t = p.L - 2 - step; act = t >= 0 && hr; sblk = p.blk / mm + t; dq = 2 * q + (t & 1); break;
    default: act = hl; sblk = p.blk / mm; dq = q; break;
  }
  // launch B's right operands (Acal_t^T, ZL_t^T before the last row) are
  // not needed when its products run in the banded kernel
  if (jobs.band && *jobs.band <= kBandMax && (jb.kind == 2 || (jb.kind == 3 && t < p.L - 1))) act = false;
  if (!act) return;
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(jb.dst);
  const long long bt = p.blk / mm + t;  // the block row
  const Shift sh = jb.kind == 0   ? Shift{jobs.be + bt * m, 1}
                   : jb.kind == 1 ? Shift{jobs.bu + (bt + 1) * m, -1}
                   : jb.kind == 5 ? Shift{jobs.be + (bt + 1) * m, -1}
                   : jb.kind == 8 ? Shift{jobs.be + sblk * m, -1}
                                  : Shift{jobs.bu + bt * m, 1};
  if (jb.kind == 0 || jb.kind == 1)
    slice_rows_group<S>(jb.src + sblk * mm, dst, dq, jb.exps, m, g, sh);
  else
    slice_cols_group<S>(jb.src + sblk * mm, dst, dq, jb.exps, m, g, sh, red, s_e, tile);
}

// The assembly's operands per separator s (blockIdx.x = s * groups + group,
// blockIdx.y = job): job 0 C_q rows -> Cq slot s; jobs 1-4 the boundary
// spike blocks as columns -> S slot 4 s + job - 1: ZR^j[q-1], ZL^j[q-1] (only
// with HA), ZL^{j+1}[q+1], ZR^{j+1}[q+1] (only with HC).
template <int S>
__global__ void __launch_bounds__(256) k_oz_slice_seps(const SepDesc* __restrict__ seps, int m,
                                                       const double* __restrict__ C, const double* __restrict__ ZL,
                                                       const double* __restrict__ ZR, __nv_bfloat16* __restrict__ Cq,
                                                       int* __restrict__ eCq, __nv_bfloat16* __restrict__ Sp,
                                                       int* __restrict__ eS, const int* __restrict__ bu,
                                                       const int* __restrict__ band) {
  __shared__ int red[8][32], s_e[32];
  __shared__ unsigned long long tile[32][33];
  if (band && *band <= kBandMax) return;  // the banded assembly needs no slices
  const int groups = (m + 31) / 32;
  const int s = blockIdx.x / groups, g = blockIdx.x - s * groups, job = blockIdx.y;
  const SepDesc sd = seps[s];
  const long long mm = (long long)m * m;
  if (job == 0) {
    slice_rows_group<S>(C + sd.blk_q, Cq, s, eCq, m, g, Shift{bu + sd.blk_next / mm * m, -1});
    return;
  }
  if ((job == 2 && !(sd.flags & HAS_HA)) || (job == 4 && !(sd.flags & HAS_HC))) return;
  const double* src = job == 1 ? ZR + sd.blk_prev : job == 2 ? ZL + sd.blk_prev : job == 3 ? ZL + sd.blk_next
                                                                                         : ZR + sd.blk_next;
  slice_cols_group<S>(src, Sp, 4LL * s + job - 1, eS, m, g,
                      Shift{bu + (job <= 2 ? sd.blk_prev : sd.blk_next) / mm * m, 1}, red, s_e, tile);
}

// ---------------------------------------------------------------- banded operands
// When every A and C block of the level has its nonzeros within w <= kBandMax
// of the diagonal (detected by the input slicing), the products with A or C
// as an operand cost (2w + 1) multiply-adds per entry instead of m: these
// float64 kernels compute them over the band (the other terms are exact
// zeros), and the tensor-core tiles and slices for them are skipped.  A CTA
// takes 32 rows of one block (blockIdx.x = unit * groups + group); a warp a
// row at a time, a lane every 32nd column; the band of the banded operand in
// shared memory, the dense operand read along rows (coalesced).

// launch A's first product: X = G_t C_t (Acal_t, or the right spike ZR_{L-1})
__global__ void __launch_bounds__(256) k_band_gc(const PartDesc* __restrict__ parts, int t, int m,
                                                 const double* __restrict__ G, const double* __restrict__ C,
                                                 double* __restrict__ Acal, double* __restrict__ ZR,
                                                 const int* __restrict__ band) {
  extern __shared__ double bd[];  // bd[(d + w) m + n] = C[n + d][n]
  const int w = *band;
  if (w > kBandMax) return;
  const int groups = (m + 31) / 32;
  const int q = blockIdx.x / groups, g = blockIdx.x - q * groups;
  const PartDesc p = parts[q];
  if (t >= p.L || (t == p.L - 1 && !(p.flags & HAS_RIGHT))) return;
  const long long mm = (long long)m * m, o = p.blk + (long long)t * mm;
  const double* Gt = G + o;
  const double* Ct = C + o;
  double* X = (t < p.L - 1 ? Acal : ZR) + o;
  for (int i = threadIdx.x; i < (2 * w + 1) * m; i += blockDim.x) {
    const int dd = i / m, n = i - dd * m, k = n + dd - w;
    bd[i] = (k >= 0 && k < m) ? Ct[(long long)k * m + n] : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = 32 * g + warp; r < min(m, 32 * g + 32); r += 8)
    for (int n = lane; n < m; n += 32) {
      double acc = 0.0;
      for (int d = -w; d <= w; ++d) {
        const int k = n + d;
        if (k >= 0 && k < m) acc = fma(Gt[(long long)r * m + k], bd[(d + w) * m + n], acc);
      }
      X[(long long)r * m + n] = acc;
    }
}

// Row r of the banded left operand L times the dense X: sum_{k=r-w..r+w} L[r][k] X[k][n].
__device__ __forceinline__ double band_row(const double* lb, const double* __restrict__ X, int r, int n, int m,
                                           int w) {
  double acc = 0.0;
  for (int d = -w; d <= w; ++d) {
    const int k = r + d;
    if (k >= 0 && k < m) acc = fma(lb[d + w], X[(long long)k * m + n], acc);
  }
  return acc;
}

// The 32 rows' bands of L into lb[row][d + w] = L[r][r + d].
__device__ __forceinline__ void load_row_band(double (*lb)[2 * kBandMax + 1], const double* __restrict__ L, int g, int m,
                                              int w) {
  for (int i = threadIdx.x; i < 32 * (2 * w + 1); i += blockDim.x) {
    const int rl = i / (2 * w + 1), dd = i - rl * (2 * w + 1), r = 32 * g + rl, k = r + dd - w;
    lb[rl][dd] = (r < m && k >= 0 && k < m) ? L[(long long)r * m + k] : 0.0;
  }
}

// launch B: D_{t+1} = B_{t+1} - A_{t+1} Acal_t (blockIdx.y = 0) and
// Y_{t+1} = -A_{t+1} Bcal_t (= ZL_t, blockIdx.y = 1, with a left spike)
__global__ void __launch_bounds__(256) k_band_b(const PartDesc* __restrict__ parts, int t, int m,
                                                const double* __restrict__ A, const double* __restrict__ B,
                                                const double* __restrict__ Acal, const double* __restrict__ ZL,
                                                double* __restrict__ G, double* __restrict__ W,
                                                double* __restrict__ Y, const int* __restrict__ gam,
                                                const int* __restrict__ rho, const int* __restrict__ band) {
  __shared__ double lb[32][2 * kBandMax + 1];
  const int w = *band;
  if (w > kBandMax) return;
  const int groups = (m + 31) / 32;
  const int q = blockIdx.x / groups, g = blockIdx.x - q * groups, j = blockIdx.y;
  const PartDesc p = parts[q];
  if (t >= p.L - 1 || (j == 1 && !(p.flags & HAS_LEFT))) return;
  const long long mm = (long long)m * m, o = p.blk + (long long)t * mm;
  load_row_band(lb, A + o + mm, g, m, w);
  __syncthreads();
  const double* X = (j == 0 ? Acal : ZL) + o;
  double* D = W ? W + (long long)q * mm : G + o + mm;  // the inversion's working matrix, if there is one
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = 32 * g + warp; r < min(m, 32 * g + 32); r += 8)
    for (int n = lane; n < m; n += 32) {
      const double v = band_row(lb[r - 32 * g], X, r, n, m, w);
      const long long e = (long long)r * m + n;
      if (j == 0)  // D_{t+1}, equilibrated in the working matrix
        D[e] = W ? scale_pow2(B[o + mm + e] - v, -(rho[(o + mm) / m + r] + gam[(o + mm) / m + n])) : B[o + mm + e] - v;
      else
        Y[(long long)q * mm + e] = -v;      // Y_{t+1}
    }
}

// the supplementary blocks (Eq. e2311): blockIdx.y = 0: HB = B_q - A_q ZR^j[q-1]
// - C_q ZL^{j+1}[q+1]; 1: HA = -A_q ZL^j[q-1]; 2: HC = -C_q ZR^{j+1}[q+1]
__global__ void __launch_bounds__(256) k_band_h(const SepDesc* __restrict__ seps, int m, const double* __restrict__ A,
                                                const double* __restrict__ B, const double* __restrict__ C,
                                                const double* __restrict__ ZL, const double* __restrict__ ZR,
                                                double* __restrict__ HA, double* __restrict__ HB,
                                                double* __restrict__ HC, const int* __restrict__ band) {
  __shared__ double ab[32][2 * kBandMax + 1], cb[32][2 * kBandMax + 1];
  const int w = *band;
  if (w > kBandMax) return;
  const int groups = (m + 31) / 32;
  const int s = blockIdx.x / groups, g = blockIdx.x - s * groups, j = blockIdx.y;
  const SepDesc sd = seps[s];
  if ((j == 1 && !(sd.flags & HAS_HA)) || (j == 2 && !(sd.flags & HAS_HC))) return;
  if (j != 2) load_row_band(ab, A + sd.blk_q, g, m, w);
  if (j != 1) load_row_band(cb, C + sd.blk_q, g, m, w);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = 32 * g + warp; r < min(m, 32 * g + 32); r += 8)
    for (int n = lane; n < m; n += 32) {
      const int rl = r - 32 * g;
      const long long e = (long long)r * m + n;
      if (j == 0)
        HB[sd.hblk + e] = B[sd.blk_q + e] - (band_row(ab[rl], ZR + sd.blk_prev, r, n, m, w) +
                                             band_row(cb[rl], ZL + sd.blk_next, r, n, m, w));
      else if (j == 1)
        HA[sd.hblk + e] = -band_row(ab[rl], ZL + sd.blk_prev, r, n, m, w);
      else
        HC[sd.hblk + e] = -band_row(cb[rl], ZR + sd.blk_next, r, n, m, w);
    }
}

// ---------------------------------------------------------------- scales of equations and unknowns
// Exponents that equilibrate a level, estimated in two ways from the largest
// entries: per unknown of its column of [C_{i-1}; B_i; A_{i+1}] (gam), then per
// equation of its row of [A_i B_i C_i] with the columns so scaled (rho); and
// rows first, then columns.  The blocks are inverted with the first (partial
// pivoting, down the columns, does not see the columns' scales).  The products
// are balanced by the mean of both: where equations alone or unknowns alone
// are scaled one estimate is right, and for sparse blocks the other may be off
// by the whole range at the border of two fields of different scale.  Where
// they differ by more than 2^kAmbiguous inside a block row, or by more than
// 2^kDoubt where the largest entries spread over more than 2^kWide, the scales
// are not to be had from the largest entries, and the level keeps float64
// products (*uneven).  Relative errors, float64 / digits with columns first /
// with the mean (block Thomas in numpy, m = 64): dense, rows scaled over 12
// decades 1.1e-13 / 1.5e-14 / 5e-16; banded with a jump between the halves of
// the blocks of 2^40 5e-16 / 4e-6 / 1e-11 (estimates 2^42 apart), of 2^10 5e-16 /
// 3e-15 / 7e-16; Laplace blocks with equations and unknowns jumping oppositely
// by 2^20 9e-16 / 3e-14 / 3e-14 (2^7 apart, spread 2^18).  Blocks of one scale are
// 2^2 apart at most, dense blocks of condition 1e4 with graded singular vectors
// 2^8, spread over 2^11; digits serve those with smaller errors than float64
// products (6.5e-14 against 2.8e-13 at m = 128).  What stays on digits with an
// opposite jump of less than 2^13 has up to 40 times float64's error, at most
// 7e-14.  Two passes over the blocks, each bound by reading them.
constexpr int kAmbiguous = 11, kDoubt = 4, kWide = 13;
constexpr int kKeyBias = 4096;

// One pass over the blocks: blockIdx.x = block row, y = 0 A, 1 B, 2 C, z =
// `rpc` rows of it; a warp a row at a time, a lane every 32nd column (at most
// CPL).  First pass: the largest exponent of every row to rowkey and of every
// column to colkey ([block row][m], zeroed before; a column of A_i belongs to
// the unknowns of block row i - 1, one of C_i to those of i + 1), and the
// largest |row - column| of a nonzero entry (any bit but the sign set) of A
// and C to *band (if not null).  Second pass: the same with every entry
// divided by its column's (for the rows) or its row's (for the columns) first
// result, in rowkey2 and colkey2.
template <int CPL, bool SECOND>
__global__ void __launch_bounds__(256) k_level_scan(const SysDesc* __restrict__ sys, int nsys,
                                                    const double* __restrict__ A, const double* __restrict__ B,
                                                    const double* __restrict__ C, int m, int rpc, int* __restrict__ rowkey,
                                                    int* __restrict__ colkey, int* __restrict__ rowkey2,
                                                    int* __restrict__ colkey2, int* __restrict__ band) {
  __shared__ int cmax[8][32 * CPL], swid[8];
  const int b = blockIdx.x, part = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const SysDesc& sd = sys[find_sys(sys, nsys, b)];
  const int cb = b + part - 1;
  if (cb < sd.row0 || cb >= sd.row0 + sd.N) return;  // A_1, C_N
  const unsigned long long* M =
      reinterpret_cast<const unsigned long long*>(part == 0 ? A : part == 1 ? B : C) + (long long)b * m * m;
  int* rk = rowkey + (long long)b * m;
  int* ck = colkey + (long long)cb * m;
  int cm[CPL], cs[CPL], wid = 0;
#pragma unroll
  for (int q = 0; q < CPL; ++q) {
    cm[q] = 0;
    cs[q] = SECOND && lane + 32 * q < m ? kKeyBias - ck[lane + 32 * q] : 0;
  }
  const int rend = min(m, (int)(blockIdx.z + 1) * rpc);
#pragma unroll 2
  for (int r = blockIdx.z * rpc + warp; r < rend; r += 8) {
    unsigned long long v[CPL];
#pragma unroll
    for (int q = 0; q < CPL; ++q) v[q] = lane + 32 * q < m ? __ldg(M + (long long)r * m + lane + 32 * q) : 0ull;
    const int rs = SECOND ? kKeyBias - rk[r] : 0;
    int rm = 0;
#pragma unroll
    for (int q = 0; q < CPL; ++q) {
      const int h = (int)(v[q] >> 32) & 0x7fffffff, ex = max(h >> 20, 1);
      if (h != 0) {
        rm = max(rm, ex + cs[q]);
        cm[q] = max(cm[q], ex + rs);
      }
      if (!SECOND && (v[q] << 1) != 0) wid = max(wid, abs(r - lane - 32 * q));
    }
    rm = __reduce_max_sync(0xffffffffu, rm);
    if (lane == 0 && rm > 0) atomicMax((SECOND ? rowkey2 + (long long)b * m : rk) + r, rm);
  }
#pragma unroll
  for (int q = 0; q < CPL; ++q) cmax[warp][lane + 32 * q] = cm[q];
  wid = __reduce_max_sync(0xffffffffu, wid);
  if (lane == 0) swid[warp] = wid;
  __syncthreads();
  for (int c = threadIdx.x; c < m; c += 256) {
    int h = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) h = max(h, cmax[w][c]);
    if (h > 0) atomicMax((SECOND ? colkey2 + (long long)cb * m : ck) + c, h);
  }
  if (!SECOND && band && part != 1 && threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) wid = max(wid, swid[w]);
    if (wid > *(volatile int*)band) atomicMax(band, wid);
  }
}

// The exponents from the keys, in place, a warp per block row: rowkey2 -> rho,
// colkey -> gam, rowkey -> be (equations), colkey2 -> bu (unknowns).
__global__ void __launch_bounds__(256) k_level_exponents(int nblocks, int m, int* __restrict__ rowkey,
                                                         int* __restrict__ colkey, int* __restrict__ rowkey2,
                                                         int* __restrict__ colkey2, int* __restrict__ uneven) {
  const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (b >= nblocks) return;
  // the differences of the estimates and the estimates from all entries, of
  // the equations and the unknowns
  int lo[4] = {1 << 20, 1 << 20, 1 << 20, 1 << 20}, hi[4] = {-(1 << 20), -(1 << 20), -(1 << 20), -(1 << 20)};
  auto take = [&](int i, int v) { lo[i] = min(lo[i], v), hi[i] = max(hi[i], v); };
  for (int k = lane; k < m; k += 32) {
    const long long i = (long long)b * m + k;
    const bool row = rowkey[i] != 0, col = colkey[i] != 0;  // not all zeros
    const int rho2 = row ? rowkey[i] - 1022 : 0, gam = col ? colkey[i] - 1022 : 0;
    const int rho = row ? rowkey2[i] - kKeyBias : 0, gam2 = col ? colkey2[i] - kKeyBias : 0;
    if (row) take(0, rho - rho2), take(2, rho2);
    if (col) take(1, gam - gam2), take(3, gam);
    rowkey2[i] = rho;
    colkey[i] = gam;
    rowkey[i] = (rho + rho2) >> 1;
    colkey2[i] = (gam + gam2) >> 1;
  }
  int sp[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) sp[i] = __reduce_max_sync(0xffffffffu, hi[i]) - __reduce_min_sync(0xffffffffu, lo[i]);
  const int apart = max(sp[0], sp[1]), wide = max(sp[2], sp[3]);
  if (lane == 0 && (apart > kAmbiguous || (apart > kDoubt && wide > kWide))) *uneven = 1;
}

// The level's band: the largest |row - column| of a nonzero entry (any bit
// but the sign set) of the A and C blocks, folded into *band.  Read only.
__global__ void __launch_bounds__(256) k_band_detect(const double* __restrict__ A, const double* __restrict__ C,
                                                     long long n, int m, int* __restrict__ band) {
  const unsigned long long* a = reinterpret_cast<const unsigned long long*>(A);
  const unsigned long long* c = reinterpret_cast<const unsigned long long*>(C);
  int wmax = 0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    if (((a[e] | c[e]) << 1) != 0) {
      const int col = (int)(e % m), row = (int)((e / m) % m);
      wmax = max(wmax, abs(row - col));
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
  if ((threadIdx.x & 31) == 0 && wmax > 0) atomicMax(band, wmax);
}

}  // namespace oz

// ---------------------------------------------------------------- host side
namespace {
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                              const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn oz_encoder() {
  static EncodeFn enc = nullptr;
  if (!enc) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn) {
      cudaGetLastError();
      return nullptr;
    }
    enc = reinterpret_cast<EncodeFn>(fn);
  }
  return enc;
}
}  // namespace

// From m = 16 on (float64 pipe / sliced, factor + solve of N = 511: m = 8 1143
// / 1332 us, 12 1494 / 1675, 16 1851 / 1756, 24 2616 / 2058, 100 18.0 / 6.5 ms,
// 200 97 / 18 ms; N = 127, m = 400 221 / 44 ms, 512 327 / 62 ms).
bool oz_eligible(int m) { return m >= 16 && m <= kMaxM; }

int oz_slices(int m) { return m <= 128 ? 7 : 8; }

int oz_slice_blocks_bytes(int m) { return oz_slices(m) * m * slice_pitch(m) * 2; }

// 4-D map [block][slice][row][column] of a slice array (rows x kdim per
// slice, rows `pitch` elements apart; kdim = m for the sweeps' blocks, 32 for
// the inversion's panels),
// box 32 x box_rows x slices x 1.
bool oz_make_map(const void* base, long long blocks, int m, int box_rows, void* out, int kdim) {
  EncodeFn enc = oz_encoder();
  if (kdim <= 0) kdim = m;
  const int S = oz_slices(kdim), pitch = slice_pitch(kdim);
  if (!enc || blocks <= 0 || !oz_eligible(m)) return false;
  cuuint64_t dims[4] = {(cuuint64_t)kdim, (cuuint64_t)m, (cuuint64_t)S, (cuuint64_t)blocks};
  cuuint64_t strides[3] = {(cuuint64_t)pitch * 2, (cuuint64_t)m * pitch * 2, (cuuint64_t)S * m * pitch * 2};
  cuuint32_t box[4] = {(cuuint32_t)oz::KS, (cuuint32_t)box_rows, (cuuint32_t)S, 1u};
  cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  CUresult r = enc(static_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims,
                   strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

int oz_box_rows_left() { return oz::MT; }
int oz_box_rows_right(int m) { return oz::nt_of(0, oz_slices(m)); }
int oz_box_rows_gj() { return oz::NT3; }

void launch_band_detect(const double* A, const double* C, long long n, int m, int* band, cudaStream_t st) {
  if (n <= 0 || !band) return;
  oz::k_band_detect<<<152 * 8, 256, 0, st>>>(A, C, n, m, band);
}

void launch_level_scales(const SysDesc* sys, int nsys, const double* A, const double* B, const double* C, int nblocks,
                         int m, const OzScales& sc, int* uneven, int* band, cudaStream_t st) {
  if (nblocks <= 0) return;
  cudaMemsetAsync(sc.be, 0, 4 * (size_t)nblocks * m * sizeof(int), st);
  const int rpc = 3 * nblocks >= 304 ? m : 32;  // a few blocks: more CTAs each
  const dim3 grid(nblocks, 3, (m + rpc - 1) / rpc);
  auto pass = [&](auto second) {
    constexpr bool S2 = decltype(second)::value;
#define DM_SCAN(CPL_) oz::k_level_scan<CPL_, S2><<<grid, 256, 0, st>>>(sys, nsys, A, B, C, m, rpc, sc.be, sc.gam, sc.rho, sc.bu, band)
    if (m <= 64) DM_SCAN(2);
    else if (m <= 128) DM_SCAN(4);
    else if (m <= 256) DM_SCAN(8);
    else DM_SCAN(16);
#undef DM_SCAN
  };
  pass(std::false_type());
  pass(std::true_type());
  oz::k_level_exponents<<<(nblocks + 7) / 8, 256, 0, st>>>(nblocks, m, sc.be, sc.gam, sc.rho, sc.bu, uneven);
}

void launch_oz_slice_all(bool cols, const double* src, int nblocks, int m, void* dst, int* exps, const OzScales& sc,
                         const int* band, cudaStream_t st) {
  if (nblocks <= 0) return;
  const long long work = (long long)nblocks * ((m + 31) / 32);
  const int grid = (int)std::min<long long>(work, 152LL * 16);
  auto* d = static_cast<__nv_bfloat16*>(dst);
  const bool s7 = oz_slices(m) == 7;
  if (cols && s7) oz::k_oz_slice_all<true, 7><<<grid, 256, 0, st>>>(src, nblocks, m, d, exps, sc.bu, sc.be, band);
  else if (cols) oz::k_oz_slice_all<true, 8><<<grid, 256, 0, st>>>(src, nblocks, m, d, exps, sc.bu, sc.be, band);
  else if (s7) oz::k_oz_slice_all<false, 7><<<grid, 256, 0, st>>>(src, nblocks, m, d, exps, sc.bu, sc.be, band);
  else oz::k_oz_slice_all<false, 8><<<grid, 256, 0, st>>>(src, nblocks, m, d, exps, sc.bu, sc.be, band);
}

void launch_oz_slice_jobs(const PartDesc* parts, int nparts, int step, int m, const OzSliceJobs& jobs, int njobs,
                          cudaStream_t st) {
  if (nparts <= 0 || njobs <= 0) return;
  const dim3 grid(nparts * ((m + 31) / 32), njobs);
  if (oz_slices(m) == 7)
    oz::k_oz_slice_jobs<7><<<grid, 256, 0, st>>>(parts, step, m, jobs);
  else
    oz::k_oz_slice_jobs<8><<<grid, 256, 0, st>>>(parts, step, m, jobs);
}

// The trailing update of one panel of the blocked inversion (dm_gj.cu).
void launch_gj_update(const PartDesc* parts, int nparts, int t, int m, int pnl, double* W, const int* piv,
                      const int* Uexp, const int* Vexp, const void* maps2, int* errflag, cudaStream_t st) {
  if (nparts <= 0) return;
  OzOut out{};
  out.W = W;
  out.piv = piv;
  unsigned char maps3[3 * 128];
  std::memcpy(maps3, maps2, 2 * 128);
  std::memcpy(maps3 + 2 * 128, static_cast<const unsigned char*>(maps2) + 128, 128);
  launch_oz_step(3, parts, nparts, pnl, m, out, Uexp, Vexp, Vexp, maps3, errflag, st, t);
}

void launch_oz_step(int kind, const PartDesc* parts, int nparts, int step, int m, const OzOut& out, const int* lexp,
                    const int* rexp0, const int* rexp1, const void* maps3, int* errflag, cudaStream_t st, int aux) {
  if (nparts <= 0) return;
  OzMaps mp;
  std::memcpy(&mp, maps3, sizeof mp);
  static int nsm = 0;
  if (!nsm) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0) nsm = 1;
  }
  // KIND 3: 32-column tiles without the one that is the panel itself
  const int ntm = (m + oz::MT - 1) / oz::MT,
            ntn = kind == 3 ? (m + oz::NT3 - 1) / oz::NT3 - 1 : (m + oz_box_rows_right(m) - 1) / oz_box_rows_right(m);
  const int ntiles = nparts * (kind == 3 ? 1 : 2) * ntm * ntn;
  if (ntiles <= 0) return;
  const int grid = std::min(ntiles, nsm);
#define DM_OZ(KIND_, S_)                                                                                          \
  do {                                                                                                            \
    constexpr int smem = oz::smem_bytes<KIND_, S_>();                                                             \
    allow_smem(oz::k_oz_step<KIND_, S_>, smem);                                                                   \
    oz::k_oz_step<KIND_, S_><<<grid, oz::threads_of(KIND_, S_), smem, st>>>(parts, step, aux, m, ntm, ntn, ntiles, out, lexp,  \
                                                               rexp0, rexp1, errflag, mp);                        \
  } while (0)
  const bool s7 = oz_slices(m) == 7;
  if (kind == 3) DM_OZ(3, 7);  // K = 32
  else if (kind == 0 && s7) DM_OZ(0, 7);
  else if (kind == 0) DM_OZ(0, 8);
  else if (kind == 1 && s7) DM_OZ(1, 7);
  else if (kind == 1) DM_OZ(1, 8);
  else if (kind == 2 && s7) DM_OZ(2, 7);
  else if (kind == 2) DM_OZ(2, 8);
  else if (kind == 4 && s7) DM_OZ(4, 7);
  else if (kind == 4) DM_OZ(4, 8);
  else if (s7) DM_OZ(5, 7);
  else DM_OZ(5, 8);
#undef DM_OZ
}

void launch_oz_assemble(const SepDesc* seps, int nseps, int m, const double* B, const double* C, const double* ZL,
                        const double* ZR, double* HA, double* HB, double* HC, const OzAsm& a, const int* eA,
                        const void* mapA, int* errflag, const int* bu, const int* band, cudaStream_t st) {
  if (nseps <= 0) return;
  const dim3 sgrid(nseps * ((m + 31) / 32), 5);
  auto *cq = static_cast<__nv_bfloat16*>(a.Cq), *sp = static_cast<__nv_bfloat16*>(a.S);
  if (oz_slices(m) == 7)
    oz::k_oz_slice_seps<7><<<sgrid, 256, 0, st>>>(seps, m, C, ZL, ZR, cq, a.eCq, sp, a.eS, bu, band);
  else
    oz::k_oz_slice_seps<8><<<sgrid, 256, 0, st>>>(seps, m, C, ZL, ZR, cq, a.eCq, sp, a.eS, bu, band);
  OzOut out{};
  out.B = B;
  out.seps = seps;
  out.HA = HA;
  out.HB = HB;
  out.HC = HC;
  out.band = band;
  unsigned char maps3[3 * 128];
  std::memcpy(maps3, mapA, 128);
  std::memcpy(maps3 + 128, a.maps[1], 128);
  std::memcpy(maps3 + 256, a.maps[1], 128);
  launch_oz_step(4, nullptr, nseps, 0, m, out, eA, a.eS, a.eS, maps3, errflag, st);
  std::memcpy(maps3, a.maps[0], 128);
  launch_oz_step(5, nullptr, nseps, 0, m, out, a.eCq, a.eS, a.eS, maps3, errflag, st);
}

void launch_band_gc(const PartDesc* parts, int nparts, int t, int m, const double* G, const double* C, double* Acal,
                    double* ZR, const int* band, cudaStream_t st) {
  if (nparts <= 0 || !band) return;
  allow_smem(oz::k_band_gc, (2 * kBandMax + 1) * m * sizeof(double));
  oz::k_band_gc<<<nparts * ((m + 31) / 32), 256, (2 * kBandMax + 1) * m * sizeof(double), st>>>(parts, t, m, G, C, Acal, ZR, band);
}

void launch_band_b(const PartDesc* parts, int nparts, int t, int m, const double* A, const double* B,
                   const double* Acal, const double* ZL, double* G, double* W, double* Y, const int* gam,
                   const int* rho, const int* band, cudaStream_t st) {
  if (nparts <= 0 || !band) return;
  oz::k_band_b<<<dim3(nparts * ((m + 31) / 32), 2), 256, 0, st>>>(parts, t, m, A, B, Acal, ZL, G, W, Y, gam, rho, band);
}

void launch_band_h(const SepDesc* seps, int nseps, int m, const double* A, const double* B, const double* C,
                   const double* ZL, const double* ZR, double* HA, double* HB, double* HC, const int* band,
                   cudaStream_t st) {
  if (nseps <= 0 || !band) return;
  oz::k_band_h<<<dim3(nseps * ((m + 31) / 32), 3), 256, 0, st>>>(seps, m, A, B, C, ZL, ZR, HA, HB, HC, band);
}

}  // namespace dm
