// romp_refine.cu -- per-patch steps of the FP16 path between scoring passes:
// candidate certification, exact re-scoring, the least-squares update and the
// residual (steps (c)-(e) of OMP, Sec. II-C).
//
// romp_init_kernel writes each patch's packed residual (= x) in fp16 for the
// first scoring pass and initialises its state.  Rows are scaled by a power
// of two chosen from a bound on their norm (rsc_internal.h), so that scores
// come back as 2^(16 - e) times their true value.  romp_refine_kernel then,
// after every scoring pass (romp_score.cu):
//   * certifies the scoring pass's candidates (per column slice: kept blocks
//     of 32 rows and a mask of columns): E bounds the fp16 error of a score
//     (rounding of both operands, accumulation, and the FP32 residual's own
//     error); every row with |score| >= s1 - 2E is row b + u of a kept block
//     b and a masked column u, unless a slice's bound on what it left out
//     (disc) is >= s1 - 2E, in which case the patch is handed to the FP32
//     path;
//   * re-scores those rows exactly in double-float as
//     <A_c, x> - sum_i a_i <A_c, A_i> (ties: smallest m*R + r);
//   * adds the Cholesky row of the winner (Gram entries and right-hand side
//     in double-float, factor and solve in FP64) and writes the new residual
//     row; after the last step the reported residual norm comes from the
//     factor instead (||x||^2 - z^T z, L z = b).
// Per-patch state lives in HBM as structure-of-arrays (coalesced over
// threads); stopped and finished patches write their outputs.
//
// One warp works on 32 patches.  What is scalar per patch (candidates, Gram
// entries, the FP64 factor) runs one thread per patch; what runs over a
// patch's row (the exact inner product with x, the new residual) runs one
// warp per row, kBatch rows at a time, its lanes over the row's slots, with
// the steered atoms read from the dictionary's tables (one 16-byte load per
// lane and term).  A thread walking its own patch's row and its own atoms'
// rows instead touches 32 cache lines per warp load; at 10^6 patches of
// 432 bytes, M = R = 64, K = 5, that kept the L1 tag stage busy for
// 1.06 ms per step (10,000 cycles per warp and step, DRAM at 16%), while
// these loads touch the 4 lines of one row.
#include <algorithm>

#include "rsc_internal.h"
#include "tc_common.cuh"

namespace {

enum : int { kPlain = 0, kPaired = 1, kLong = 2 };

// State arrays of P patches and K steps (element of patch p at field * P + p).
// The factor grows by one row per step: L row t (packed lower triangle), its
// inverse diagonal and z entry are written once, the weights at every step.
struct StateIdx {
  int dL, dInv, dZ, dA, nD;        // doubles
  int fHi, fLo, fX, fR, fX2h, fX2l, nF;  // weights in double-float, ||x||, ||r||, ||x||^2
  int iM, iR, iT, iE, nI;          // atoms, angles, steps of a handed-over patch, row exponent
  __host__ __device__ explicit StateIdx(int K)
      : dL(0), dInv(K * (K + 1) / 2), dZ(dInv + K), dA(dZ + K), nD(dA + K),
        fHi(0), fLo(K), fX(2 * K), fR(2 * K + 1), fX2h(2 * K + 2), fX2l(2 * K + 3), nF(2 * K + 4),
        iM(0), iR(K), iT(2 * K), iE(2 * K + 1), nI(2 * K + 2) {}
};

// The slots a lane owns of a packed row: slots 4 lane .. + 3, and for rows of
// 256 slots 128 + 4 lane .. + 3 too.
template <int LAY>
struct LaneSlots {
  static constexpr int NQ = LAY == kLong ? 2 : 1;
  int off[4 * NQ];    // float index into the patch's half spectrum, -1: zero slot
  float wk[4 * NQ];   // weight of the slot in the inner product: 1 (k = 0) or 2
  unsigned odd;       // slots of odd harmonics
  bool in;            // the lane's slots are inside the row
  __device__ LaneSlots(int lane, int J, int kmax) {
    odd = 0;
    in = LAY == kLong || 4 * lane < kTcKst;
#pragma unroll
    for (int u = 0; u < 4 * NQ; ++u) {
      const int q = (u >> 2) * 128 + 4 * lane + (u & 3);
      const int code = in ? rsc_slot_code(q, J, kmax, LAY == kPaired) : -1;
      off[u] = code < 0 ? -1 : 2 * (code >> 8) + (code & 1);
      const int k = (code >> 1) & 127;
      wk[u] = code >= 0 && k ? 2.0f : 1.0f;
      if (code >= 0 && (k & 1)) odd |= 1u << u;
    }
  }
  __device__ __forceinline__ void load_x(const float *__restrict__ xp, float (&v)[4 * NQ]) const {
#pragma unroll
    for (int u = 0; u < 4 * NQ; ++u) v[u] = off[u] >= 0 ? __ldg(xp + off[u]) : 0.0f;
  }
  // slots of this lane of table row `row` (rows of L floats)
  __device__ __forceinline__ void load_row(const float *__restrict__ tab, int row, int lane,
                                           float (&v)[4 * NQ]) const {
    constexpr int L = LAY == kLong ? kTcKstLong : kTcKst;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in) t = __ldg(reinterpret_cast<const float4 *>(tab + (size_t)row * L) + 32 * q + lane);
      v[4 * q] = t.x;
      v[4 * q + 1] = t.y;
      v[4 * q + 2] = t.z;
      v[4 * q + 3] = t.w;
    }
  }
};

__device__ __forceinline__ df shfl_df(df v, int src) {
  return {__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}

// Sum kept as a value and the sum of its rounding errors (Dot2, Ogita, Rump,
// Oishi).
__device__ __forceinline__ df pair_add(df a, df b) {
  const df s = two_sum(a.hi, b.hi);
  return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}

// Sums of v[0 .. B) over the lanes (B = 2 or 4): afterwards lane l holds the
// sum of v[l mod B], over all 32 lanes or (HALF) over its half of the warp.
// The first log2(B) exchanges halve the values a lane still carries.
template <int B, bool HALF>
__device__ __forceinline__ df batch_sum(const df (&v)[B], int lane) {
  static_assert(B == 2 || B == 4, "batch of two or four rows");
  df z;
  if constexpr (B == 4) {
    df w[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const df mine = (lane & 1) ? v[2 * h + 1] : v[2 * h];
      const df give = (lane & 1) ? v[2 * h] : v[2 * h + 1];
      w[h] = pair_add(mine, df_shfl_xor(give, 1));
    }
    const df mine = (lane & 2) ? w[1] : w[0];
    const df give = (lane & 2) ? w[0] : w[1];
    z = pair_add(mine, df_shfl_xor(give, 2));
  } else {
    const df mine = (lane & 1) ? v[1] : v[0];
    const df give = (lane & 1) ? v[0] : v[1];
    z = pair_add(mine, df_shfl_xor(give, 1));
    z = pair_add(z, df_shfl_xor(z, 2));
  }
  z = pair_add(z, df_shfl_xor(z, 4));
  z = pair_add(z, df_shfl_xor(z, 8));
  if constexpr (!HALF) z = pair_add(z, df_shfl_xor(z, 16));
  return z;
}

template <int B>
__device__ __forceinline__ float batch_sum_f(const float (&v)[B], int lane) {
  float z;
  if constexpr (B == 4) {
    float w[2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      w[h] = ((lane & 1) ? v[2 * h + 1] : v[2 * h]) +
             __shfl_xor_sync(0xffffffffu, (lane & 1) ? v[2 * h] : v[2 * h + 1], 1);
    z = ((lane & 2) ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? w[0] : w[1], 2);
  } else {
    z = ((lane & 1) ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, (lane & 1) ? v[0] : v[1], 1);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
  }
  z += __shfl_xor_sync(0xffffffffu, z, 4);
  z += __shfl_xor_sync(0xffffffffu, z, 8);
  z += __shfl_xor_sync(0xffffffffu, z, 16);
  return z;
}

// The next up to B set lanes of `todo` (removed from it); a short batch
// repeats its first lane.  slot = this lane's place in the batch, or -1.
template <int B>
__device__ __forceinline__ void next_batch(unsigned &todo, int lane, int (&src)[B], int &slot) {
  slot = -1;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    if (todo) {
      src[j] = __ffs(todo) - 1;
      todo &= todo - 1;
      if (lane == src[j]) slot = j;
    } else {
      src[j] = src[0];
    }
  }
}

// This lane's slots of a packed row: v (raw entries) times sqrt(2) for k >= 1
// and `scale`, rounded to fp16; returns the sum of squares of the unscaled
// packed values.
template <int LAY>
__device__ __forceinline__ float store_row(const LaneSlots<LAY> &ls, unsigned char *A, int64_t p,
                                           int lane, float scale, float (&v)[4 * LaneSlots<LAY>::NQ]) {
  constexpr int L = LAY == kLong ? kTcKstLong : kTcKst;
  float n2 = 0.0f;
#pragma unroll
  for (int q = 0; q < LaneSlots<LAY>::NQ; ++q) {
#pragma unroll
    for (int u = 4 * q; u < 4 * q + 4; ++u) {
      if (ls.wk[u] == 2.0f) v[u] *= 1.41421356237309515f;
      n2 = fmaf(v[u], v[u], n2);
    }
    __half2 b0 = __floats2half2_rn(v[4 * q] * scale, v[4 * q + 1] * scale);
    __half2 b1 = __floats2half2_rn(v[4 * q + 2] * scale, v[4 * q + 3] * scale);
    uint2 pk;
    pk.x = *reinterpret_cast<uint32_t *>(&b0);
    pk.y = *reinterpret_cast<uint32_t *>(&b1);
    if (ls.in) reinterpret_cast<uint2 *>(A + p * (int64_t)(2 * L))[32 * q + lane] = pk;
  }
  return n2;
}

__device__ __forceinline__ void write_none(const RefineArgs &a, int64_t p, int from) {
  for (int i = from; i < a.K; ++i) {
    const int64_t o = p * a.K + i;
    a.atom[o] = -1;
    a.angle_idx[o] = -1;
    if (a.angle) a.angle[o] = 0.0f;
    a.coef[o] = 0.0;
  }
}

__device__ __forceinline__ void write_code(const RefineArgs &a, int64_t p, int i, int m, int r,
                                           double w) {
  const int64_t o = p * a.K + i;
  a.atom[o] = m;
  a.angle_idx[o] = r;
  if (a.angle) a.angle[o] = (float)(6.283185307179586 * r / a.R);
  a.coef[o] = w;
}

// Error bound of one fp16 score of a row of L slots, times 1.25, without the
// key term: 2^-10 ||r|| (both operands rounded, unit atoms) + 2^-18 ||r||
// (second order) + L 2^-21 ||r|| (the accumulation, at 4x unit roundoff) +
// s 2^-33 ||r|| and s 2^(e-33) (subnormal rounding of a dictionary entry,
// <= 2^-25 / kDictScale, and of a row entry, <= 2^-25 / row scale, over
// sqrt(L) <= s entries: s = 11 for 112 slots, 16 for 256); plus the FP32
// residual's own error 2 dr.
__device__ __forceinline__ float score_err_base(float rnorm, float dr, int e, int L) {
  const float sq = L <= kTcKst ? 11.0f : 16.0f;
  return 1.25f * (9.765625e-4f + 3.814697265625e-6f + (float)L * 4.76837158203125e-7f +
                  sq * 1.16415321826934814e-10f) *
             rnorm +
         1.25f * sq * ldexpf(1.0f, e - 33) + 2.0f * dr;
}

// The scoring pass's window for a row: 2.02 E in accumulator units
// (2^(16 - e) times true scores), with the key term 2^-16 s1 bounded through
// s1 <= 1.01 ||r|| (Cauchy-Schwarz over unit atoms plus the score error).
__device__ __forceinline__ float score_window(float rnorm, float dr, int e, int L) {
  return 2.02f * (score_err_base(rnorm, dr, e, L) + 1.52587890625e-5f * 1.01f * rnorm) *
         ldexpf(1.0f, 16 - e);
}

// Bound on the error of the FP32 residual after t steps with weights whose
// moduli sum to asum (t = 0: x itself).
__device__ __forceinline__ float residual_err(int t, float xnorm, float asum) {
  return t == 0 ? 2.0f * kU32 * xnorm : 2.0f * (t + 6) * kU32 * (xnorm + 1.5f * asum);
}

template <int LAY>
struct Batch {  // rows a warp has in flight: registers for B rows of 4 or 8 slots
  static constexpr int B = LAY == kLong ? 2 : 4;
};

template <int LAY>
__global__ void __launch_bounds__(128) romp_init_kernel(const RefineArgs a) {
  constexpr int NS = 4 * LaneSlots<LAY>::NQ, B = Batch<LAY>::B;
  const StateIdx I(a.K);
  const int lane = threadIdx.x & 31, vec = 2 * a.H * a.J;
  const LaneSlots<LAY> ls(lane, a.J, a.kmax);
  const int64_t P = a.P, step = (int64_t)gridDim.x * (blockDim.x >> 5) * a.warp_patches;
  for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * a.warp_patches;
       base < P; base += step) {
    const int64_t p = base + lane;
    float xnorm = 0.0f, n2 = 0.0f;
    df x2 = df_make(0.0f);
    int e = 0;
    const bool mine = lane < a.warp_patches && p < P;
    unsigned todo = __ballot_sync(0xffffffffu, mine);
    while (todo) {
      int src[B], slot;
      next_batch<B>(todo, lane, src, slot);
      float v[B][NS];
#pragma unroll
      for (int j = 0; j < B; ++j) ls.load_x(a.x + (base + src[j]) * vec, v[j]);
      df s[B];
#pragma unroll
      for (int j = 0; j < B; ++j) {
        s[j] = df_make(0.0f);
#pragma unroll
        for (int u = 0; u < NS; ++u) dot2_acc(s[j].hi, s[j].lo, v[j][u], ls.wk[u] * v[j][u]);
      }
      df z = batch_sum<B, false>(s, lane);
      z = fast_two_sum(z.hi, z.lo);  // lane l: the sum of row l mod B
      const float xn = sqrtf(fmaxf(z.hi + z.lo, 0.0f));
      const int ez = rsc_row_exponent(xn);
      float m2[B];
#pragma unroll
      for (int j = 0; j < B; ++j) {
        const int ej = __shfl_sync(0xffffffffu, ez, j);
        m2[j] = store_row<LAY>(ls, a.A, base + src[j], lane, ldexpf(1.0f, kRowLog2 - ej), v[j]);
      }
      const float q2 = batch_sum_f<B>(m2, lane);
      const int from = slot < 0 ? 0 : slot;
      const df zx = shfl_df(z, from);
      const float xr = __shfl_sync(0xffffffffu, xn, from), qr = __shfl_sync(0xffffffffu, q2, from);
      const int er = __shfl_sync(0xffffffffu, ez, from);
      if (slot >= 0) {
        x2 = zx;
        xnorm = xr;
        n2 = qr;
        e = er;
      }
    }
    if (mine) {
      const float rn = sqrtf(n2), dr = residual_err(0, xnorm, 0.0f);
      a.sI[I.iE * P + p] = e;
      a.sF[I.fX * P + p] = xnorm;
      a.sF[I.fX2h * P + p] = x2.hi;
      a.sF[I.fX2l * P + p] = x2.lo;
      a.sF[I.fR * P + p] = rn;
      a.win[p] = score_window(rn, dr, e, a.L);
      a.status[p] = 1;
    }
  }
}

// Step T of every patch still being coded (each has T atoms: a patch that adds
// none stops), compile-time so that the factor's loops unroll.
//
// 10^6 patches, M = R = 64, K = 5: 0.69 ms per step on average (0.62 / 0.81 /
// 0.98 at T = 1 / 2 / 3) against 1.06 for a thread per patch; the call 9.00 ->
// 7.29 ms, 1,000 patches at M = 16 261 -> 129 us (one kernel per step, not a
// memset and two passes; 81 with fewer patches a warp, see the launch), the
// 21 x 21 image sizes 21.8 -> 16.3 ms.  Issue is at 50%, so both instructions
// (12,000 to 17,000 per warp) and the loads' latency count.  Registers: at most 128 (4 blocks an SM) 3.79 ms per call of
// init and refines; without a cap (up to 255) 4.24, 5 or 6 blocks 3.96 / 3.91
// (spills).
template <int T, int LAY>
__global__ void __launch_bounds__(128, 4) romp_refine_kernel(const RefineArgs a) {
  constexpr int NS = 4 * LaneSlots<LAY>::NQ, B = Batch<LAY>::B;
  constexpr int TA = T > 0 ? T : 1;
  constexpr bool PAIRED = LAY == kPaired;
  constexpr int NP = PAIRED ? 2 : 1;
  const StateIdx I(a.K);
  const int lane = threadIdx.x & 31, vec = 2 * a.H * a.J;
  const int R = a.R, M = a.M, Rr = a.Rr;
  const LaneSlots<LAY> ls(lane, a.J, a.kmax);
  const TwS tw{a.tw, a.H, R};  // only for Gram entries without a table
  const int64_t P = a.P, step = (int64_t)gridDim.x * (blockDim.x >> 5) * a.warp_patches;
  for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * a.warp_patches;
       base < P; base += step) {
    const int64_t p = base + lane;
    const bool act = lane < a.warp_patches && p < P && a.status[p] > 0;
    if (!__any_sync(0xffffffffu, act)) continue;
    Ls<T + 1> S;
    int e = 0;
    float xnorm = 0.0f, rnorm = 0.0f;
    float thr = 0.0f, stop_level = 0.0f, unscale = 0.0f;
    int outcome = 0;  // 0 continue, 1 finished/stopped, 2 hand-off
    unsigned bmask = 0;
    int qf = -1, uf = 0;
    unsigned umk[kTcSplit] = {};
    if (act) {
      e = a.sI[I.iE * P + p];
      xnorm = a.sF[I.fX * P + p];
      rnorm = a.sF[I.fR * P + p];
      float asum = 0.0f;
#pragma unroll
      for (int i = 0; i < T; ++i) {
        S.ahi[i] = a.sF[(I.fHi + i) * P + p];
        S.alo[i] = a.sF[(I.fLo + i) * P + p];
        S.m[i] = a.sI[(I.iM + i) * P + p];
        S.r[i] = a.sI[(I.iR + i) * P + p];
        asum += fabsf(S.ahi[i]);
      }
      const float dr = residual_err(T, xnorm, asum);
      // accumulator scores are 2^(16 - e) times the true scores
      unscale = ldexpf(1.0f, e - 16);
      // the scoring pass's lists of kept blocks (one per column slice of each
      // chunk, each sorted by block maximum in descending order)
      static_assert(kTcTop == 4, "slots read as float4 / int4 per slice");
      const float *cvp = a.cand_val + p * kTcCand;
      const int *cip = a.cand_idx + p * kTcCand;
      float vv[kTcCand], discm = -INFINITY, head = -INFINITY;
      int iv[kTcCand];
      unsigned ubk[kTcSplit];
#pragma unroll
      for (int sl = 0; sl < kTcSplit; ++sl) {
        const float4 v4 = *reinterpret_cast<const float4 *>(cvp + kTcTop * sl);
        const int4 i4 = *reinterpret_cast<const int4 *>(cip + kTcTop * sl);
        const uint2 mk = *reinterpret_cast<const uint2 *>(a.cand_mask + 2 * (kTcSplit * p + sl));
        vv[kTcTop * sl] = v4.x;
        vv[kTcTop * sl + 1] = v4.y;
        vv[kTcTop * sl + 2] = v4.z;
        vv[kTcTop * sl + 3] = v4.w;
        iv[kTcTop * sl] = i4.x;
        iv[kTcTop * sl + 1] = i4.y;
        iv[kTcTop * sl + 2] = i4.z;
        iv[kTcTop * sl + 3] = i4.w;
        umk[sl] = mk.x;
        ubk[sl] = mk.y;
        discm = fmaxf(discm, a.cand_disc[kTcSplit * p + sl]);
        head = fmaxf(head, v4.x);
      }
      const float disc = discm * unscale, s1 = head * unscale;
      stop_level = 1e-10f * xnorm;
      // fp16 error of a score (score_err_base) plus a spare 2^-16 s1
      const float E = score_err_base(rnorm, dr, e, a.L) + 1.52587890625e-5f * fabsf(s1);
      if (!(s1 + E > stop_level)) {
        outcome = 1;
      } else {
        thr = s1 - 2.0f * E;
        if (disc >= thr) {
          outcome = 2;
        } else {
          // the kept blocks inside the window as a bit mask (slot q = slice
          // q / kTcTop); the block with the largest maximum and its slice's
          // best column come first
          float vbest = -1.0f;
#pragma unroll
          for (int q = 0; q < kTcCand; ++q)
            if (iv[q] >= 0 && vv[q] * unscale >= thr) {
              bmask |= 1u << q;
              if (vv[q] > vbest) {
                vbest = vv[q];
                qf = q;
              }
            }
          // (the best column is masked, so that candidates left undefined by
          // a scoring pass that gave up cannot name a row outside the table)
          unsigned ub = ubk[0];
#pragma unroll
          for (int sl = 1; sl < kTcSplit; ++sl) ub = qf / kTcTop == sl ? ubk[sl] : ub;
          uf = (int)(ub & 31u);
        }
      }
    }
    // a patch of zeros (a blank window) has nothing to code.  Its scores are all
    // 0 and all inside the window: a small dictionary's were all re-scored, a
    // large one's patch was handed off (100,000 blank patches at M = R = 16:
    // 2.66 ms, 0.12 now; with a thread per patch it was 0.70)
    if constexpr (T == 0) {
      unsigned todo = __ballot_sync(0xffffffffu, act && xnorm == 0.0f);
      while (todo) {
        int src[B], slot;
        next_batch<B>(todo, lane, src, slot);
        unsigned some[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
          float v[NS];
          ls.load_x(a.x + (base + src[j]) * vec, v);
          some[j] = 0;
#pragma unroll
          for (int u = 0; u < NS; ++u) some[j] |= v[u] != 0.0f;
        }
#pragma unroll
        for (int j = 0; j < B; ++j)
          if (!__any_sync(0xffffffffu, some[j]) && slot == j) {
            outcome = 1;
            qf = -1;
          }
      }
    }
    auto umask_of = [&](int sl) {
      unsigned r = umk[0];
#pragma unroll
      for (int i = 1; i < kTcSplit; ++i) r = sl == i ? umk[i] : r;
      return r;
    };
    // A candidate unit is one steered atom (row r*M + m), or in the paired
    // layout the two angles r and r + R/2 of atom m (row r*M + m, r < R/2,
    // scored by max(|s(r)|, |s(r + R/2)|)).  Every unit in the certified
    // window is row b + u of a kept block b (slot q) whose maximum reaches
    // the window and a column u in its slice's class mask.  A round of the
    // loop re-scores one unit of every lane that still has one (c1: 89% of
    // the patches have one unit, so rounds after the first hold a few lanes).
    const int Rh = R / 2;
    const int MR = PAIRED ? M * Rh : M * R;
    df best = df_make(0.0f), best_ax = df_make(0.0f);
    df bg[TA];
#pragma unroll
    for (int i = 0; i < TA; ++i) bg[i] = df_make(0.0f);
    int bm = -1, br = 0;
    int q = qf, u = uf;
    bool more = qf >= 0;
    unsigned uleft = more ? (umask_of(qf / kTcTop) & ~(1u << uf)) : 0u;
    unsigned bleft = more ? (bmask & ~(1u << qf)) : 0u;
    while (__any_sync(0xffffffffu, more)) {
      int id = -1;
      if (more) {
        const int b0 = a.cand_idx[p * kTcCand + q];
        if (b0 >= 0 && b0 < MR && b0 + u < MR) id = b0 + u;
      }
      const bool go = id >= 0;
      const int m = go ? id % M : 0, r = go ? id / M : 0;
      const bool flip = !PAIRED && r >= Rr;
      const int row = go ? (flip ? id - Rr * M : id) | (flip ? 1 << 30 : 0) : 0;
      // this unit's Gram entries with the selected atoms (one load each)
      df gq[NP][TA];
      if (go) {
#pragma unroll
        for (int i = 0; i < T; ++i) {
          int dr = r - S.r[i];
          if (dr < 0) dr += R;
          if (a.gram) {
            const float2 *gp = a.gram + ((size_t)m * M + S.m[i]) * R;
            const float2 g0 = __ldg(gp + dr);
            gq[0][i] = df{g0.x, g0.y};
            if (PAIRED) {
              const float2 g1 = __ldg(gp + (dr >= Rh ? dr - Rh : dr + Rh));
              gq[NP - 1][i] = df{g1.x, g1.y};
            }
          } else if (PAIRED) {
            const DF2 g2 = gram_entry_pair(a.xgram, M, a.H, R, m, r, S.m[i], S.r[i], tw);
            gq[0][i] = g2.a;
            gq[NP - 1][i] = g2.b;
          } else {
            gq[0][i] = gram_entry(a.xgram, M, a.H, R, m, r, S.m[i], S.r[i], tw);
          }
        }
      }
      // <A_c, x> in double-float, B rows at a time
      df axe = df_make(0.0f), axo = df_make(0.0f);
      unsigned todo = __ballot_sync(0xffffffffu, go);
      while (todo) {
        int src[B], slot;
        next_batch<B>(todo, lane, src, slot);
        float v[B][NS], h[B][NS];
        int rw[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
          rw[j] = __shfl_sync(0xffffffffu, row, src[j]);
          ls.load_x(a.x + (base + src[j]) * vec, v[j]);
          ls.load_row(a.rows_hi, rw[j] & ~(1 << 30), lane, h[j]);
        }
        df s[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
          s[j] = df_make(0.0f);
          float lo[NS];
          ls.load_row(a.rows_lo, rw[j] & ~(1 << 30), lane, lo);
#pragma unroll
          for (int w = 0; w < NS; ++w) {
            // weight 1 or 2 (exact); odd harmonics change sign with half a turn
            float xw = ls.wk[w] * v[j][w];
            if (!PAIRED && (rw[j] >> 30) && ((ls.odd >> w) & 1u)) xw = -xw;
            dot2_acc(s[j].hi, s[j].lo, h[j][w], xw);
            s[j].lo = __fmaf_rn(lo[w], xw, s[j].lo);
          }
        }
        // paired rows hold the even harmonics in slots 0 .. 63 (lanes 0 .. 15)
        // and the odd ones behind them: the two halves of the warp sum E and O
        const df z = batch_sum<B, PAIRED>(s, lane);
        const int from = slot < 0 ? 0 : slot;
        const df ze = shfl_df(z, from);
        if (slot >= 0) axe = fast_two_sum(ze.hi, ze.lo);
        if (PAIRED) {
          const df zo = shfl_df(z, from + 16);
          if (slot >= 0) axo = fast_two_sum(zo.hi, zo.lo);
        }
      }
      if (go) {
        df ax[NP];
        ax[0] = PAIRED ? df_add(axe, axo) : axe;
        if (PAIRED) ax[NP - 1] = df_sub(axe, axo);
#pragma unroll
        for (int h = 0; h < NP; ++h) {
          df sc = ax[h];
#pragma unroll
          for (int i = 0; i < T; ++i) sc = df_sub(sc, df_mul(df{S.ahi[i], S.alo[i]}, gq[h][i]));
          const int rr = r + h * Rh;
          if (bm < 0 || df_abs_gt(sc, best) ||
              (df_abs_eq(sc, best) && m * R + rr < bm * R + br)) {
            best = sc;
            bm = m;
            br = rr;
            best_ax = ax[h];
#pragma unroll
            for (int i = 0; i < T; ++i) bg[i] = gq[h][i];
          }
        }
      }
      // next unit: the next column of this block, else the first column of
      // the next kept block with a non-empty mask
      if (more) {
        while (uleft == 0 && bleft != 0) {
          q = __ffs(bleft) - 1;
          bleft &= bleft - 1;
          uleft = umask_of(q / kTcTop);
        }
        more = uleft != 0;
        if (more) {
          u = __ffs(uleft) - 1;
          uleft &= uleft - 1;
        }
      }
    }
    bool have_weights = false;
    int en = 0;
    float dr1 = 0.0f;
    if (act && outcome == 0) {
      if (bm < 0 || !(fabsf(best.hi) > stop_level)) {
        outcome = 1;
      } else {
        double gr[T + 1];
#pragma unroll
        for (int i = 0; i < T; ++i) gr[i] = df_to_d(bg[i]);
        gr[T] = 0.0;
        // <S_r d_m, S_r d_m> = ||d_m||^2: steering preserves the norm
        const float2 na = __ldg(a.anorm + bm);
        const double diag = (double)na.x + (double)na.y;
        const double rhs = df_to_d(best_ax);
#pragma unroll
        for (int i = 0; i < T * (T + 1) / 2; ++i) S.L[i] = a.sD[(I.dL + i) * P + p];
#pragma unroll
        for (int i = 0; i < T; ++i) {
          S.inv[i] = a.sD[(I.dInv + i) * P + p];
          S.z[i] = a.sD[(I.dZ + i) * P + p];
        }
        if (!chol_add<T + 1, T>(S, gr, diag, rhs)) {
          outcome = 1;
        } else {
          have_weights = true;
          S.m[T] = bm;
          S.r[T] = br;
          float asum = 0.0f;
#pragma unroll
          for (int i = 0; i <= T; ++i) asum += fabsf(S.ahi[i]);
          dr1 = residual_err(T + 1, xnorm, asum);
          if (T + 1 >= a.K) {
            outcome = 1;
            // final residual norm from the least-squares solution: with
            // L z = b (b_i = <A_i, x>, the factor of the Gram of the
            // selected steered atoms), ||x - sum_i a_i A_i||^2 =
            // ||x||^2 - z^T z, in FP64 from ||x||^2 in double-float (no
            // residual is formed: the fp16 row is not needed any more)
            double zz = 0.0;
#pragma unroll
            for (int i = 0; i <= T; ++i) zz = fma(S.z[i], S.z[i], zz);
            const double x2 = (double)a.sF[I.fX2h * P + p] + (double)a.sF[I.fX2l * P + p];
            rnorm = (float)sqrt(fmax(x2 - zz, 0.0));
          } else {
            // the previous residual's norm bounds the new one (least squares
            // over a larger support)
            en = rsc_row_exponent(rnorm);
#pragma unroll
            for (int i = 0; i <= T; ++i) {
              a.sD[(I.dL + T * (T + 1) / 2 + i) * P + p] = S.L[T * (T + 1) / 2 + i];
              a.sD[(I.dA + i) * P + p] = S.a[i];
              a.sF[(I.fHi + i) * P + p] = S.ahi[i];
              a.sF[(I.fLo + i) * P + p] = S.alo[i];
            }
            a.sD[(I.dInv + T) * P + p] = S.inv[T];
            a.sD[(I.dZ + T) * P + p] = S.z[T];
            a.sI[(I.iM + T) * P + p] = bm;
            a.sI[(I.iR + T) * P + p] = br;
            a.sI[I.iE * P + p] = en;
          }
        }
      }
    }
    // ---- new residual rows x - sum_i a_i S_{r_i} d_{m_i} (FP32) of the
    // patches that go on, B rows at a time
    const bool wr = act && outcome == 0;
    int rows[T + 1];
#pragma unroll
    for (int i = 0; i <= T; ++i) {
      const bool flip = wr && S.r[i] >= Rr;
      rows[i] = wr ? ((flip ? S.r[i] - Rr : S.r[i]) * M + S.m[i]) | (flip ? 1 << 30 : 0) : 0;
    }
    unsigned todo = __ballot_sync(0xffffffffu, wr);
    float rn2 = 0.0f;
    while (todo) {
      int src[B], slot;
      next_batch<B>(todo, lane, src, slot);
      float v[B][NS];
#pragma unroll
      for (int j = 0; j < B; ++j) ls.load_x(a.x + (base + src[j]) * vec, v[j]);
#pragma unroll
      for (int i = 0; i <= T; ++i) {
        float h[B][NS], w[B];
        int rw[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
          rw[j] = __shfl_sync(0xffffffffu, rows[i], src[j]);
          w[j] = __shfl_sync(0xffffffffu, S.ahi[i], src[j]);
          ls.load_row(a.rows_hi, rw[j] & ~(1 << 30), lane, h[j]);
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
          const float wo = (rw[j] >> 30) ? -w[j] : w[j];
#pragma unroll
          for (int s = 0; s < NS; ++s)
            v[j][s] = fmaf(-(((ls.odd >> s) & 1u) ? wo : w[j]), h[j][s], v[j][s]);
        }
      }
      float m2[B];
#pragma unroll
      for (int j = 0; j < B; ++j) {
        const int ej = __shfl_sync(0xffffffffu, en, src[j]);
        m2[j] = store_row<LAY>(ls, a.A, base + src[j], lane, ldexpf(1.0f, kRowLog2 - ej), v[j]);
      }
      const float z = batch_sum_f<B>(m2, lane);
      const float zr = __shfl_sync(0xffffffffu, z, slot < 0 ? 0 : slot);
      if (slot >= 0) rn2 = zr;
    }
    if (wr) {
      const float rn = sqrtf(rn2);
      a.sF[I.fR * P + p] = rn;
      a.win[p] = score_window(rn, dr1, en, a.L);
    } else if (act && outcome == 1) {
      if (have_weights) {
#pragma unroll
        for (int i = 0; i <= T; ++i) write_code(a, p, i, S.m[i], S.r[i], S.a[i]);
        write_none(a, p, T + 1);
      } else {
#pragma unroll
        for (int i = 0; i < T; ++i)
          write_code(a, p, i, S.m[i], S.r[i], a.sD[(I.dA + i) * P + p]);
        write_none(a, p, T);
      }
      if (a.resid_norm2) a.resid_norm2[p] = rnorm * rnorm;
      a.status[p] = 0;
    } else if (act) {
      a.sI[I.iT * P + p] = T;
      const int at = atomicAdd(a.redo_count, 1);
      a.redo_list[at] = (int)p;
      if (a.fallbacks) atomicAdd(a.fallbacks, 1ull);
      a.status[p] = -1;
    }
  }
}

template <int LAY>
int launch_refine_l(const RefineArgs &a, int step, unsigned grid, cudaStream_t stream) {
  switch (step) {
    case -1: romp_init_kernel<LAY><<<grid, 128, 0, stream>>>(a); break;
    case 0: romp_refine_kernel<0, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 1: romp_refine_kernel<1, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 2: romp_refine_kernel<2, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 3: romp_refine_kernel<3, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 4: romp_refine_kernel<4, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 5: romp_refine_kernel<5, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 6: romp_refine_kernel<6, LAY><<<grid, 128, 0, stream>>>(a); break;
    case 7: romp_refine_kernel<7, LAY><<<grid, 128, 0, stream>>>(a); break;
    default: return RSC_ERR_UNSUPPORTED;
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
}

}  // namespace

void rsc_state_layout(int K, int *nD, int *nF, int *nI) {
  const StateIdx I(K);
  *nD = I.nD;
  *nF = I.nF;
  *nI = I.nI;
}

int rsc_launch_refine(const RefineArgs &a, int step, cudaStream_t stream) {
  if (a.P == 0) return RSC_OK;
  int dev = 0, nsm = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // A warp takes 32 patches, or fewer (whole batches of rows, the other lanes
  // idle in the scalar parts) while that still leaves the SMs' 16 warps each
  // with work: a small call is one warp's chain of batches long.  1,000 patches
  // at M = 16, R = 32, K = 3: 127 us a call with 32 patches a warp, 81 with 4.
  RefineArgs w = a;
  const int64_t share = (a.P + 16 * nsm - 1) / (16 * nsm);
  w.warp_patches = (int)std::min<int64_t>(32, (share + 3) / 4 * 4);
  const int64_t per_block = 4 * w.warp_patches, blocks = (a.P + per_block - 1) / per_block;
  const int64_t cap = (int64_t)nsm * (a.blocks_per_sm > 0 ? a.blocks_per_sm : 32);
  const unsigned grid = (unsigned)(blocks < cap ? blocks : cap);
  if (a.L == kTcKstLong) return launch_refine_l<kLong>(w, step, grid, stream);
  return a.paired ? launch_refine_l<kPaired>(w, step, grid, stream)
                  : launch_refine_l<kPlain>(w, step, grid, stream);
}
