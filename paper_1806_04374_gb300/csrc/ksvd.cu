// ksvd.cu -- the rotational K-SVD dictionary update (inner loop of the
// R-K-SVD pseudocode, Fig. "code", Sec. II-C) on the GPU.
//
// For atom m, every patch whose code uses m at angle r0 contributes the
// column y = S_{-r0}(x_p - D_aug b_p), b_p being the patch's code with the
// (m, r0) entry removed -- equivalently y = S_{-r0} e_p + a_{i0} d_m with the
// full coding residual e_p = x_p - sum_i a_i S_{r_i} d_{m_i}.  The new atom is
// the first left singular vector of [y ...], i.e. the leading eigenvector of
// C_m = sum y y^T.  Every atom is updated from the same (old) dictionary and
// the same codes.  Readings: a repeated atom uses its occurrence with the
// largest |weight| (ties: earliest); an unused atom is reset to the
// unit-normalised patch with the largest coding error (successive patches in
// descending error for several, ties: smaller index); the eigenvector's
// largest-magnitude packed entry is made positive.
//
// Kernels: per chunk of patches (count samples per atom; then the per-atom
// sample lists in patch order and the residuals in double-float); the
// covariances, each split over `split` CTAs that take slices of the atom's
// samples, on the tensor cores for n <= 112 (exact products of 8-bit slices)
// and on the CUDA cores otherwise (exact FP32 products with their cross
// terms); the partials added in a fixed order, so that the update is
// FP64-grade and the same on every run; one CTA per atom running an FP64
// power iteration from the old atom; one CTA for the resets.  Packed vectors
// are real (k = 0 real parts, sqrt(2) Re/Im of k >= 1).
#include <math.h>

#include <algorithm>

#include "df.cuh"
#include "rsc_internal.h"
#include "rsc_trace.h"
#include "tc_ptx.cuh"

#include <cuda_bf16.h>

namespace {

constexpr int kCovThreads = 384;  // one 4 x 4 tile each: all 351 tiles of n = 102 in one round
// patches per chunk of the sample lists: 1,563 blocks at 200,000 patches, so that
// the last of them leave few SMs idle (256 patches 0.39 ms, 128 0.33, 64 0.31, but
// a count per chunk and atom to scan)
constexpr int kFillChunk = 128;
constexpr int kMaxAtomsKsvd = 12288;  // per-atom cursors of a chunk in shared memory
constexpr int kCovBatch = 32;
constexpr int kEigThreads = 256;
constexpr int kMaxPacked = 2 * kMaxEntries;

struct KsvdArgs {
  const float *x;
  int64_t P;
  int K, M, J, H, R, n;
  const float *d;   // [M][H][J][2]
  const float *tw;  // [4][H][R]
  const int32_t *atom;
  const int32_t *angle;
  const double *coef;
  float4 *E;        // [P][H*J] residuals with their packing weight, double-float (re hi, im hi, re lo, im lo)
  float *err2;      // [P] coding errors ||e_p||^2
  int *count;       // [M]
  int *offset;      // [M + 1]
  int *chunk_cnt;   // [nchunk][M] samples of each atom in each chunk of patches
  int *chunk_base;  // [nchunk][M] first slot of each atom's samples of each chunk, from the atom's first
  int nchunk;
  int4 *samples;    // [sum count] (patch, angle, weight hi, lo), patch order within an atom
  int split;        // slices of an atom's samples, a CTA each
  double *C;        // [M][n][n]
  double *Cpart;    // [split][M] partial sums of `stride` doubles: [n][n], the upper triangle
                    // written, or from the tensor cores float2 pieces (kCvPair)
  size_t stride;
  int *state;       // [split][M] what a slice's partial sum is (null: kCvFull64 all)
  int *expo;        // [split][M][128] exponents of a kCvPair slice's rows
  int *err;         // the dictionary's device error word
  uint64_t wait_ns; // limit of the tensor-core kernel's pipeline waits
  float *new_coef;  // [M][H][J][2]
  int32_t *n_used;  // [M] or null
  // the patches of largest coding error (descending, ties: smaller index),
  // unit-normalised, for the reset of unused atoms
  int ntop;         // entries of the list
  int top_needed;   // 1: list only as long as the atoms with count 0 need (one rank)
  float *top_err;   // [ntop]
  int64_t *top_idx; // [ntop] patch index (-1: none)
  float *top_vec;   // [ntop][H][J][2]
};

enum : int { kCvPair = 0, kCvFull64 = 1, kCvNone = 2, kCvFailed = 3 };

constexpr int kTopMax = 64;  // patches kept for the resets (unused atoms beyond: unchanged)

// Occurrence i of patch p is the one that represents its atom (largest
// |weight| among the occurrences of that atom, ties: earliest).
__device__ __forceinline__ bool chosen(const KsvdArgs &a, int64_t p, int i) {
  const int m = a.atom[p * a.K + i];
  if (m < 0) return false;
  const double w = fabs(a.coef[p * a.K + i]);
  for (int q = 0; q < a.K; ++q) {
    if (q == i || a.atom[p * a.K + q] != m) continue;
    const double v = fabs(a.coef[p * a.K + q]);
    if (v > w || (v == w && q < i)) return false;
  }
  return true;
}

// Samples of each atom in each chunk of kFillChunk patches (shared-memory
// histogram; integer counts do not depend on the order of the additions).
__global__ void ksvd_chunk_count_kernel(const KsvdArgs a) {
  extern __shared__ int hist[];  // [M]
  for (int m = threadIdx.x; m < a.M; m += blockDim.x) hist[m] = 0;
  __syncthreads();
  const int64_t p0 = (int64_t)blockIdx.x * kFillChunk;
  const int64_t p1 = min(a.P, p0 + kFillChunk);
  for (int64_t p = p0 + threadIdx.x; p < p1; p += blockDim.x)
    for (int i = 0; i < a.K; ++i)
      if (chosen(a, p, i)) atomicAdd(&hist[a.atom[p * a.K + i]], 1);
  __syncthreads();
  for (int m = threadIdx.x; m < a.M; m += blockDim.x)
    a.chunk_cnt[(size_t)blockIdx.x * a.M + m] = hist[m];
}

// Block-wide exclusive prefix sum of one value per thread (256 threads).
__device__ __forceinline__ int block_prefix(int v, int *ws, int *total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (i < w) before += ws[i];
    all += ws[i];
  }
  __syncthreads();
  *total = all;
  return before + x - v;
}

// One block per atom: its count, and for every chunk the samples of the
// chunks before it.
__global__ void __launch_bounds__(256) ksvd_atom_scan_kernel(const KsvdArgs a) {
  __shared__ int ws[8];
  const int m = blockIdx.x;
  int base = 0;
  for (int c0 = 0; c0 < a.nchunk; c0 += 256) {
    const int c = c0 + threadIdx.x;
    const int v = c < a.nchunk ? a.chunk_cnt[(size_t)c * a.M + m] : 0;
    int total;
    const int x = block_prefix(v, ws, &total);
    if (c < a.nchunk) a.chunk_base[(size_t)c * a.M + m] = base + x;
    base += total;
  }
  if (threadIdx.x == 0) {
    a.count[m] = base;
    if (a.n_used) a.n_used[m] = base;
  }
}

// First slot of every atom (atoms in order); one block.
__global__ void __launch_bounds__(256) ksvd_offset_kernel(const KsvdArgs a) {
  __shared__ int ws[8];
  int base = 0;
  for (int m0 = 0; m0 < a.M; m0 += 256) {
    const int m = m0 + threadIdx.x;
    int total;
    const int x = block_prefix(m < a.M ? a.count[m] : 0, ws, &total);
    if (m < a.M) a.offset[m] = base + x;
    base += total;
  }
  if (threadIdx.x == 0) a.offset[a.M] = base;
}

// Per chunk: the residuals e_p = x_p - sum_i a_i S_{r_i} d_{m_i} of its
// patches in double-float with their coding errors, a warp per patch, and the
// chunk's sample slots in patch order: warp 0 takes 32 occurrences at a time in
// order, those of the same atom ranked by a match over the warp, so every
// atom's list is in patch order on every run.
//
// Bound by the double-float arithmetic: 0.33 ms per 200,000 patches at K = 5 and
// n = 102 (0.93 with a thread per patch, which read 32 rows with every load;
// 0.45 with patches dealt to the warps, the seven others waiting for warp 0).
constexpr int kFillThreads = 256;

__device__ __forceinline__ unsigned char *smem_align16(unsigned char *p) {
  return reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15));
}

// ||e||^2 of the residual at E (each lane its own entries, as it wrote them) in
// FP64, rounded once: infinity past FP32's range.
__device__ __noinline__ float coding_error64(const float4 *E, int HJ, int lane) {
  double s = 0.0;
  bool some = false;
  for (int e = lane; e < HJ; e += 32) some |= E[e].x != 0.0f || E[e].y != 0.0f;
  if (!__any_sync(0xffffffffu, some)) return 0.0f;  // (NaN is not 0)
  for (int e = lane; e < HJ; e += 32) {
    const float4 v = E[e];
    const double re = (double)v.x + (double)v.z, im = (double)v.y + (double)v.w;
    s = fma(re, re, fma(im, im, s));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return (float)s;
}

template <bool TW>
__global__ void __launch_bounds__(kFillThreads) ksvd_fill_kernel(const KsvdArgs a) {
  // [kFillChunk][K] code (weight hi, lo, atom or -1, angle); [M] next slot of
  // each atom in this chunk; [kFillChunk][K] slot of each chosen occurrence
  extern __shared__ __align__(16) int4 s_code[];
  const int J = a.J, H = a.H, HJ = H * J, R = a.R, K = a.K;
  int *cur = reinterpret_cast<int *>(s_code + kFillChunk * K), *slot = cur + a.M;
  // the steering factors as [R][H] (cos hi, lo, sin hi, lo) where they fit: one
  // load of 16 bytes in place of four in different lines
  float4 *s_tw = reinterpret_cast<float4 *>(
      smem_align16(reinterpret_cast<unsigned char *>(slot + kFillChunk * K)));
  __shared__ int s_next;
  if (threadIdx.x == 0) s_next = 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * kFillChunk;
  const int np = (int)min((int64_t)kFillChunk, a.P - p0);
  for (int m = threadIdx.x; m < a.M; m += kFillThreads)
    cur[m] = a.offset[m] + a.chunk_base[(size_t)blockIdx.x * a.M + m];
  auto factors = [&](int k, int r) {
    return make_float4(a.tw[(0 * H + k) * R + r], a.tw[(1 * H + k) * R + r],
                       a.tw[(2 * H + k) * R + r], a.tw[(3 * H + k) * R + r]);
  };
  if (TW)
    for (int i = threadIdx.x; i < R * H; i += kFillThreads) {
      const int k = i / R, r = i - k * R;
      s_tw[r * H + k] = factors(k, r);
    }
  for (int i = threadIdx.x; i < np * K; i += kFillThreads) {
    const df w = df_from_d(a.coef[p0 * K + i]);
    s_code[i] = make_int4(__float_as_int(w.hi), __float_as_int(w.lo), a.atom[p0 * K + i],
                          a.angle[p0 * K + i]);
  }
  __syncthreads();
  if (warp == 0) {
    for (int i0 = 0; i0 < np * K; i0 += 32) {
      const int i = i0 + lane;
      const int m = i < np * K && chosen(a, p0 + i / K, i % K) ? s_code[i].z : -1;
      const unsigned same = __match_any_sync(0xffffffffu, m);
      const int rank = __popc(same & ((1u << lane) - 1u));
      if (i < np * K) slot[i] = m >= 0 ? cur[m] + rank : -1;
      __syncwarp();
      if (m >= 0 && rank == 0) cur[m] += __popc(same);
      __syncwarp();
    }
  }
  const df sqrt2 = df_from_d(1.4142135623730951);
  // (patches are drawn, not dealt: warp 0 comes later)
  for (;;) {
    int pl = 0;
    if (lane == 0) pl = atomicAdd(&s_next, 1);
    pl = __shfl_sync(0xffffffffu, pl, 0);
    if (pl >= np) break;
    const int64_t p = p0 + pl;
    df n2 = df_make(0.0f);
    for (int e = lane; e < HJ; e += 32) {
      const int k = e / J;
      const float2 v = reinterpret_cast<const float2 *>(a.x)[p * HJ + e];
      df re = df_make(v.x), im = df_make(k ? v.y : 0.0f);
      for (int i = 0; i < K; ++i) {
        const int4 c4 = s_code[pl * K + i];
        if (c4.z < 0) continue;
        const float4 f = TW ? s_tw[c4.w * H + k] : factors(k, c4.w);
        const df c = {f.x, f.y}, sn = {f.z, f.w};
        const float2 dv = __ldg(reinterpret_cast<const float2 *>(a.d) + (size_t)c4.z * HJ + e);
        const float dim = k ? dv.y : 0.0f;
        const df w = {__int_as_float(c4.x), __int_as_float(c4.y)};
        // S_r d: harmonic k times exp(-i k theta_r)
        const df sre = df_add(df_mul_f(c, dv.x), df_mul_f(sn, dim));
        const df sim = df_sub(df_mul_f(c, dim), df_mul_f(sn, dv.x));
        re = df_sub(re, df_mul(w, sre));
        im = df_sub(im, df_mul(w, sim));
      }
      if (k) {
        re = df_mul(re, sqrt2);
        im = df_mul(im, sqrt2);
      } else {
        im = df_make(0.0f);
      }
      a.E[p * HJ + e] = make_float4(re.hi, im.hi, re.lo, im.lo);
      n2 = df_add(n2, df_add(df_mul(re, re), df_mul(im, im)));
    }
    n2 = df_warp_sum(n2);
    // squares outside FP32's range (infinite, or tails lost below it): FP64
    float err = n2.hi;
    if (!(err > 1e-30f && err < 1e38f)) err = coding_error64(a.E + p * HJ, HJ, lane);
    if (lane == 0) a.err2[p] = err;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < np * K; i += kFillThreads) {
    if (slot[i] < 0) continue;
    const int pl = i / K;
    const int4 c4 = s_code[i];
    // the code entry of (m, r0): every occurrence of that pair (Fig. "code"
    // zeroes the whole entry b_{r0}[m])
    df w = {__int_as_float(c4.x), __int_as_float(c4.y)};
    bool twice = false;
    for (int q = 0; q < K; ++q)
      twice |= q != i - pl * K && s_code[pl * K + q].z == c4.z && s_code[pl * K + q].w == c4.w;
    if (twice) {
      double sum = 0.0;
      for (int q = 0; q < K; ++q)
        if (s_code[pl * K + q].z == c4.z && s_code[pl * K + q].w == c4.w)
          sum += a.coef[(p0 + pl) * K + q];
      w = df_from_d(sum);
    }
    a.samples[slot[i]] =
        make_int4((int)(p0 + pl), c4.w, __float_as_int(w.hi), __float_as_int(w.lo));
  }
}

// C_m = sum over the atom's samples of y y^T, y = S_{-r0} e_p + a_{i0} d_m.
// CUDA-core form, for packed lengths over kTcvMaxN and for the slices that the
// tensor-core kernel leaves (kCvFull64): a.split CTAs per atom, slices in list
// order; each thread owns 4 x 4 tiles of the upper triangle.  The columns y of a
// batch of kCovBatch samples are built in double-float in shared memory; a
// product y_i y_j is the exact product of the hi parts (TwoProd) plus the
// cross terms hi_i lo_j + lo_i hi_j, and the batch's products are summed
// Dot2-style (TwoSum of the hi parts, the errors and lo parts summed apart),
// then added to FP64 accumulators.  Each CTA writes its partial sums to its
// own slice of Cpart (every entry, zero when it has no samples); a second
// kernel adds the slices in order.
__global__ void __launch_bounds__(kCovThreads) ksvd_cov_kernel(const KsvdArgs a) {
  extern __shared__ __align__(16) float ysm[];  // 2 x kCovBatch rows of ldy floats
  __shared__ int s_p[kCovBatch], s_r0[kCovBatch];
  __shared__ df s_w[kCovBatch];
  const int m = blockIdx.x / a.split, part = blockIdx.x - m * a.split;
  if (a.state && a.state[part * a.M + m] != kCvFull64) return;
  const int n = a.n, J = a.J, H = a.H, HJ = H * J, R = a.R;
  const int nb4 = (n + 3) / 4, ldy = 4 * nb4 + 4;  // +4: rows start in different banks
  float *yhi = ysm, *ylo = ysm + kCovBatch * ldy;
  // (a.state: the slices may be longer than the eighth of an atom's samples
  // that they are without it; FP64 takes over earlier to make up for it)
  const int batch = a.state ? kCovBatch / 2 : kCovBatch;
  const int beg0 = a.offset[m], cnt = a.offset[m + 1] - beg0;
  const int per = (cnt + a.split - 1) / a.split;
  const int beg = beg0 + part * per, end = min(beg0 + cnt, beg + per);
  double *Cm = a.Cpart + ((size_t)part * a.M + m) * a.stride;
  const df sqrt2 = df_from_d(1.4142135623730951);
  const int ntiles = nb4 * (nb4 + 1) / 2;
  for (int t = threadIdx.x; t - threadIdx.x < ntiles; t += kCovThreads) {
    // tile (bi, bj), bi <= bj, of the upper triangle (row bi starts at
    // bi*nb4 - bi(bi-1)/2)
    int bi = -1, bj = -1;
    if (t < ntiles) {
      int lo = 0, hi = nb4 - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (mid * nb4 - mid * (mid - 1) / 2 <= t) lo = mid; else hi = mid - 1;
      }
      bi = lo;
      bj = bi + (t - (bi * nb4 - bi * (bi - 1) / 2));
    }
    double acc[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) acc[u] = 0.0;
    for (int b0 = beg; b0 < end; b0 += batch) {
      const int nb = min(batch, end - b0);
      __syncthreads();
      for (int w = threadIdx.x; w < nb * ldy; w += blockDim.x) {
        yhi[w] = 0.0f;
        ylo[w] = 0.0f;
      }
      if (threadIdx.x < nb) {
        const int4 smp = a.samples[b0 + threadIdx.x];
        s_p[threadIdx.x] = smp.x;
        s_r0[threadIdx.x] = smp.y;
        s_w[threadIdx.x] = df{__int_as_float(smp.z), __int_as_float(smp.w)};
      }
      __syncthreads();
      for (int w = threadIdx.x; w < nb * HJ; w += blockDim.x) {
        const int s = w / HJ, e = w - s * HJ;
        const int64_t p = s_p[s];
        const int r0 = s_r0[s];
        const df w0 = s_w[s];
        const int k = e / J;
        const float4 ev = a.E[p * HJ + e];
        const float2 dv = reinterpret_cast<const float2 *>(a.d)[(size_t)m * HJ + e];
        if (k == 0) {
          const df y = df_add(df{ev.x, ev.z}, df_mul_f(w0, dv.x));
          yhi[s * ldy + e] = y.hi;
          ylo[s * ldy + e] = y.lo;
        } else {
          const int q = 2 * e - J;
          const df re = {ev.x, ev.z}, im = {ev.y, ev.w};
          // S_{-theta}: harmonic k times exp(+i k theta)
          const df c = {a.tw[(0 * H + k) * R + r0], a.tw[(1 * H + k) * R + r0]};
          const df sn = {a.tw[(2 * H + k) * R + r0], a.tw[(3 * H + k) * R + r0]};
          const df w2 = df_mul(w0, sqrt2);
          const df yr = df_add(df_sub(df_mul(re, c), df_mul(im, sn)), df_mul_f(w2, dv.x));
          const df yi = df_add(df_add(df_mul(re, sn), df_mul(im, c)), df_mul_f(w2, dv.y));
          yhi[s * ldy + q] = yr.hi;
          ylo[s * ldy + q] = yr.lo;
          yhi[s * ldy + q + 1] = yi.hi;
          ylo[s * ldy + q + 1] = yi.lo;
        }
      }
      __syncthreads();
      if (bi >= 0) {
        float sh[16], sl[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) sh[u] = sl[u] = 0.0f;
        for (int s = 0; s < nb; ++s) {
          const float4 hi4 = *reinterpret_cast<const float4 *>(&yhi[s * ldy + 4 * bi]);
          const float4 hj4 = *reinterpret_cast<const float4 *>(&yhi[s * ldy + 4 * bj]);
          const float4 li4 = *reinterpret_cast<const float4 *>(&ylo[s * ldy + 4 * bi]);
          const float4 lj4 = *reinterpret_cast<const float4 *>(&ylo[s * ldy + 4 * bj]);
          const float hi[4] = {hi4.x, hi4.y, hi4.z, hi4.w}, hj[4] = {hj4.x, hj4.y, hj4.z, hj4.w};
          const float li[4] = {li4.x, li4.y, li4.z, li4.w}, lj[4] = {lj4.x, lj4.y, lj4.z, lj4.w};
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const df pp = two_prod(hi[u], hj[v]);
              const float cross = __fmaf_rn(hi[u], lj[v], __fmaf_rn(li[u], hj[v], pp.lo));
              const df ts = two_sum(sh[u * 4 + v], pp.hi);
              sh[u * 4 + v] = ts.hi;
              sl[u * 4 + v] = __fadd_rn(sl[u * 4 + v], __fadd_rn(ts.lo, cross));
            }
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) acc[u] += (double)sh[u] + (double)sl[u];
      }
    }
    if (bi >= 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          const int i = 4 * bi + u, j = 4 * bj + v;
          if (i < n && j < n && i <= j) Cm[(size_t)i * n + j] = acc[u * 4 + v];
        }
    }
  }
}

// C_m on the tensor cores, n <= kTcvMaxN.  The columns y are built in
// double-float; every row of a slice's samples is scaled by a power of two of
// its own, |y_i| < 1/2 (from a first pass in FP32), and cut into six bf16
// values y = b0 + ... + b5: b0, b1, b2 and b3 multiples of 2^-8, 2^-16, 2^-24
// and 2^-32 below 2^-1, 2^-9, 2^-17 and 2^-24, b4 and b5 what is left, 8 bits
// each.  The 26 products b_i b_j^T down to 2^-53 are summed by order i + j:
// orders 0 to 3 are integers (in units of 2^-16, 2^-24, 2^-32, 2^-40), at most
// 2^14, 2^15, 3 2^14 and 5 2^14 a sample.  Sums of orders 0 to 2 stay below 2^24
// for a window of samples, those of order 3 for three stages of it, so FP32
// holds them exactly; the rest, 2^-32 of the whole, is summed as it comes.
// Orders 0 to 2 have an accumulator each; order 3 and the rest take turns in a
// fourth, read out after each turn.  A slice's sums are kept in three floats without loss
// but for the third's own rounding, 2^-24 of 2^-28 (FP64 at 64 cycles an
// instruction held the accumulators up).
//
// Bound by the MMAs (104 a stage of 64 samples, 61 cycles each) and the slicing
// beside them.  Per CTA (one slice of one atom):
//   * warps 0-14 build a stage (64 samples x 128 rows x 6 values, K-major,
//     128-byte swizzle): a thread takes one entry of eight samples;
//   * warps 15-22 read the accumulators (some columns of 32 rows a warp);
//   * warp 23 (one lane) issues the MMAs (M = 128, N = n padded to 16).
// Rows hold the real parts of the entries first, then the imaginary parts of
// k >= 1, so that neighbouring lanes store to neighbouring rows.
// 200,000 patches, K = 5, M = 128, n = 102, R = 64 (10^6 samples): 1.06 ms, and
// the whole accumulation and update 1.60 ms (6.86 ms with every covariance on
// the CUDA cores); C off by 1.8e-15 of its norm, 1.9e-15 there.
// Every wait is bounded.  One that runs out is reported twice: in the
// dictionary's error word, and as a slice without a sum (kCvFailed), which
// makes all of its atom's C not a number, so that neither the covariance nor
// what is added to it or made of it passes for a result.
constexpr int kTcvBuild = 15, kTcvSum = 8;  // warps
constexpr int kTcvThreads = 32 * (kTcvBuild + kTcvSum + 1);  // six warps a scheduler: 80 registers
constexpr int kTcvSamples = 64;          // samples of a stage
constexpr int kTcvSlices = 6;
constexpr int kTcvSlice = 128 * 128;     // one slice of a stage (bytes)
constexpr int kTcvStage = kTcvSlices * kTcvSlice;
constexpr int kTcvStages = 5;            // stages per window: order 2, 3 * 2^14 * 320 < 2^24
constexpr int kTcvThird = 3;             // of these, order 3 at once: 5 * 2^14 * 192 < 2^24
// the sum of order 3 that two stages more leave below 2^24 (units of 2^-40)
constexpr float kTcvThirdMax =
    (float)((1 << 24) - 5 * (1 << 14) * kTcvSamples * (kTcvStages - kTcvThird)) / 1099511627776.0f;
constexpr int kTcvMaxN = 112;            // packed lengths up to here
constexpr int kTcvUnits = 5;             // pieces of eight columns of a summing warp
constexpr int kTcvTwMax = 28 * 1024;     // steering factors kept in shared memory (bytes)
constexpr int kTcvPlaces = kTcvSum * 8 * kTcvUnits * 32;  // of a slice's sums
constexpr uint64_t kTcvWaitNs = 2000000000ull;  // drain waits (and the default pipeline limit)
enum : int { kCvFull = 0, kCvEmpty = 2, kCvXFull = 4, kCvXFree = 5, kCvAccFull = 6, kCvAccFree = 7, kCvRec = 8, kCvBars = 12 };
constexpr int kTcvBarOff = 2 * kTcvStage;
constexpr int kTcvScOff = kTcvBarOff + 128;       // [128] exponents of the rows
constexpr int kTcvMaxOff = kTcvScOff + 128 * 4;   // [128] their largest values
constexpr int kTcvRecOff = kTcvMaxOff + 128 * 4;  // [4][kTcvSamples] sample records of coming stages
constexpr int kTcvTwOff = kTcvRecOff + 4 * kTcvSamples * 16;

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {  // a in the low half
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// The six values of one row of two samples, two bf16 to a word.
__device__ __forceinline__ void slice2(df y0, df y1, uint32_t (&o)[kTcvSlices]) {
  // adding 1.5 2^15, 1.5 2^7, 1.5 2^-1 and 1.5 2^-9 leaves multiples of 2^-8,
  // 2^-16, 2^-24 and 2^-32
  const float big[4] = {49152.0f, 192.0f, 0.75f, 0.0029296875f};
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const float b0 = __fsub_rn(__fadd_rn(y0.hi, big[s]), big[s]);
    const float b1 = __fsub_rn(__fadd_rn(y1.hi, big[s]), big[s]);
    y0.hi = __fsub_rn(y0.hi, b0);
    y1.hi = __fsub_rn(y1.hi, b1);
    o[s] = pack_bf16(b0, b1);
  }
  const df t0 = two_sum(y0.hi, y0.lo), t1 = two_sum(y1.hi, y1.lo);
  o[3] = pack_bf16(__fsub_rn(__fadd_rn(t0.hi, big[3]), big[3]),
                   __fsub_rn(__fadd_rn(t1.hi, big[3]), big[3]));
  float c0 = __fadd_rn(__fsub_rn(t0.hi, __uint_as_float(o[3] << 16)), t0.lo);
  float c1 = __fadd_rn(__fsub_rn(t1.hi, __uint_as_float(o[3] & 0xffff0000u)), t1.lo);
  o[4] = pack_bf16(c0, c1);
  c0 = __fsub_rn(c0, __uint_as_float(o[4] << 16));
  c1 = __fsub_rn(c1, __uint_as_float(o[4] & 0xffff0000u));
  o[5] = pack_bf16(c0, c1);
}

// First column of piece s of a summing warp, N for none.  Every pair of 32-row
// blocks comes once: rows 32 quarter .. + 31 take the blocks {0, 1, 3},
// {1, 2, 3}, {2, 0, 3} and {3} of columns (block 3 has at most 16), in pieces of
// eight, every other one of them.
__device__ __forceinline__ int cov_column(int quarter, int group, int s, int N) {
  const int t = 2 * s + group, i = t >> 2;
  if (quarter == 3 && i > 0) return N;
  const int blk = i == 2 || quarter == 3 ? 3 : (quarter + i) % 3;
  return min(N, 32 * blk + 8 * (t & 3));
}
// Packed coordinate of row r of the operands (the real parts of all entries,
// then the imaginary parts of k >= 1).
__device__ __forceinline__ int cov_coord(int r, int J, int HJ) {
  return r < J ? r : (r < HJ ? 2 * r - J : 2 * (r - HJ) + J + 1);
}

// 8 consecutive 32-bit TMEM columns of this thread's lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7])
      : "r"(taddr));
}

__global__ void __launch_bounds__(kTcvThreads, 1) ksvd_cov_tc_kernel(const KsvdArgs a, int N) {
  extern __shared__ unsigned char cv_raw[];
  unsigned char *smem = reinterpret_cast<unsigned char *>(
      (reinterpret_cast<uintptr_t>(cv_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + kTcvBarOff);
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(bars + kCvBars);
  volatile int *s_abort = reinterpret_cast<volatile int *>(bars + kCvBars) + 1;
  int *s_exp = reinterpret_cast<int *>(smem + kTcvScOff);       // exponent of each row
  int *s_max = reinterpret_cast<int *>(smem + kTcvMaxOff);      // bits of non-negative floats
  float4 *s_tw = reinterpret_cast<float4 *>(smem + kTcvTwOff);  // [R][H] cos hi, lo, sin hi, lo
  const uint32_t bar0 = tc::smem_u32(bars);
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  auto arrive = [&](int i) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar(i)) : "memory");
  };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, J = a.J, H = a.H, HJ = H * J, R = a.R;
  const int m = blockIdx.x / a.split, part = blockIdx.x - m * a.split;
  const int beg0 = a.offset[m], cnt = a.offset[m + 1] - beg0;
  const int per = (cnt + a.split - 1) / a.split;
  const int beg = beg0 + part * per, ns = max(0, min(beg0 + cnt, beg + per) - beg);
  const size_t slice = (size_t)part * a.M + m;

  for (int i = tid; i < 128; i += kTcvThreads) s_max[i] = 0;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(bar(kCvFull + i), kTcvBuild);
      tc::mbar_init(bar(kCvEmpty + i), 1);
    }
    tc::mbar_init(bar(kCvXFull), 1);
    tc::mbar_init(bar(kCvXFree), kTcvSum);
    tc::mbar_init(bar(kCvAccFull), 1);
    tc::mbar_init(bar(kCvAccFree), kTcvSum);
    for (int i = 0; i < 4; ++i) tc::mbar_init(bar(kCvRec + i), 1);
    *s_abort = 0;
    tc::fence_mbar_init();
  }
  // rows n .. 127 stay zero
  for (int i = tid; i < 2 * kTcvSlices * (128 - n) * 8; i += kTcvThreads) {
    const int sl = i / ((128 - n) * 8), rem = i - sl * (128 - n) * 8;
    reinterpret_cast<uint4 *>(smem + sl * kTcvSlice + n * 128)[rem] = make_uint4(0, 0, 0, 0);
  }
  for (int i = tid; i < R * H; i += kTcvThreads) {
    const int k = i / R, r = i - k * R;
    s_tw[r * H + k] = make_float4(a.tw[(0 * H + k) * R + r], a.tw[(1 * H + k) * R + r],
                                  a.tw[(2 * H + k) * R + r], a.tw[(3 * H + k) * R + r]);
  }
  __syncthreads();
  // ---- the largest |y| of every row over the slice, in FP32: off by less than
  // 2^-20 of the sum of moduli |e| + |w| |d|, which is added
  for (int e0 = 0; e0 < HJ; e0 += 32) {
    const int e = e0 + lane, k = e / J;
    float mr = 0.0f, mi = 0.0f, mq = 0.0f;
    if (e < HJ) {
      float2 dv = __ldg(reinterpret_cast<const float2 *>(a.d) + (size_t)m * HJ + e);
      // the residual carries the packing weight sqrt(2) of k >= 1, the atom not
      if (k) {
        dv.x *= 1.41421356f;
        dv.y *= 1.41421356f;
      }
      const float d1 = fabsf(dv.x) + fabsf(dv.y);
#pragma unroll 4
      for (int i = warp; i < ns; i += kTcvThreads / 32) {
        const int4 smp = __ldg(a.samples + beg + i);
        const float4 ev = __ldg(a.E + (size_t)smp.x * HJ + e);
        const float4 f = s_tw[smp.y * H + k];
        const float w = __int_as_float(smp.z);
        mr = fmaxf(mr, fabsf(fmaf(ev.x, f.x, fmaf(-ev.y, f.z, w * dv.x))));
        mi = fmaxf(mi, fabsf(fmaf(ev.x, f.z, fmaf(ev.y, f.x, w * dv.y))));
        const float q = fmaf(fabsf(w), d1, fabsf(ev.x) + fabsf(ev.y));
        mq = q <= mq ? mq : (q == q ? q : INFINITY);
      }
      const float slack = 9.5367431640625e-7f * mq;
      atomicMax(&s_max[e], __float_as_int(mr + slack));
      if (k) atomicMax(&s_max[HJ + e - J], __float_as_int(mi + slack));
    }
  }
  __syncthreads();
  // exponents: |y| < 2^(E - 1); rows that are zero throughout take any.
  // Outside the range of FP32 scaling (also infinities) the CUDA cores take
  // the slice.
  bool fits = true;
  for (int r = tid; r < n; r += kTcvThreads) {
    const float q = __int_as_float(s_max[r]);
    int E = 0;
    if (q > 0.0f) {
      fits = q > 1e-12f && q < 1e15f;
      if (fits) (void)frexpf(1.0001f * q, &E);
    }
    s_exp[r] = E + 1;
  }
  const bool mine = __syncthreads_and(fits || ns == 0) != 0;
  if (tid == 0) a.state[slice] = ns == 0 ? kCvNone : (mine ? kCvPair : kCvFull64);
  if (ns == 0 || !mine) return;
  for (int r = tid; r < n; r += kTcvThreads) a.expo[slice * 128 + r] = s_exp[r];
  if (warp == 0) tc::tmem_alloc(tc::smem_u32(s_tmem), 512);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = *s_tmem;
  const int nst = (ns + kTcvSamples - 1) / kTcvSamples;
  auto fail = [&]() {
    *s_abort = 1;
    a.state[slice] = kCvFailed;
    if (a.err) atomicCAS(a.err, 0, RSC_ERR_TIMEOUT);
  };

  if (warp == kTcvBuild + kTcvSum) {
    // ---------------------------------------------------------------- MMA
    if (lane == 0) {
      // bf16 A and B (format code 1), f32 D
      const uint32_t idesc = tc::idesc_f16_f32(128, N) | (1u << 7) | (1u << 10);
      // (accumulator, i, j); order 3 and the rest share accumulator 3
      constexpr int kRest = 16;
      constexpr int rest[kRest][2] = {{1, 5}, {5, 1}, {2, 4}, {4, 2}, {3, 3}, {1, 4}, {4, 1}, {2, 3},
                                     {3, 2}, {0, 5}, {5, 0}, {2, 2}, {1, 3}, {3, 1}, {0, 4}, {4, 0}};
      constexpr int low[3][3] = {{0, 0, 0}, {1, 0, 1}, {1, 1, 0}};
      constexpr int order3[4][2] = {{1, 2}, {2, 1}, {0, 3}, {3, 0}};
      constexpr int two[3][3] = {{2, 0, 2}, {2, 2, 0}, {2, 1, 1}};
      int st = 0;
      for (; st < nst; ++st) {
        const int b = st & 1, win = st / kTcvStages;
        const bool opens = st == win * kTcvStages;
        const uint64_t d0 = tc::smem_desc_sw128(tc::smem_u32(smem + b * kTcvStage));
        const int ks_n = (min(kTcvSamples, ns - st * kTcvSamples) + 15) / 16;
        auto product = [&](int acc, int i, int j, bool clear) {
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)
            if (ks < ks_n)
              tc::mma_f16(tmem + acc * N, tc::desc_at(d0, i * kTcvSlice + ks * 32),
                          tc::desc_at(d0, j * kTcvSlice + ks * 32), idesc,
                          clear && ks == 0 ? 0u : 1u);
        };
        if (*s_abort || !tc::mbar_wait_bounded(bar(kCvFull + b), (st >> 1) & 1, a.wait_ns) ||
            (st > 0 && !tc::mbar_wait_bounded(bar(kCvXFree), 1, a.wait_ns))) {
          fail();
          break;
        }
        tc::fence_after_sync();
        // the shared accumulator is read while the others' products run
#pragma unroll
        for (int q = 0; q < kRest; ++q) product(3, rest[q][0], rest[q][1], q == 0);
        tc::mma_commit(bar(kCvXFull));
        bool ok = !(opens && win > 0) ||
                  tc::mbar_wait_bounded(bar(kCvAccFree), (win - 1) & 1, a.wait_ns);
        tc::fence_after_sync();
        if (ok) {
#pragma unroll
          for (int q = 0; q < 3; ++q) product(low[q][0], low[q][1], low[q][2], opens && q < 2);
          ok = tc::mbar_wait_bounded(bar(kCvXFree), 0, a.wait_ns);
        }
        tc::fence_after_sync();
        if (ok) {
#pragma unroll
          for (int q = 0; q < 4; ++q) product(3, order3[q][0], order3[q][1], q == 0);
          tc::mma_commit(bar(kCvXFull));
#pragma unroll
          for (int q = 0; q < 3; ++q) product(two[q][0], two[q][1], two[q][2], opens && q == 0);
        }
        // (also after a wait that gave up: this commit covers what was issued)
        tc::mma_commit(bar(kCvEmpty + b));
        if (!ok) {
          fail();
          ++st;
          break;
        }
        if (st == win * kTcvStages + kTcvStages - 1 || st == nst - 1)
          tc::mma_commit(bar(kCvAccFull));
      }
      // the last stage's commit covers every MMA before it
      if (st)
        tc::mbar_wait_bounded(bar(kCvEmpty + ((st - 1) & 1)), ((st - 1) >> 1) & 1, kTcvWaitNs);
    }
  } else if (warp >= kTcvBuild) {
    // ------------------------------------------------------------- sums
    const int quarter = warp & 3, sw = warp - kTcvBuild;
    const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16);
    auto column = [&](int s) { return cov_column(quarter, sw >> 2, s, N); };
    // Sums of this lane's row, in three parts in their places of Cpart: two
    // that take the orders 0 to 3 exactly and one for the rest and what the
    // other two lose.  (Atomic adds so that nothing waits for them: a place
    // has one thread.)  Order 3 is summed in registers over a window, exactly:
    // in two parts where one could pass 2^24.
    float2 *sum = reinterpret_cast<float2 *>(a.Cpart + slice * a.stride) +
                  (size_t)sw * 8 * kTcvUnits * 32 + lane;
    float *rest = reinterpret_cast<float *>(a.Cpart + slice * a.stride) + 2 * kTcvPlaces +
                  (size_t)sw * 8 * kTcvUnits * 32 + lane;
    float third[8 * kTcvUnits];
#pragma unroll
    for (int u = 0; u < 8 * kTcvUnits; ++u) third[u] = 0.0f;
    bool ok = true, moved = false;
    auto wait = [&](int i, int parity) {
      const bool done = !*s_abort && tc::mbar_wait_bounded(bar(i), parity, a.wait_ns);
      ok = __all_sync(0xffffffffu, done);
      tc::fence_after_sync();
      return ok;
    };
    auto release = [&](int i) {
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) arrive(i);
    };
    for (int st = 0; st < nst && ok; ++st) {
      const int win = st / kTcvStages;
      // sums of order 3 that the window's other stages could take past 2^24
      // move to their places first (equal columns; others stay far below)
      if (st - win * kTcvStages == kTcvThird) {
        float most = 0.0f;
#pragma unroll
        for (int u = 0; u < 8 * kTcvUnits; ++u) most = fmaxf(most, fabsf(third[u]));
        moved = __any_sync(0xffffffffu, most > kTcvThirdMax);
        if (moved) {
#pragma unroll
          for (int s = 0; s < kTcvUnits; ++s) {
            if (column(s) < N) {
#pragma unroll
              for (int u = 0; u < 8; ++u) {
                float2 *to = &sum[(8 * s + u) * 32];
                const float2 old = win ? *to : make_float2(0.0f, 0.0f);
                const df t = two_sum(old.y, third[8 * s + u]);
                *to = make_float2(old.x, t.hi);
                if (win) atomicAdd(&rest[(8 * s + u) * 32], t.lo);  // (else 0)
                third[8 * s + u] = 0.0f;
              }
            }
          }
        }
      }
      for (int turn = 0; turn < 2; ++turn) {
        if (!wait(kCvXFull, turn)) break;
#pragma unroll
        for (int s = 0; s < kTcvUnits; ++s) {
          const int c0 = column(s);
          if (c0 < N) {
            uint32_t v[8];
            tmem_ld8(tlane + 3 * N + c0, v);
            tc::tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              if (turn) {
                third[8 * s + u] = __fadd_rn(third[8 * s + u], __uint_as_float(v[u]));
              } else if (st) {
                atomicAdd(&rest[(8 * s + u) * 32], __uint_as_float(v[u]));
              } else {
                rest[(8 * s + u) * 32] = __uint_as_float(v[u]);
              }
            }
          }
        }
        release(kCvXFree);
      }
      if (ok && (st == win * kTcvStages + kTcvStages - 1 || st == nst - 1)) {
        if (!wait(kCvAccFull, win & 1)) break;
#pragma unroll
        for (int s = 0; s < kTcvUnits; ++s) {
          const int c0 = column(s);
          if (c0 < N) {
            uint32_t v0[8], v1[8];
            tmem_ld8(tlane + c0, v0);
            tmem_ld8(tlane + N + c0, v1);
            tc::tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const df t = two_sum(__uint_as_float(v0[u]), __uint_as_float(v1[u]));
              v0[u] = __float_as_uint(t.hi);
              v1[u] = __float_as_uint(t.lo);
            }
            float2 old[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
              old[u] = win || moved ? sum[(8 * s + u) * 32] : make_float2(0.0f, 0.0f);
            uint32_t v2[8];
            tmem_ld8(tlane + 2 * N + c0, v2);
            tc::tmem_wait_ld();
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              float &r = third[8 * s + u];
              const df t = two_sum(__uint_as_float(v0[u]), __uint_as_float(v2[u]));
              const df q = two_sum(old[u].x, t.hi);
              const df m0 = two_sum(old[u].y, q.lo);
              const df m1 = two_sum(__uint_as_float(v1[u]), t.lo);
              const df m2 = two_sum(m0.hi, m1.hi);
              const df m3 = two_sum(m2.hi, r);
              r = 0.0f;
              sum[(8 * s + u) * 32] = make_float2(q.hi, m3.hi);
              atomicAdd(&rest[(8 * s + u) * 32],
                        __fadd_rn(__fadd_rn(m0.lo, m1.lo), __fadd_rn(m2.lo, m3.lo)));
            }
          }
        }
        release(kCvAccFree);
      }
    }
    if (!ok && lane == 0) fail();
  } else {
    // ------------------------------------------------------------ slices
    const df sqrt2 = {1.41421354f, 2.42032346e-08f};
    const int4 *s_rec = reinterpret_cast<const int4 *>(smem + kTcvRecOff);
    // the records of a stage, two stages ahead of its use (a slot is free once
    // the MMAs of the stage four before are done)
    auto fetch = [&](int st) {
      if (tid == 0 && st < nst) {
        const uint32_t bytes = 16u * (uint32_t)min(kTcvSamples, ns - st * kTcvSamples);
        tc::mbar_arrive_expect_tx(bar(kCvRec + (st & 3)), bytes);
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                tc::smem_u32(s_rec + (st & 3) * kTcvSamples)),
            "l"(a.samples + beg + st * kTcvSamples), "r"(bytes), "r"(bar(kCvRec + (st & 3)))
            : "memory");
      }
    };
    int fetched = min(nst, 2);
    fetch(0);
    fetch(1);
    for (int st = 0; st < nst; ++st) {
      const int b = st & 1;
      bool done = !*s_abort && (st < 2 || tc::mbar_wait_bounded(bar(kCvEmpty + b),
                                                                ((st >> 1) - 1) & 1, a.wait_ns));
      if (__all_sync(0xffffffffu, done)) {
        fetch(st + 2);
        fetched = min(nst, st + 3);
        done = tc::mbar_wait_bounded(bar(kCvRec + (st & 3)), (st >> 2) & 1, a.wait_ns);
      }
      if (!__all_sync(0xffffffffu, done)) {
        if (lane == 0) fail();
        break;
      }
      unsigned char *dst = smem + b * kTcvStage;
      const int nb = min(kTcvSamples, ns - st * kTcvSamples);
      const int ng = ((nb + 15) / 16) * 2;  // groups of eight samples that the MMAs read
      const int4 *rec = s_rec + (st & 3) * kTcvSamples;
      for (int task = tid; task < HJ * ng; task += 32 * kTcvBuild) {
        const int g = task / HJ, e = task - g * HJ, k = e / J;
        const float2 dv = __ldg(reinterpret_cast<const float2 *>(a.d) + (size_t)m * HJ + e);
        const int i1 = HJ + e - J;  // row of the imaginary part
        const float sr = ldexpf(1.0f, -s_exp[e]), si = k ? ldexpf(1.0f, -s_exp[i1]) : 0.0f;
        unsigned char *o0 = dst + e * 128 + ((g ^ (e & 7)) << 4);
        unsigned char *o1 = dst + i1 * 128 + ((g ^ (i1 & 7)) << 4);
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {  // four samples: eight bytes a slice
          const int i0 = 8 * g + 4 * half;
          // (past the end: the last sample, times zero)
          float4 ev[4];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            ev[u] = __ldg(a.E + (size_t)rec[min(i0 + u, nb - 1)].x * HJ + e);
          uint32_t re[2][kTcvSlices], im[2][kTcvSlices];
#pragma unroll
          for (int pair = 0; pair < 2; ++pair) {
            df yr[2], yi[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int i = i0 + 2 * pair + u;
              const int4 smp = rec[min(i, nb - 1)];
              const float4 f = s_tw[smp.y * H + k];
              df w = {__int_as_float(smp.z), __int_as_float(smp.w)};
              if (k) w = df_mul(w, sqrt2);
              const float4 q = ev[2 * pair + u];
              const df er = {q.x, q.z}, ei = {q.y, q.w}, c = {f.x, f.y}, sn = {f.z, f.w};
              // S_{-theta}: harmonic k times exp(+i k theta); k = 0 has no
              // imaginary part and angle factors 1 and 0
              yr[u] = df_add(df_sub(df_mul(er, c), df_mul(ei, sn)), df_mul_f(w, dv.x));
              yi[u] = df_add(df_add(df_mul(er, sn), df_mul(ei, c)), df_mul_f(w, dv.y));
              const float mr = i < nb ? sr : 0.0f, mi = i < nb ? si : 0.0f;
              yr[u].hi *= mr;
              yr[u].lo *= mr;
              yi[u].hi *= mi;
              yi[u].lo *= mi;
            }
            slice2(yr[0], yr[1], re[pair]);
            slice2(yi[0], yi[1], im[pair]);
          }
#pragma unroll
          for (int sl = 0; sl < kTcvSlices; ++sl) {
            *reinterpret_cast<uint2 *>(o0 + sl * kTcvSlice + 8 * half) = make_uint2(re[0][sl], re[1][sl]);
            if (k)
              *reinterpret_cast<uint2 *>(o1 + sl * kTcvSlice + 8 * half) = make_uint2(im[0][sl], im[1][sl]);
          }
        }
      }
      tc::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) arrive(kCvFull + b);
    }
    // records on their way land before the CTA gives up its memory
    if (tid == 0)
      for (int st = max(0, fetched - 4); st < fetched; ++st)
        tc::mbar_wait_bounded(bar(kCvRec + (st & 3)), (st >> 2) & 1, kTcvWaitNs);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// C_m[i][j] = sum over the partial sums in slice order (upper
// triangle), mirrored to the lower triangle.
__global__ void ksvd_cov_sum_kernel(const KsvdArgs a) {
  const int n = a.n;
  const size_t nn = (size_t)n * n, per_part = (size_t)a.M * nn;
  for (size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x; w < per_part;
       w += (size_t)gridDim.x * blockDim.x) {
    const size_t m = w / nn, ij = w - m * nn;
    const int i = (int)(ij / n), j = (int)(ij - (size_t)i * n);
    if (i > j) continue;
    double s = 0.0;
    for (int part = 0; part < a.split; ++part)
      s += a.Cpart[((size_t)part * a.M + m) * a.stride + ij];
    a.C[w] = s;
    if (i != j) a.C[m * nn + (size_t)j * n + i] = s;
  }
}

// The same for partial sums of the tensor-core kernel: a thread per place of
// their layout.  Double-float with a third part, FP64 at the end only: 2^k of a
// slice, |k| <= 102 by the range of the exponents, keeps all in range.
__global__ void ksvd_cov_pair_sum_kernel(const KsvdArgs a, int N) {
  const int n = a.n, J = a.J, HJ = a.H * a.J;
  for (size_t w = (size_t)blockIdx.x * blockDim.x + threadIdx.x; w < (size_t)a.M * kTcvPlaces;
       w += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(w / kTcvPlaces), q = (int)(w - (size_t)m * kTcvPlaces);
    const int lane = q & 31, idx = (q >> 5) % (8 * kTcvUnits), sw = (q >> 5) / (8 * kTcvUnits);
    const int quarter = (kTcvBuild + sw) & 3, row = quarter * 32 + lane;
    const int c0 = cov_column(quarter, sw >> 2, idx >> 3, N), c = c0 + (idx & 7);
    if (c0 >= N || row >= n || c >= n || ((c >> 5) == quarter && row > c)) continue;
    const int qr = cov_coord(row, J, HJ), qc = cov_coord(c, J, HJ);
    const int i = min(qr, qc), j = max(qr, qc);
    double other = 0.0;
    float hi = 0.0f, mid = 0.0f, lo = 0.0f;
#pragma unroll 4
    for (int part = 0; part < a.split; ++part) {
      const size_t slice = (size_t)part * a.M + m;
      const double *from = a.Cpart + slice * a.stride;
      const int state = a.state[slice];
      if (state == kCvPair) {
        const float2 v = reinterpret_cast<const float2 *>(from)[q];
        const float r = reinterpret_cast<const float *>(from)[2 * kTcvPlaces + q];
        const int k = a.expo[slice * 128 + row] + a.expo[slice * 128 + c];
        const float f = __int_as_float((k + 127) << 23);
        const df s0 = two_sum(hi, f * v.x), s1 = two_sum(mid, f * v.y), s2 = two_sum(s1.hi, s0.lo);
        hi = s0.hi;
        mid = s2.hi;
        lo = __fadd_rn(lo, __fadd_rn(f * r, __fadd_rn(s1.lo, s2.lo)));
      } else if (state == kCvFull64) {
        other += from[(size_t)i * n + j];
      } else if (state == kCvFailed) {
        other = __longlong_as_double(0x7ff8000000000000ll);
      }
    }
    const double s = ((double)hi + (double)mid) + ((double)lo + other);
    a.C[((size_t)m * n + i) * n + j] = s;
    if (i != j) a.C[((size_t)m * n + j) * n + i] = s;
  }
}

__device__ double block_sum(double v, double *red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;
}

// Leading eigenvector of C_m by FP64 power iteration from the old atom.
__global__ void __launch_bounds__(kEigThreads) ksvd_eig_kernel(const KsvdArgs a, int max_iter) {
  extern __shared__ __align__(16) double es[];
  const int m = blockIdx.x;
  const int n = a.n, J = a.J, H = a.H, HJ = H * J;
  if (a.count[m] == 0) {  // unused: the old atom, unless the reset replaces it
    for (int i = threadIdx.x; i < 2 * HJ; i += blockDim.x)
      a.new_coef[(size_t)m * HJ * 2 + i] = a.d[(size_t)m * HJ * 2 + i];
    return;
  }
  double *Cs = es;                 // n * n
  double *u = Cs + n * n;          // n
  double *v = u + n;               // n
  double *red = v + n;             // 32
  const double *Cm = a.C + (size_t)m * n * n;
  for (int i = threadIdx.x; i < n * n; i += blockDim.x) Cs[i] = Cm[i];
  // start: the old atom, packed
  for (int e = threadIdx.x; e < HJ; e += blockDim.x) {
    const int k = e / J;
    const float2 dv = reinterpret_cast<const float2 *>(a.d)[(size_t)m * HJ + e];
    if (k == 0) {
      u[e] = dv.x;
    } else {
      u[2 * e - J] = 1.4142135623730951 * dv.x;
      u[2 * e - J + 1] = 1.4142135623730951 * dv.y;
    }
  }
  __syncthreads();
  double lam_old = 0.0;
  for (int it = 0; it < max_iter; ++it) {
    double loc = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      double s = 0.0;
      for (int j = 0; j < n; ++j) s = fma(Cs[i * n + j], u[j], s);
      v[i] = s;
      loc = fma(s, s, loc);
    }
    const double nv2 = block_sum(loc, red);
    double dot = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) dot = fma(v[i], u[i], dot);
    const double lam = block_sum(dot, red);  // Rayleigh quotient (u unit)
    const double inv = nv2 > 0.0 ? 1.0 / sqrt(nv2) : 0.0;
    double dif = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const double nu = v[i] * inv;
      dif = fma(nu - u[i], nu - u[i], dif);
      u[i] = nu;
    }
    const double d2 = block_sum(dif, red);
    if (nv2 == 0.0) break;
    if (it > 0 && d2 < 1e-26 && fabs(lam - lam_old) <= 1e-15 * fabs(lam)) break;
    lam_old = lam;
  }
  __syncthreads();
  // sign: the largest-magnitude entry positive (first index on ties)
  if (threadIdx.x == 0) {
    int arg = 0;
    for (int i = 1; i < n; ++i)
      if (fabs(u[i]) > fabs(u[arg])) arg = i;
    red[0] = u[arg] < 0.0 ? -1.0 : 1.0;
  }
  __syncthreads();
  const double sg = red[0];
  float *out = a.new_coef + (size_t)m * HJ * 2;
  for (int e = threadIdx.x; e < HJ; e += blockDim.x) {
    const int k = e / J;
    if (k == 0) {
      out[2 * e] = (float)(sg * u[e]);
      out[2 * e + 1] = 0.0f;
    } else {
      out[2 * e] = (float)(sg * u[2 * e - J] * 0.7071067811865476);
      out[2 * e + 1] = (float)(sg * u[2 * e - J + 1] * 0.7071067811865476);
    }
  }
}

// The a.ntop patches of largest coding error, in descending error (ties:
// smaller index), each unit-normalised (one CTA of 1024 threads).
__global__ void ksvd_top_kernel(const KsvdArgs a) {
  __shared__ float bv[1024];
  __shared__ long long bi[1024];
  __shared__ float prev_e;
  __shared__ long long prev_i;
  __shared__ double nrm;
  const int J = a.J, HJ = a.H * J;
  __shared__ int ntop;
  if (threadIdx.x == 0) {
    prev_e = INFINITY;
    prev_i = -1;
    int n = a.ntop;
    if (a.top_needed) {  // the counts are final: as many entries as unused atoms
      int unused = 0;
      for (int m = 0; m < a.M; ++m) unused += a.count[m] == 0;
      n = min(n, unused);
      for (int t = n; t < a.ntop; ++t) a.top_idx[t] = -1;
    }
    ntop = n;
  }
  __syncthreads();
  for (int t = 0; t < ntop; ++t) {
    // the t-th entry is the largest (error, then smaller index) below the
    // previous one in that order
    const float pe = prev_e;
    const long long pi = prev_i;
    float best = -1.0f;
    long long bp = -1;
    for (int64_t p = threadIdx.x; p < a.P; p += blockDim.x) {
      const float e = a.err2[p];
      if (!(e < pe || (e == pe && p > pi))) continue;
      if (e > best) {
        best = e;
        bp = p;
      }
    }
    bv[threadIdx.x] = best;
    bi[threadIdx.x] = bp;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        const float o = bv[threadIdx.x + s];
        const long long oi = bi[threadIdx.x + s];
        if (o > bv[threadIdx.x] || (o == bv[threadIdx.x] && oi >= 0 &&
                                    (bi[threadIdx.x] < 0 || oi < bi[threadIdx.x]))) {
          bv[threadIdx.x] = o;
          bi[threadIdx.x] = oi;
        }
      }
      __syncthreads();
    }
    const long long p = bi[0];
    __syncthreads();
    if (threadIdx.x == 0) {
      if (p >= 0) {
        prev_e = bv[0];
        prev_i = p;
      }
      a.top_idx[t] = p;
      a.top_err[t] = p >= 0 ? bv[0] : -1.0f;
      double s2 = 0.0;
      if (p >= 0) {
        const float *xp = a.x + p * (int64_t)(2 * HJ);
        for (int e = 0; e < HJ; ++e) {
          const double re = xp[2 * e], im = e < J ? 0.0 : xp[2 * e + 1];
          s2 += (e < J ? 1.0 : 2.0) * (re * re + im * im);
        }
      }
      nrm = s2 > 0.0 ? 1.0 / sqrt(s2) : 0.0;
    }
    __syncthreads();
    float *out = a.top_vec + (size_t)t * HJ * 2;
    const float *xp = a.x + (p >= 0 ? p : 0) * (int64_t)(2 * HJ);
    for (int e = threadIdx.x; e < HJ; e += blockDim.x) {
      out[2 * e] = p >= 0 ? (float)(xp[2 * e] * nrm) : 0.0f;
      out[2 * e + 1] = (p >= 0 && e >= J) ? (float)(xp[2 * e + 1] * nrm) : 0.0f;
    }
    __syncthreads();
  }
}

// Unused atoms (count 0), in atom order, take the successive entries of the
// top list; atoms beyond the list (or beyond its valid entries) keep the
// eigen-kernel's output, which is the old atom for an atom with no samples.
__global__ void ksvd_reset_kernel(const KsvdArgs a) {
  const int HJ = a.H * a.J;
  int t = 0;
  for (int m = 0; m < a.M; ++m) {
    if (a.count[m] != 0) continue;
    if (t >= a.ntop || a.top_idx[t] < 0) break;
    const float *v = a.top_vec + (size_t)t * HJ * 2;
    float *out = a.new_coef + (size_t)m * HJ * 2;
    for (int i = threadIdx.x; i < 2 * HJ; i += blockDim.x) out[i] = v[i];
    ++t;
  }
}

}  // namespace

namespace {

// Checks shared by the entry points; fills the sizes of `a`.
int ksvd_setup(const rsc_dict *dict, int64_t P, int K, KsvdArgs &a) {
  if (!dict || P < 1 || K < 1 || K > kMaxK) return RSC_ERR_INVALID;
  if (P >= ((int64_t)1 << 31)) return RSC_ERR_UNSUPPORTED;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  if (dev != dict->device) return RSC_ERR_INVALID;
  a = KsvdArgs{};
  a.P = P;
  a.K = K;
  a.M = dict->M;
  a.J = dict->J;
  a.H = dict->H;
  a.R = dict->R;
  a.n = dict->J + 2 * dict->kmax * dict->J;
  if (a.n > kMaxPacked || a.M > kMaxAtomsKsvd) return RSC_ERR_UNSUPPORTED;
  a.err = dict->err;
  a.wait_ns = dict->wait_ns ? dict->wait_ns : kTcvWaitNs;
  a.d = dict->d;
  a.tw = dict->tw;
  return RSC_OK;
}

// Accumulation: sample lists, residuals, C (written here) and counts, and the
// top list of a.ntop patches; the per-patch scratch comes from one
// stream-ordered allocation freed on `st`.
int ksvd_accumulate(KsvdArgs &a, cudaStream_t st) {
  const int64_t P = a.P;
  const int M = a.M, n = a.n;
  a.nchunk = (int)((P + kFillChunk - 1) / kFillChunk);
  int nsm = 0, dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int HJ = a.H * a.J;
  const bool tensor = n <= kTcvMaxN && (size_t)a.R * a.H * 16 <= kTcvTwMax;
  // slices of about 512 samples or more, up to eight CTAs for every SM; eight
  // at least on the CUDA cores
  const int64_t per_atom = P * a.K / M, most = std::min<int64_t>((int64_t)8 * nsm / M, 32);
  a.split = (int)std::max<int64_t>(tensor ? 1 : 8, std::min(per_atom / 512, most));
  if (tensor) {
    // one CTA an SM: of the counts down to half of that, the one whose last
    // wave is fullest (M = 128: 7 slices, 5.9 waves, 1.63 ms an update of 200,000
    // patches; 9 slices, 7.6 waves, 1.66)
    auto fill = [&](int split) {
      const int ctas = M * split, waves = (ctas + nsm - 1) / nsm;
      return (double)ctas / ((double)waves * nsm);
    };
    const int upper = a.split;
    for (int c = upper - 1; c > upper / 2; --c)
      if (fill(c) > fill(a.split)) a.split = c;
  }
  a.stride = (size_t)n * n;
  if (tensor) a.stride = std::max(a.stride, (size_t)kTcvPlaces * 3 / 2);
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t bE = al((size_t)P * HJ * 16), bErr = al((size_t)P * 4),
               bOff = al((size_t)(M + 1) * 4), bCh = al((size_t)a.nchunk * M * 4),
               bSmp = al((size_t)P * a.K * 16), bCp = al((size_t)a.split * M * a.stride * 8),
               bSt = al((size_t)a.split * M * 4), bEx = al((size_t)a.split * M * 128 * 4);
  unsigned char *scratch = nullptr;
  cudaError_t e = rsc_scratch_alloc(reinterpret_cast<void **>(&scratch),
                                  bE + bErr + bOff + 2 * bCh + bSmp + bCp + (tensor ? bSt + bEx : 0), st);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return RSC_ERR_OOM;
  }
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  unsigned char *q = scratch;
  auto take = [&](size_t b) {
    unsigned char *r = q;
    q += b;
    return r;
  };
  a.E = reinterpret_cast<float4 *>(take(bE));
  a.err2 = reinterpret_cast<float *>(take(bErr));
  a.offset = reinterpret_cast<int *>(take(bOff));
  a.chunk_cnt = reinterpret_cast<int *>(take(bCh));
  a.chunk_base = reinterpret_cast<int *>(take(bCh));
  a.samples = reinterpret_cast<int4 *>(take(bSmp));
  a.Cpart = reinterpret_cast<double *>(take(bCp));
  a.state = tensor ? reinterpret_cast<int *>(take(bSt)) : nullptr;
  a.expo = tensor ? reinterpret_cast<int *>(take(bEx)) : nullptr;
  const size_t hist_smem = (size_t)M * 4;
  const bool fill_tw = (size_t)a.R * a.H * 16 <= kTcvTwMax;
  const size_t fill_smem =
      (size_t)kFillChunk * a.K * 20 + hist_smem + (fill_tw ? (size_t)a.R * a.H * 16 + 16 : 0);
  auto fill = fill_tw ? ksvd_fill_kernel<true> : ksvd_fill_kernel<false>;
  const size_t cov_smem = (size_t)2 * kCovBatch * (4 * ((n + 3) / 4) + 4) * 4;
  const size_t tc_smem = kTcvTwOff + (size_t)a.R * a.H * 16 + 1024;
  e = rsc_allow_smem(ksvd_cov_kernel, cov_smem);
  if (e == cudaSuccess) e = rsc_allow_smem(fill, fill_smem);
  if (e == cudaSuccess && tensor) e = rsc_allow_smem(ksvd_cov_tc_kernel, tc_smem);
  if (e == cudaSuccess) {
    ksvd_chunk_count_kernel<<<a.nchunk, 256, hist_smem, st>>>(a);
    ksvd_atom_scan_kernel<<<M, 256, 0, st>>>(a);
    ksvd_offset_kernel<<<1, 256, 0, st>>>(a);
    fill<<<a.nchunk, kFillThreads, fill_smem, st>>>(a);
    if (tensor) ksvd_cov_tc_kernel<<<M * a.split, kTcvThreads, tc_smem, st>>>(a, (n + 15) / 16 * 16);
    ksvd_cov_kernel<<<M * a.split, kCovThreads, cov_smem, st>>>(a);
    const size_t work = tensor ? (size_t)M * kTcvPlaces : (size_t)M * n * n;
    const unsigned gsum = (unsigned)std::min<size_t>((work + 255) / 256, (size_t)nsm * 8);
    if (tensor)
      ksvd_cov_pair_sum_kernel<<<gsum, 256, 0, st>>>(a, (n + 15) / 16 * 16);
    else
      ksvd_cov_sum_kernel<<<gsum, 256, 0, st>>>(a);
    if (a.ntop > 0) ksvd_top_kernel<<<1, 1024, 0, st>>>(a);
    e = cudaGetLastError();
  }
  int rc = e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
  const cudaError_t e2 = rsc_scratch_free(scratch, st);
  if (rc == RSC_OK && e2 != cudaSuccess) rc = rsc_cuda_fail(e2);
  return rc;
}

// New atoms from C, the counts and the top list.
int ksvd_finish(KsvdArgs &a, cudaStream_t st) {
  const int n = a.n;
  const size_t eig_smem = ((size_t)n * n + 2 * n + 32) * 8;
  cudaError_t e = rsc_allow_smem(ksvd_eig_kernel, eig_smem);
  if (e == cudaSuccess) {
    ksvd_eig_kernel<<<a.M, kEigThreads, eig_smem, st>>>(a, 5000);
    ksvd_reset_kernel<<<1, 256, 0, st>>>(a);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && a.n_used)
    e = cudaMemcpyAsync(a.n_used, a.count, (size_t)a.M * 4, cudaMemcpyDeviceToDevice, st);
  return e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
}

}  // namespace

extern "C" int rsc_ksvd_update(const rsc_dict *dict, const float *x, int64_t P, int32_t K,
                               const int32_t *atom, const int32_t *angle_idx, const double *coef,
                               float *new_coef, int32_t *n_used, void *stream) {
  RscRange nvtx_range("rsc_ksvd_update");
  if (!x || !atom || !angle_idx || !coef || !new_coef) return RSC_ERR_INVALID;
  KsvdArgs a;
  int rc = ksvd_setup(dict, P, K, a);
  if (rc != RSC_OK) return rc;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int M = a.M, n = a.n, HJ = a.H * a.J;
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t bC = al((size_t)M * n * n * 8), bCnt = al((size_t)M * 4),
               bTe = al(kTopMax * 4), bTi = al(kTopMax * 8), bTv = al((size_t)kTopMax * HJ * 8);
  unsigned char *scratch = nullptr;
  cudaError_t e = rsc_scratch_alloc(reinterpret_cast<void **>(&scratch), bC + bCnt + bTe + bTi + bTv,
                                  st);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return RSC_ERR_OOM;
  }
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  unsigned char *q = scratch;
  a.C = reinterpret_cast<double *>(q);
  q += bC;
  a.count = reinterpret_cast<int *>(q);
  q += bCnt;
  a.top_err = reinterpret_cast<float *>(q);
  q += bTe;
  a.top_idx = reinterpret_cast<int64_t *>(q);
  q += bTi;
  a.top_vec = reinterpret_cast<float *>(q);
  a.ntop = kTopMax;
  a.top_needed = 1;
  a.x = x;
  a.atom = atom;
  a.angle = angle_idx;
  a.coef = coef;
  a.new_coef = new_coef;
  a.n_used = n_used;
  rc = ksvd_accumulate(a, st);
  if (rc == RSC_OK) rc = ksvd_finish(a, st);
  e = rsc_scratch_free(scratch, st);
  if (rc == RSC_OK && e != cudaSuccess) rc = rsc_cuda_fail(e);
  return rc;
}

extern "C" int rsc_ksvd_accumulate(const rsc_dict *dict, const float *x, int64_t P, int32_t K,
                                   const int32_t *atom, const int32_t *angle_idx,
                                   const double *coef, double *C, int32_t *count, float *top_err,
                                   int64_t *top_idx, float *top_vec, int32_t ntop, void *stream) {
  RscRange nvtx_range("rsc_ksvd_accumulate");
  if (!x || !atom || !angle_idx || !coef || !C || !count) return RSC_ERR_INVALID;
  if (ntop < 0 || ntop > kTopMax || (ntop > 0 && (!top_err || !top_idx || !top_vec)))
    return RSC_ERR_INVALID;
  KsvdArgs a;
  int rc = ksvd_setup(dict, P, K, a);
  if (rc != RSC_OK) return rc;
  a.x = x;
  a.atom = atom;
  a.angle = angle_idx;
  a.coef = coef;
  a.C = C;
  a.count = count;
  a.ntop = ntop;
  a.top_err = top_err;
  a.top_idx = top_idx;
  a.top_vec = top_vec;
  return ksvd_accumulate(a, reinterpret_cast<cudaStream_t>(stream));
}

extern "C" int rsc_ksvd_finish(const rsc_dict *dict, const double *C, const int32_t *count,
                               const int64_t *top_idx, const float *top_vec, int32_t ntop,
                               float *new_coef, int32_t *n_used, void *stream) {
  RscRange nvtx_range("rsc_ksvd_finish");
  if (!dict || !C || !count || !new_coef) return RSC_ERR_INVALID;
  if (ntop < 0 || ntop > kTopMax || (ntop > 0 && (!top_idx || !top_vec))) return RSC_ERR_INVALID;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  if (dev != dict->device) return RSC_ERR_INVALID;
  KsvdArgs a{};
  a.M = dict->M;
  a.J = dict->J;
  a.H = dict->H;
  a.R = dict->R;
  a.n = dict->J + 2 * dict->kmax * dict->J;
  if (a.n > kMaxPacked) return RSC_ERR_UNSUPPORTED;
  a.d = dict->d;
  a.tw = dict->tw;
  a.C = const_cast<double *>(C);
  a.count = const_cast<int *>(count);
  a.ntop = ntop;
  a.top_idx = const_cast<int64_t *>(top_idx);
  a.top_vec = const_cast<float *>(top_vec);
  a.new_coef = new_coef;
  a.n_used = n_used;
  return ksvd_finish(a, reinterpret_cast<cudaStream_t>(stream));
}
