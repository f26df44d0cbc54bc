// reconstruct.cu -- the way back from codes to patches: step 4 of the
// proposed algorithm (Sec. II-E: the learned dictionary returns to the patch
// domain as D = Phi D_hat) and the reconstruction of coded patches.
//
// rsc_reconstruct: x_hat_p = sum_i a_i S_{r_i} d_{m_i} for each patch's code
//   (steering of Eq. (Sr): harmonic k of an atom times exp(-i k 2 pi r / R)),
//   from the dictionary's FP32 atoms and its double-float steering factors;
//   every entry its FP64 value rounded to FP32 (to 2^-24 + 2^-27 of itself).
// rsc_synthesize: pixels = Phi x_hat over the circular patch, a tiled FP32
//   matrix product with the basis's real synthesis matrix (rows in the half
//   spectrum's order, the packing weights folded in).
#include <algorithm>

#include "df.cuh"
#include "rsc_internal.h"
#include "rsc_trace.h"

namespace {

// Two FP32 operations in one instruction (each rounded as its scalar form).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 halves(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// ------------------------------------------------------------ reconstruct
//
// Bound by FP32 issue: 32 operations per term and entry, two to an
// instruction.  A warp takes a tile of patches, a lane up to kRecEntries
// entries of one patch's harmonic: it forms the steered weights
// a_i e^{-i k theta_i} in double-float once per term and applies them to its
// entries' FP32 atoms, accumulating to about 60 bits.
// 10^6 patches of 54 entries, K = 5: 0.52 ms (the operations themselves 0.21
// at the FP32 peak; a two-element FMA takes 2.3 cycles, so it saves issue
// slots and no time on the pipe), against 7.0 ms for FP64 throughout (15
// operations per term on a pipe of 1/64 of the FP32 rate, every factor formed
// again for every entry); the memory floor is 75 us.  With two floats for an
// accumulator (48 bits, 0.42 ms) entries that cancel to 2^-20 of the weights
// came out up to 7 x 2^-24 off.  Four entries a lane 0.73 ms, a third block an
// SM (80 registers, spills) 0.54; of the time 5% are the entries in FP64.
constexpr int kRecThreads = 256;
constexpr int kRecTile = 32;   // patches per warp and tile
constexpr int kRecEntries = 6;

// Accumulators of products w d, |sum| < 2^(E-1) throughout: acc starts at
// 1.5 2^E, so that every partial sum stays in [2^E, 2^(E+1)) and acc holds it
// rounded to a multiple of 2^(E-23), exactly tracked: acc - t and the
// remainder l = w.hi d - (t - acc) (one FMA) are exact.  The remainders, up to
// 2K of 2^(E-24), are summed the same way from 1.5 2^(E-17), and r collects what
// that leaves and the lo parts: eight operations instead of the eleven of
// TwoProd + TwoSum.  The weights are off by 2^-46 of themselves and r, below
// 2^(E-25), is rounded 4K times: (K + 1) 2^(E-48) in all.
__device__ __forceinline__ void acc_prod2(f32x2 &acc, f32x2 &c, f32x2 &r, f32x2 whi, f32x2 wlo,
                                          f32x2 d) {
  const f32x2 minus1 = pack2(-1.0f, -1.0f);
  const f32x2 t = fma2(whi, d, acc);
  const f32x2 l = fma2(whi, d, fma2(t, minus1, acc));
  acc = t;
  const f32x2 u = add2(c, l);
  r = fma2(wlo, d, add2(r, add2(l, fma2(u, minus1, c))));
  c = u;
}

// One entry in FP64 straight from the code, for patches and entries outside
// the range of acc_prod2 (weights that are not finite or far from 1; an entry
// that cancels so far that the accumulators' error would show).
__device__ __forceinline__ float2 reconstruct_entry(const float *__restrict__ d,
                                                 const float *__restrict__ tw, int H, int HJ, int R,
                                                 int K, const int32_t *__restrict__ atom,
                                                 const int32_t *__restrict__ angle_idx,
                                                 const double *__restrict__ coef, int64_t p, int e,
                                                 int k) {
  double re = 0.0, im = 0.0;
#pragma unroll 1
  for (int i = 0; i < K; ++i) {
    const int m = atom[p * K + i];
    if (m < 0) continue;
    const int r = angle_idx[p * K + i];
    const double a = coef[p * K + i];
    const float2 dv = reinterpret_cast<const float2 *>(d)[(int64_t)m * HJ + e];
    const double dr = dv.x, di = k ? (double)dv.y : 0.0;
    const double c = (double)tw[(0 * H + k) * R + r] + (double)tw[(1 * H + k) * R + r];
    const double s = (double)tw[(2 * H + k) * R + r] + (double)tw[(3 * H + k) * R + r];
    re += a * (dr * c + di * s);
    im += a * (di * c - dr * s);
  }
  return make_float2((float)re, k ? (float)im : 0.0f);
}

// PAIRS: entries move two at a time in 16-byte pieces (J even, 16-byte
// aligned output).  A harmonic's J entries are split over nsub lanes, `per`
// each (the last fewer; even with PAIRS).
template <bool PAIRS>
__global__ void __launch_bounds__(kRecThreads, 2)
    reconstruct_kernel(const float *__restrict__ d, const float *__restrict__ tw, int H, int J,
                       int R, int64_t P, int K, int tile, int nsub, int per,
                       const int32_t *__restrict__ atom, const int32_t *__restrict__ angle_idx,
                       const double *__restrict__ coef, float *__restrict__ out) {
  extern __shared__ __align__(16) unsigned char rec_smem[];
  const int HJ = H * J, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  constexpr int nw = kRecThreads / 32;
  float4 *s_tw = reinterpret_cast<float4 *>(rec_smem);  // [R][H] cos hi, lo, sin hi, lo
  int4 *s_a = reinterpret_cast<int4 *>(s_tw + R * H) + w * tile * K;  // weight hi, lo, angle row, atom row
  for (int i = threadIdx.x; i < R * H; i += kRecThreads) {
    const int k = i / R, r = i - k * R;
    s_tw[r * H + k] = make_float4(tw[(0 * H + k) * R + r], tw[(1 * H + k) * R + r],
                                  tw[(2 * H + k) * R + r], tw[(3 * H + k) * R + r]);
  }
  __syncthreads();
  const int64_t ntiles = (P + tile - 1) / tile;
  const int items = H * nsub;
  for (int64_t t = (int64_t)blockIdx.x * nw + w; t < ntiles; t += (int64_t)gridDim.x * nw) {
    const int64_t p0 = t * tile;
    const int np = (int)min((int64_t)tile, P - p0);
    __syncwarp();  // the previous tile is read
    for (int i = lane; i < np * K; i += 32) {
      const int m = __ldg(atom + p0 * K + i), r = __ldg(angle_idx + p0 * K + i);
      const double a = __ldg(coef + p0 * K + i);
      const df v = m < 0 ? df{0.0f, 0.0f} : df_from_d(a);
      s_a[i] = make_int4(__float_as_int(v.hi), __float_as_int(v.lo), m < 0 ? 0 : r * H,
                         m < 0 ? 0 : m * HJ);
    }
    __syncwarp();
    // lane l: 1.5 2^E of patch l (0: FP64; negative: nothing coded, zeros)
    float sigl = 0.0f;
    if (lane < np) {
      float sum = 0.0f;
      for (int q = 0; q < K; ++q) sum += fabsf(__int_as_float(s_a[lane * K + q].x));
      // atoms have norm 1 to 1e-4: no entry of a partial sum exceeds 1.01 sum
      int E = 0;
      (void)frexpf(1.01f * sum, &E);
      if (sum > 1e-20f && sum < 1e25f) sigl = 1.5f * exp2f((float)(E + 1));  // NaN: 0
      if (sum == 0.0f) sigl = -1.5f;
    }
    for (int base = 0; base < np * items; base += 32) {
      const int it = base + lane;
      const int pl = min(it / items, np - 1), ks = it - pl * items;
      const float sig = __shfl_sync(0xffffffffu, sigl, pl);
      if (it >= np * items) continue;
      const int k = ks / nsub, e0 = k * J + (ks - k * nsub) * per;
      const int cnt = min(per, (k + 1) * J - e0);
      f32x2 acc[kRecEntries], cor[kRecEntries], rem[kRecEntries];
      const float sig2 = sig * 7.62939453125e-6f;  // 1.5 2^(E-17)
#pragma unroll
      for (int j = 0; j < kRecEntries; ++j) {
        acc[j] = pack2(sig, sig);
        cor[j] = pack2(sig2, sig2);
        rem[j] = 0;
      }
      if (sig > 0.0f) {
        const float2 *dp = reinterpret_cast<const float2 *>(d) + e0;
        const int4 *ap = s_a + pl * K;
#pragma unroll 1
        for (int i = 0; i < K; ++i) {
          const int4 a4 = ap[i];
          const float4 f = s_tw[a4.z + k];
          float2 dv[kRecEntries];
#pragma unroll
          for (int j = 0; j < kRecEntries; j += PAIRS ? 2 : 1) {
            if constexpr (PAIRS) {
              float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
              if (j < cnt) q = __ldg(reinterpret_cast<const float4 *>(dp + a4.w + j));
              dv[j] = make_float2(q.x, q.y);
              dv[j + 1] = make_float2(q.z, q.w);
            } else {
              dv[j] = make_float2(0.f, 0.f);
              if (j < cnt) dv[j] = __ldg(dp + a4.w + j);
            }
          }
          const df a = {__int_as_float(a4.x), __int_as_float(a4.y)};
          const df wc = df_mul(a, df{f.x, f.y}), ws = df_mul(a, df{f.z, f.w});
          const f32x2 ch = pack2(wc.hi, wc.hi), cl = pack2(wc.lo, wc.lo);
          const f32x2 sh = pack2(ws.hi, -ws.hi), sl = pack2(ws.lo, -ws.lo);
#pragma unroll
          for (int j = 0; j < kRecEntries; ++j) {
            // (re, im) += a c (dr, di) + (a s, -a s) (di, dr); k = 0 holds
            // real numbers: the table's sine and the atoms' di are 0 there
            acc_prod2(acc[j], cor[j], rem[j], ch, cl, pack2(dv[j].x, dv[j].y));
            acc_prod2(acc[j], cor[j], rem[j], sh, sl, pack2(dv[j].y, dv[j].x));
          }
        }
      }
      // sig = 1.5 2^E: entries below (K + 1) 2^(E-21) would show more than 2^-27
      // of themselves of the accumulators' error, beside the one rounding to
      // FP32, and are formed in FP64 (the line lies at 6 to 12 x 10^-6 sum |a_i|
      // for K = 5: about 0.01% of the values of random atoms are below it)
      const float tiny = sig * ((float)(K + 1) * 3.178914388e-7f);  // (K + 1) 2^-21 / 1.5
      float2 o[kRecEntries];
      unsigned low = 0;
#pragma unroll
      for (int j = 0; j < kRecEntries; ++j) {
        const float2 h = halves(add2(acc[j], pack2(-sig, -sig)));
        const float2 c = halves(add2(cor[j], pack2(-sig2, -sig2))), q = halves(rem[j]);
        const df x = two_sum(h.x, c.x), y = two_sum(h.y, c.y);
        o[j] = make_float2(__fadd_rn(x.hi, __fadd_rn(x.lo, q.x)),
                           __fadd_rn(y.hi, __fadd_rn(y.lo, q.y)));
        // (an exact zero is what it is)
        const bool lx = fabsf(o[j].x) < tiny && (x.hi != 0.0f || q.x != 0.0f);
        const bool ly = fabsf(o[j].y) < tiny && (y.hi != 0.0f || q.y != 0.0f);
        if (lx || ly || sig == 0.0f) low |= 1u << j;
      }
      low &= (1u << cnt) - 1u;
      while (low) {
        const int j = __ffs(low) - 1;
        low &= low - 1;
        const float2 q = reconstruct_entry(d, tw, H, HJ, R, K, atom, angle_idx, coef, p0 + pl,
                                           e0 + j, k);
#pragma unroll
        for (int u = 0; u < kRecEntries; ++u)
          if (u == j) o[u] = q;
      }
      float2 *op = reinterpret_cast<float2 *>(out) + (p0 + pl) * HJ + e0;
#pragma unroll
      for (int j = 0; j < kRecEntries; j += PAIRS ? 2 : 1) {
        if (j < cnt) {
          if constexpr (PAIRS)
            *reinterpret_cast<float4 *>(op + j) = make_float4(o[j].x, o[j].y, o[j + 1].x, o[j + 1].y);
          else
            op[j] = o[j];
        }
      }
    }
  }
}

template <bool PAIRS>
cudaError_t launch_reconstruct(const rsc_dict *dict, int dev, int64_t P, int K, const int32_t *atom,
                               const int32_t *angle_idx, const double *coef, float *out,
                               cudaStream_t st) {
  const int H = dict->H, J = dict->J, R = dict->R;
  constexpr int nw = kRecThreads / 32;
  int nsm = 0;
  cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // few patches: smaller tiles, so that every SM has warps to run
  int tile = kRecTile;
  while (tile > 1 && (P + tile - 1) / tile < (int64_t)nsm * nw) tile >>= 1;
  const int nsub = (J + kRecEntries - 1) / kRecEntries;
  int per = (J + nsub - 1) / nsub;
  if (PAIRS) per = (per + 1) & ~1;
  const size_t smem = (size_t)R * H * 16 + (size_t)nw * tile * K * 16;
  auto kern = reconstruct_kernel<PAIRS>;
  e = rsc_allow_smem(kern, smem);
  int per_sm = 1;
  const int64_t blk = (int64_t)tile * nw, blocks = (P + blk - 1) / blk;
  if (e == cudaSuccess && blocks > nsm)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRecThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t cap = (int64_t)nsm * std::max(per_sm, 1);
  kern<<<(unsigned)std::min(blocks, cap), kRecThreads, smem, st>>>(
      dict->d, dict->tw, H, J, R, P, K, tile, nsub, per, atom, angle_idx, coef, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------- synthesize
//
// C[P][npix] = coef[P][nk] X[nk][npix], FP32 FMA in the order of the half
// spectrum (the error of the plain sum; the tensor cores' accumulation is
// coarser).  A block takes 16 RT rows and up to 128 pixels; thread (tx, ty)
// of ct x 16 holds RT x 8 outputs.  Both operands stream through shared memory
// in chunks of kc coordinates with cp.async, two chunks in flight.  ct, the
// threads across the pixels, is chosen so that the last tile of pixels is full
// (97 pixels: 13 x 8 = 104).
// The result leaves through shared memory, so that its rows are written with
// full lines.
// 10^6 patches of 102 coordinates to 97 pixels: 0.68 ms (issue at 65%: seven
// warps share four schedulers), against 4.0 ms for one output per thread (an X
// and a coefficient load for every FMA); the FP32 floor is 0.25, the memory
// floor 0.12.  Two-element FMAs took 0.80 ms (each takes 2.3 cycles on this
// part), lanes along the pixels instead of the rows 0.80 (13 groups of pixels
// meet banks twice).
constexpr int kSynK = kSynPad;  // longest chunk (coordinates)
constexpr int kSynRows = 16;    // threads down the rows

// A chunk of coefficients is kept transposed, [k][16 RT rows]; groups of four
// rows are permuted by k so that the transposing copies meet no bank twice.
__device__ __forceinline__ int syn_a_group(int kq, int group) {
  return group ^ (kq & 7);
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const float *src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

template <int RT>
__global__ void __launch_bounds__(256, RT == 8 ? 2 : 4)
    synthesize_kernel(const float *__restrict__ X, int nk, int ldx, int npix, int J, int kc,
                      int64_t P, const float *__restrict__ coef, int ct, int ntn, bool vec,
                      float *__restrict__ pix) {
  constexpr int BM = kSynRows * RT;
  extern __shared__ __align__(16) float syn_smem[];
  const int BN = 8 * ct, nthr = kSynRows * ct;
  const int stage = kc * (BM + BN), kq4 = kc / 4, inv = 65536 / kq4 + 1;
  const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(syn_smem));
  // rows vary fastest over the lanes: a warp reads 16 different row groups and
  // two pixel groups, which meets no bank twice
  const int tid = threadIdx.x, ty = tid % kSynRows, tx = tid / kSynRows;
  const int64_t ntiles = (P + BM - 1) / BM * ntn;
  const int nchunk = (nk + kc - 1) / kc;
  for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int64_t p0 = t / ntn * BM;
    const int n0 = (int)(t % ntn) * BN, nn = min(BN, npix - n0);
    const int rows = (int)min((int64_t)BM, P - p0);
    const float *cp0 = coef + p0 * nk;
    auto load = [&](int c) {
      const uint32_t sa = s0 + (uint32_t)((c & 1) * stage) * 4, sx = sa + kc * BM * 4;
      const int k0 = c * kc;
      // coefficients: kc / 4 threads along a row's chunk, 4 values each
      for (int i = tid; i < BM * kq4; i += nthr) {
        const int row = (i * inv) >> 16, kq = i - row * kq4, g = k0 + 4 * kq;  // i < 2^11
        const uint32_t dst =
            sa + 16 * (kq * BM + syn_a_group(kq, row >> 2)) + 4 * (row & 3);
        const float *src = cp0 + row * nk + g;
        if (row < rows && g >= 2 * J && g + 4 <= nk) {
#pragma unroll
          for (int u = 0; u < 4; ++u) cp_async4(dst + 4 * BM * u, src + u, true);
        } else {
          // rows past the end, coordinates past nk and the imaginary parts of
          // k = 0 read as zero
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const bool in = row < rows && g + u < nk && !(g + u < 2 * J && (u & 1));
            cp_async4(dst + 4 * BM * u, in ? src + u : coef, in);
          }
        }
      }
      // X is padded with zeros to whole tiles of BN columns and by kSynK rows
      const float *xs = X + (size_t)k0 * ldx + n0;
      for (int i = tid; i < kc * 2 * ct; i += nthr) {
        const int k = i / (2 * ct), q = i - k * 2 * ct;
        cp_async16(sx + 4 * (k * BN + 4 * q), xs + (size_t)k * ldx + 4 * q);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[RT][8];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    load(0);
    for (int c = 0; c < nchunk; ++c) {
      if (c + 1 < nchunk) {
        load(c + 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      const float *sa = syn_smem + (c & 1) * stage, *sx = sa + kc * BM + 8 * tx;
#pragma unroll 1
      for (int kq = 0; kq < kq4; ++kq, sa += 4 * BM, sx += 4 * BN) {
        const float *g0, *g1 = nullptr;
        if constexpr (RT == 8) {
          g0 = sa + 4 * syn_a_group(kq, ty);
          g1 = sa + 4 * syn_a_group(kq, 16 + ty);
        } else {
          g0 = sa + 4 * syn_a_group(kq, ty >> 1) + 2 * (ty & 1);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          float a[RT], b[8];
          if constexpr (RT == 8) {
            const float4 a0 = *reinterpret_cast<const float4 *>(g0 + u * BM);
            const float4 a1 = *reinterpret_cast<const float4 *>(g1 + u * BM);
            a[0] = a0.x; a[1] = a0.y; a[2] = a0.z; a[3] = a0.w;
            a[4] = a1.x; a[5] = a1.y; a[6] = a1.z; a[7] = a1.w;
          } else {
            const float2 a0 = *reinterpret_cast<const float2 *>(g0 + u * BM);
            a[0] = a0.x; a[1] = a0.y;
          }
          const float4 b0 = *reinterpret_cast<const float4 *>(sx + u * BN);
          const float4 b1 = *reinterpret_cast<const float4 *>(sx + u * BN + 4);
          b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w;
          b[4] = b1.x; b[5] = b1.y; b[6] = b1.z; b[7] = b1.w;
#pragma unroll
          for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
      }
      __syncthreads();
    }
    // ---- out through shared memory: the tile's rows of nn pixels, packed
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int row = RT == 8 ? (i < 4 ? 4 * ty + i : 60 + 4 * ty + i) : 2 * ty + i;
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (8 * tx + j < nn) syn_smem[row * nn + 8 * tx + j] = acc[i][j];
    }
    __syncthreads();
    if (ntn == 1) {  // whole rows: the tile is one contiguous piece
      float *o = pix + p0 * npix;
      const int total = rows * npix, quads = vec ? total / 4 : 0;
      for (int i = tid; i < quads; i += nthr)
        reinterpret_cast<float4 *>(o)[i] = reinterpret_cast<const float4 *>(syn_smem)[i];
      for (int i = 4 * quads + tid; i < total; i += nthr) o[i] = syn_smem[i];
    } else {
      const int lane = tid & 31, w = tid >> 5, nw = nthr >> 5;
      for (int r = w; r < rows && w < nw; r += nw)
        for (int j = lane; j < nn; j += 32) pix[(p0 + r) * npix + n0 + j] = syn_smem[r * nn + j];
    }
    __syncthreads();
  }
}

// One output per thread, its coordinates in the same order (the same result,
// bit for bit), for calls of a block an SM at most: their time is one chain of
// loads, where the tiles also fill shared memory and meet at barriers.  A call
// of one patch of 349 pixels and 250 coordinates 15.6 us against 24.5, of 100
// 16.3 against 24.5; of 300 patches of 97 pixels and 102 coordinates 11.7
// against 13.9, of 1,000 (three blocks an SM) 14.7 against 14.2.  Eight loads
// ahead: with four 20.1 us for the first of these, with sixteen 16.4.
__global__ void __launch_bounds__(256)
    synthesize_small_kernel(const float *__restrict__ X, int nk, int ldx, int npix, int J,
                            int total, const float *__restrict__ coef, float *__restrict__ pix) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= total) return;
  const int p = i / npix;
  const float *c = coef + p * nk, *x = X + (i - p * npix);
  float acc = 0.0f;
#pragma unroll 8
  for (int j = 0; j < J; ++j) acc = fmaf(x[(int64_t)(2 * j) * ldx], c[2 * j], acc);
#pragma unroll 8
  for (int g = 2 * J; g < nk; ++g) acc = fmaf(x[(int64_t)g * ldx], c[g], acc);
  pix[i] = acc;
}

template <int RT>
cudaError_t launch_synthesize(const rsc_basis_view &v, int dev, int64_t P, const float *coef,
                              float *pixels, cudaStream_t st) {
  constexpr int BM = kSynRows * RT;
  const int ct = v.syn_cols / 8, ntn = (v.npix + v.syn_cols - 1) / v.syn_cols;
  // chunk length: the one that pads the coordinates least
  int kc = kSynK;
  for (int c = kSynK - 4; c >= 24; c -= 4)
    if ((v.nout + c - 1) / c * c < (v.nout + kc - 1) / kc * kc) kc = c;
  const size_t smem = std::max((size_t)2 * kc * (BM + 8 * ct), (size_t)BM * 8 * ct) * 4;
  auto kern = synthesize_kernel<RT>;
  cudaError_t e = rsc_allow_smem(kern, smem);
  int nsm = 0, per_sm = 1;
  const int64_t tiles = (P + BM - 1) / BM * ntn;
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && tiles > nsm)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSynRows * ct, smem);
  if (e != cudaSuccess) return e;
  const int64_t cap = (int64_t)nsm * std::max(per_sm, 1);
  const bool vec = (reinterpret_cast<uintptr_t>(pixels) & 15) == 0;
  kern<<<(unsigned)std::min(tiles, cap), kSynRows * ct, smem, st>>>(
      v.X, v.nout, v.ldx, v.npix, v.J, kc, P, coef, ct, ntn, vec, pixels);
  return cudaGetLastError();
}

}  // namespace

extern "C" int rsc_reconstruct(const rsc_dict *dict, int64_t P, int32_t K, const int32_t *atom,
                               const int32_t *angle_idx, const double *coef, float *out,
                               void *stream) {
  RscRange nvtx_range("rsc_reconstruct");
  if (!dict || P < 0 || K < 1 || K > kMaxK) return RSC_ERR_INVALID;
  if (P == 0) return RSC_OK;
  if (!atom || !angle_idx || !coef || !out) return RSC_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(out) & 7) || (reinterpret_cast<uintptr_t>(coef) & 7) ||
      (reinterpret_cast<uintptr_t>(atom) & 3) || (reinterpret_cast<uintptr_t>(angle_idx) & 3))
    return RSC_ERR_INVALID;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  if (dev != dict->device) return RSC_ERR_INVALID;
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const bool pairs = dict->J % 2 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  e = pairs ? launch_reconstruct<true>(dict, dev, P, K, atom, angle_idx, coef, out, st)
            : launch_reconstruct<false>(dict, dev, P, K, atom, angle_idx, coef, out, st);
  return e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
}

extern "C" int rsc_synthesize(const rsc_basis *basis, const float *coef, int64_t P, float *pixels,
                              void *stream) {
  RscRange nvtx_range("rsc_synthesize");
  if (!basis || P < 0) return RSC_ERR_INVALID;
  if (P == 0) return RSC_OK;
  if (!coef || !pixels) return RSC_ERR_INVALID;
  rsc_basis_view v;
  int rc = rsc_basis_internals(basis, &v);
  if (rc != RSC_OK) return rc;
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return rsc_cuda_fail(e);
  if (dev != v.device) return RSC_ERR_INVALID;
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (P <= 256 * nsm / v.npix) {
    const int total = (int)P * v.npix;
    synthesize_small_kernel<<<(total + 255) / 256, 256, 0, st>>>(v.X, v.nout, v.ldx, v.npix, v.J,
                                                                 total, coef, pixels);
    e = cudaGetLastError();
    return e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
  }
  // tiles of 128 patches when they fill the SMs, else of 32
  e = (P + 127) / 128 >= nsm ? launch_synthesize<8>(v, dev, P, coef, pixels, st)
                             : launch_synthesize<2>(v, dev, P, coef, pixels, st);
  return e == cudaSuccess ? RSC_OK : rsc_cuda_fail(e);
}
