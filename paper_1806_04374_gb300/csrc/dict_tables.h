// dict_tables.h -- device memory of a dictionary's tables for the refine
// (rsc_capi.cu): what each takes, and what is left out when the allocator
// refuses it.  Host code only.
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>

constexpr size_t kGramMax = (size_t)1 << 28;  // largest Gram table of the refine (bytes)

// Bytes of the parts of the one allocation, in this order.
struct RefineTables {
  size_t xgram, anorm, rows, gram;  // gram 0: above kGramMax, entries from xgram
};

inline RefineTables plan_refine_tables(int M, int H, int R, int Rr, int L) {
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t m = (size_t)M, gram = m * m * R * 8;
  return RefineTables{al(m * m * H * 16), al(m * 8), al((size_t)Rr * m * L * 8),
                      gram <= kGramMax ? gram : 0};
}

// Takes the tables in one allocation; refused, without the Gram table (the
// refine then forms its entries from xgram), and refused again, without the
// rows (no FP16 coding by rsc_encode then, but everything that needs neither:
// the FP32 paths, rsc_encode_noalloc, the K-SVD update, the way back).  The
// parts that were left out are 0 in `t` afterwards.
template <class Alloc>  // cudaError_t alloc(void **, size_t)
cudaError_t alloc_refine_tables(RefineTables &t, Alloc alloc, void **base) {
  cudaError_t e = alloc(base, t.xgram + t.anorm + t.rows + t.gram);
  if (e == cudaErrorMemoryAllocation && t.gram) {
    t.gram = 0;
    e = alloc(base, t.xgram + t.anorm + t.rows);
  }
  if (e == cudaErrorMemoryAllocation) {
    t.gram = t.rows = 0;
    e = alloc(base, t.xgram + t.anorm);
  }
  return e;
}
