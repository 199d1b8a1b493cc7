// The mixed Newton solve's triangular solves and refinement (refine.cu):
// explicit inverses of the FP32 factor's diagonal blocks, and one launch that
// runs every refinement step.
#pragma once
#include "internal.h"

namespace spsvm {

// FP64 -> FP32 with round to nearest even, from the IEEE-754 encodings with
// integer operations only (GB300 issues the FP64 conversion instruction at
// its FP64 rate).  Results below the FP32 normal range flush to signed zero
// and results above it become infinity (an FP32 factor then breaks down and
// the caller falls back to FP64).
__device__ __forceinline__ float f64_to_f32_rn(double v) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  const unsigned sign = (unsigned)(u >> 32) & 0x80000000u;
  const int e = (int)((u >> 52) & 0x7ff) - 1023 + 127;
  const unsigned long long man = u & 0xfffffffffffffull;
  if ((int)((u >> 52) & 0x7ff) == 0x7ff)   // inf / nan
    return __uint_as_float(sign | 0x7f800000u | (man ? 0x400000u : 0u));
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7f800000u);
  const unsigned m23 = (unsigned)(man >> 29);
  const unsigned rem = (unsigned)(man & 0x1fffffffu);
  const unsigned up = (rem > 0x10000000u) || (rem == 0x10000000u && (m23 & 1u));
  unsigned bits = ((unsigned)e << 23) + m23 + up;   // a carry moves into the exponent
  if (bits >= 0x7f800000u) bits = 0x7f800000u;
  return __uint_as_float(sign | bits);
}

// The refinement's result: stop (0 steps used up, 1 backward error reached, 2
// stagnation, 3 not finite, 4 the FP32 factorisation broke down), steps taken
// and the last backward error.
struct RefineState {
  int32_t stop, iters;
  double be;
};

// Diagonal blocks of the solve: inv_size(m) rows (a power of two times 64, at
// most 1,024), the last one short.  W holds each block's inverse (lower,
// row-major, pitch inv_size), WT its transpose, T the products in between.
constexpr int64_t kInvMax = 1024;
inline int64_t inv_size(int64_t m) {
  int64_t s = 64;
  while (s < m && s < kInvMax) s *= 2;
  return s;
}
inline int64_t inv_elems(int64_t m) { return ceil_div(m, inv_size(m)) * inv_size(m) * inv_size(m); }
inline int64_t inv_temp_elems(int64_t m) { return ceil_div(m, inv_size(m)) * inv_size(m) * inv_size(m) / 4; }

// Inverses of the diagonal blocks of the lower factor L (m rows, pitch ldl, a
// multiple of 4, 16-byte aligned).  Also stores the 64 x 64 blocks' inverses
// transposed in their upper triangles.
int launch_block_inverse(float* L, int64_t ldl, int64_t m, float* W, float* WT, float* T, cudaStream_t s);

struct RefineArgs {
  const float* L;       // the factor and its blocks' inverses
  int64_t ldl, m;
  const float *W, *WT;
  const double* H;      // the matrix, FP64
  int64_t ldh;
  double shift;
  const double* b;
  double* x;
  float *v, *z, *xs;    // m each
  double* red;          // 4 per CTA
  const double* rowsum; // m: row sums of |H + shift I|
  const int32_t* finfo; // the factorisation's info, or NULL
  RefineState* state;
  unsigned* bar;        // zeroed
  int32_t max_iter;
  double tol;
  const float *V, *Ci;  // low-rank correction (V NULL: none)
  float* sp;            // ldv per CTA
  int64_t ldv;
  int32_t k;
};
constexpr int64_t kRefineRows = 8;    // rows per CTA, at least (their FP64 residual is its longest part)
int launch_refine(const RefineArgs& a, cudaStream_t s);

}  // namespace spsvm
