// HBM-bound passes over the stored kernel matrix K_nJ (basis-major):
//   * o = K_nJ beta with the active set, loss and error count of Eq. 4;
//   * u = K_nJ v (line-search direction);
//   * active-set compaction K_SJ with the masked transposed products
//     K_SJ^T w (gradient and Newton right-hand side of Eq. 4).
// Products are FP32.  The first two promote the running sum to FP64 every 32
// terms, the compaction keeps its sums as compensated FP32 pairs.
#include <cooperative_groups.h>

#include "internal.h"

namespace cg = cooperative_groups;

namespace spsvm {

namespace {

constexpr int GV_T = 256;          // threads per block
constexpr int GV_P = 2;            // consecutive points per thread
constexpr int GV_PTS = GV_T * GV_P;
constexpr int GV_CHUNK = 32;       // terms summed in FP32 before promotion (all in flight)
constexpr int GV_BETA = 2048;      // beta entries staged in shared memory per pass

__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// Loads the thread's 2 consecutive kernel values of row j from point i
// (i even, i + 1 < n) as FP32: one 8-byte load (FP32), or one 4-byte load
// per BF16 plane.  A warp's load instruction covers 256 contiguous bytes of
// a row; with a whole chunk of 32 rows in flight per thread this layout
// streams at the HBM read rate (fewer, wider loads per thread kept fewer
// bytes in flight).  kSplitOdd: planes an odd number of elements apart, whose
// second plane is read singly.
constexpr int kSplitOdd = 2;
static_assert(SPSVM_FP32 != kSplitOdd && SPSVM_BF16SPLIT != kSplitOdd, "a form of its own");
template <int FMT>
__device__ __forceinline__ void load2(const KView& K, int64_t j, int64_t i, float k[2]) {
  if (FMT == SPSVM_FP32) {
    const float2 a = *reinterpret_cast<const float2*>(static_cast<const float*>(K.data) + j * K.ld + i);
    k[0] = a.x;
    k[1] = a.y;
  } else {
    const uint16_t* base = static_cast<const uint16_t*>(K.data);
    const uint32_t h = *reinterpret_cast<const uint32_t*>(base + j * K.ld + i);
    const uint16_t* lo = base + K.plane + j * K.ld + i;
    const uint32_t l = FMT == kSplitOdd ? (uint32_t)lo[0] | ((uint32_t)lo[1] << 16)
                                        : *reinterpret_cast<const uint32_t*>(lo);
    k[0] = bf_lo(h) + bf_lo(l);
    k[1] = bf_hi(h) + bf_hi(l);
  }
}

// acc[p] = sum_j K[j][i + p] v_j for the thread's points.
template <int FMT>
__device__ __forceinline__ void row_products(const KView& K, int64_t rows, int64_t n,
                                             const double* __restrict__ v, int64_t i,
                                             float* vs, double acc[GV_P]) {
#pragma unroll
  for (int p = 0; p < GV_P; ++p) acc[p] = 0.0;
  const bool full = (i + GV_P <= n);
  for (int64_t j0 = 0; j0 < rows; j0 += GV_BETA) {
    const int cnt = (int)min64(GV_BETA, rows - j0);
    __syncthreads();
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) vs[t] = (float)v[j0 + t];
    __syncthreads();
    if (i >= n) continue;
    for (int c0 = 0; c0 < cnt; c0 += GV_CHUNK) {
      float f[GV_P];
#pragma unroll
      for (int p = 0; p < GV_P; ++p) f[p] = 0.f;
      if (full && c0 + GV_CHUNK <= cnt) {
#pragma unroll
        for (int c = c0; c < c0 + GV_CHUNK; ++c) {
          float k[GV_P];
          load2<FMT>(K, j0 + c, i, k);
          const float b = vs[c];
#pragma unroll
          for (int p = 0; p < GV_P; ++p) f[p] = fmaf(k[p], b, f[p]);
        }
      } else {
        const int ce = min(cnt, c0 + GV_CHUNK);
        for (int c = c0; c < ce; ++c) {
          const float b = vs[c];
          for (int p = 0; p < GV_P; ++p)
            if (i + p < n) f[p] = fmaf(K.at(j0 + c, i + p), b, f[p]);
        }
      }
#pragma unroll
      for (int p = 0; p < GV_P; ++p) acc[p] += (double)f[p];
    }
  }
}

// Where the points alone leave SMs idle (a block takes 512), a cluster of
// blocks shares a tile of points: rank r sums the r-th share of the rows, in
// whole chunks, and rank 0 adds the ranks' sums in order through distributed
// shared memory.  HBM (or L2) bound: n = 30,000, 1,024 rows (123 MB) 28 us, 114
// with 59 blocks.
constexpr int GV_CLUSTER = 8;
template <int FMT>
__device__ __forceinline__ bool cluster_products(const KView& K, int64_t rows, int64_t n,
                                                 const double* __restrict__ v, int64_t i, float* vs,
                                                 double acc[GV_P]) {
  __shared__ double red[GV_T][GV_P];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int64_t per = ceil_div(ceil_div(rows, (int64_t)GV_CHUNK), (int64_t)cs) * GV_CHUNK;
  const int64_t j0 = min64(rows, rank * per);
  KView Kr = K;
  if (FMT == SPSVM_FP32) Kr.data = static_cast<const float*>(K.data) + j0 * K.ld;
  else Kr.data = static_cast<const uint16_t*>(K.data) + j0 * K.ld;
  row_products<FMT>(Kr, min64(rows, j0 + per) - j0, n, v + j0, i, vs, acc);
#pragma unroll
  for (int p = 0; p < GV_P; ++p) red[threadIdx.x][p] = acc[p];
  cl.sync();
  if (rank == 0)
    for (int r = 1; r < cs; ++r)
#pragma unroll
      for (int p = 0; p < GV_P; ++p) acc[p] += *cl.map_shared_rank(&red[threadIdx.x][p], r);
  cl.sync();   // no block leaves while rank 0 reads its sums
  return rank == 0;
}

// The thread's products over all rows; false in the blocks of a cluster that
// have given theirs away.  CL: a cluster per tile of points.
template <int FMT, bool CL>
__device__ __forceinline__ bool tile_products(const KView& K, int64_t rows, int64_t n,
                                              const double* __restrict__ v, int64_t i, float* vs,
                                              double acc[GV_P]) {
  if constexpr (CL) return cluster_products<FMT>(K, rows, n, v, i, vs, acc);
  row_products<FMT>(K, rows, n, v, i, vs, acc);
  return true;
}
template <bool CL>
__device__ __forceinline__ int64_t tile_of_block() {
  if constexpr (CL) return blockIdx.x / cg::this_cluster().num_blocks();
  return blockIdx.x;
}

// o = K beta (or given), active flags, per-block loss / errors / |S|.
template <int FMT, bool CL>
__device__ __forceinline__ void outputs_tile(
    const KView& K, int64_t rows, int64_t n, const double* __restrict__ beta,
    const float* __restrict__ y, float* __restrict__ o, uint8_t* __restrict__ active,
    double* __restrict__ part) {
  __shared__ float vs[GV_BETA];
  __shared__ double sh[32];
  const int64_t tile = tile_of_block<CL>();
  const int64_t i = (tile * GV_T + threadIdx.x) * GV_P;
  double acc[GV_P];
  if (beta && !tile_products<FMT, CL>(K, rows, n, beta, i, vs, acc)) return;
  double loss = 0.0, err = 0.0, act = 0.0;
  {
#pragma unroll
    for (int p = 0; p < GV_P; ++p) {
      const int64_t ii = i + p;
      if (ii >= n) break;
      float oi;
      if (beta) {
        oi = (float)acc[p];
        o[ii] = oi;
      } else {
        oi = o[ii];
      }
      const float yi = y[ii];
      const float margin = yi * oi;
      const bool s = margin < 1.0f;
      if (active) active[ii] = s ? 1 : 0;
      if (s) {
        const double xi = 1.0 - (double)margin;
        loss += xi * xi;
        act += 1.0;
      }
      if (margin <= 0.0f) err += 1.0;
    }
  }
  if (part) {
    loss = block_sum(loss, sh);
    __syncthreads();
    err = block_sum(err, sh);
    __syncthreads();
    act = block_sum(act, sh);
    if (threadIdx.x == 0) {
      part[3 * tile + 0] = 0.5 * loss;
      part[3 * tile + 1] = err;
      part[3 * tile + 2] = act;
    }
  }
}

template <int FMT, bool CL>
__global__ void __launch_bounds__(GV_T) outputs_kernel(
    KView K, int64_t rows, int64_t n, const double* __restrict__ beta, const float* __restrict__ y,
    float* __restrict__ o, uint8_t* __restrict__ active, double* __restrict__ part) {
  outputs_tile<FMT, CL>(K, rows, n, beta, y, o, active, part);
}
// In 32 registers, for more blocks than SMs hold six of each (n = 500,000, 4,000
// rows 1.14 ms against 1.34 with 40; but 100,000 points by 30 rows in split form
// 16.1 us against 13.5).
template <int FMT, bool>
__global__ void __launch_bounds__(GV_T, 8) outputs_dense_kernel(
    KView K, int64_t rows, int64_t n, const double* __restrict__ beta, const float* __restrict__ y,
    float* __restrict__ o, uint8_t* __restrict__ active, double* __restrict__ part) {
  outputs_tile<FMT, false>(K, rows, n, beta, y, o, active, part);
}

template <int FMT, bool CL>
__global__ void __launch_bounds__(GV_T) gemv_kernel(KView K, int64_t rows, int64_t n,
                                                    const double* __restrict__ v,
                                                    float* __restrict__ u, int accumulate) {
  __shared__ float vs[GV_BETA];
  const int64_t i = (tile_of_block<CL>() * GV_T + threadIdx.x) * GV_P;
  double acc[GV_P];
  if (!tile_products<FMT, CL>(K, rows, n, v, i, vs, acc)) return;
#pragma unroll
  for (int p = 0; p < GV_P; ++p) {
    const int64_t ii = i + p;
    if (ii < n) u[ii] = accumulate ? (float)((double)u[ii] + acc[p]) : (float)acc[p];
  }
}

// Fixed-order sum of per-block triples.
__global__ void sum_triples(const double* __restrict__ part, int64_t blocks, double* out) {
  __shared__ double sh[32];
  for (int c = 0; c < 3; ++c) {
    double s = 0.0;
    for (int64_t b = threadIdx.x; b < blocks; b += blockDim.x) s += part[3 * b + c];
    s = block_sum(s, sh);
    __syncthreads();
    if (threadIdx.x == 0) out[c] = s;
  }
}

// ---- active-set scan -----------------------------------------------------
constexpr int SC_T = 256;
constexpr int SC_PTS = SC_T * 4;

// The scanned flag of point i: whether it is active (any nonzero byte), or with
// ref, whether that differs.
__device__ __forceinline__ int scan_flag(const uint8_t* __restrict__ active,
                                         const uint8_t* __restrict__ ref, int64_t i) {
  const bool a = active[i] != 0;
  return ref ? (int)(a != (ref[i] != 0)) : (int)a;
}

__global__ void scan_count(const uint8_t* __restrict__ active, const uint8_t* __restrict__ ref,
                           int64_t n, int32_t* __restrict__ counts) {
  __shared__ int sh[32];
  const int64_t base = (int64_t)blockIdx.x * SC_PTS;
  int c = 0;
  for (int p = 0; p < 4; ++p) {
    const int64_t i = base + threadIdx.x + (int64_t)SC_T * p;
    if (i < n) c += scan_flag(active, ref, i);
  }
  c = block_sum(c, sh);
  if (threadIdx.x == 0) counts[blockIdx.x] = c;
}

// What a block of step_points leaves beside its count of active points.
struct StepPart {
  double loss;
  int32_t err, diff;
};

// The step of StepArgs over SC_PTS points per block, with the block's count
// for the scan.  Latency bound: one launch where the updates of beta and o, the
// flags, their count, the count of changes and the residuals took seven.  FP64
// would take longer than the rest (64 cycles an instruction and warp): o + t u
// and the loss are FP32 pairs, about 2^-46 before their last rounding.
__global__ void __launch_bounds__(SC_T) step_points(StepArgs a, int64_t n, int32_t* __restrict__ counts,
                                                    StepPart* __restrict__ part) {
  __shared__ float2 shl[SC_T / 32];
  __shared__ int shc[SC_T / 32], she[SC_T / 32], shd[SC_T / 32];
  constexpr int P = SC_PTS / SC_T;
  const int64_t base = (int64_t)blockIdx.x * SC_PTS + threadIdx.x;
  const double t = *a.t;
  float ov[P], uv[P], yv[P];
  uint8_t bv[P];
#pragma unroll
  for (int p = 0; p < P; ++p) {   // all in flight together with t
    const int64_t i = min64(n - 1, base + (int64_t)SC_T * p);
    ov[p] = a.o[i];
    uv[p] = a.u[i];
    yv[p] = a.y[i];
    bv[p] = a.before[i];
  }
  const float th = (float)t, tl = (float)(t - (double)th);
  float hi = 0.f, lo = 0.f;
  int c = 0, err = 0, diff = 0;
#pragma unroll
  for (int p = 0; p < P; ++p) {
    const int64_t i = base + (int64_t)SC_T * p;
    if (i >= n) break;
    float oi = ov[p];
    const float yi = yv[p];
    if (t != 0.0) {
      const float ui = uv[p];
      const float q = __fmul_rn(th, ui);
      const float s = __fadd_rn(oi, q);
      const float b = __fsub_rn(s, oi);
      const float e = __fadd_rn(__fsub_rn(oi, __fsub_rn(s, b)), __fsub_rn(q, b));
      const float f = __fmaf_rn(tl, ui, __fmaf_rn(th, ui, -q));
      oi = __fsub_rn(s, s) == 0.0f ? __fadd_rn(s, __fadd_rn(e, f)) : s;
      a.o[i] = oi;
    }
    const float margin = yi * oi;
    const bool act = margin < 1.0f;
    c += act;
    err += margin <= 0.0f;
    diff += (bv[p] != 0) != act;
    a.active[i] = act ? 1 : 0;
    a.res[i] = oi - yi;
    if (act) {   // (1 - margin)^2, 1 - margin exact as a pair
      const float x = __fsub_rn(1.0f, margin);
      const float b = __fsub_rn(x, 1.0f);
      const float e = __fadd_rn(__fsub_rn(1.0f, __fsub_rn(x, b)), -__fadd_rn(margin, b));
      lo = __fmaf_rn(2.0f * x, e, lo);
      pair_add_sq(hi, lo, x);
    }
  }
  if (t != 0.0)
    for (int64_t k = (int64_t)blockIdx.x * SC_T + threadIdx.x; k < a.m; k += (int64_t)gridDim.x * SC_T)
      a.beta[k] += t * a.dir[k];
#pragma unroll
  for (int q = 16; q > 0; q >>= 1) {
    const float oh = __shfl_xor_sync(0xffffffffu, hi, q), ol = __shfl_xor_sync(0xffffffffu, lo, q);
    pair_add(hi, lo, make_float2(oh, ol));
  }
  c = __reduce_add_sync(0xffffffffu, c);
  err = __reduce_add_sync(0xffffffffu, err);
  diff = __reduce_add_sync(0xffffffffu, diff);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    shl[w] = make_float2(hi, lo);
    shc[w] = c;
    she[w] = err;
    shd[w] = diff;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int k = 1; k < SC_T / 32; ++k) {
    pair_add(hi, lo, shl[k]);
    c += shc[k];
    err += she[k];
    diff += shd[k];
  }
  counts[blockIdx.x] = c;
  part[blockIdx.x] = StepPart{0.5 * pair_value(hi, lo), err, diff};
}

// Sums of the blocks' parts, in a fixed order (all threads of one block).
__device__ void step_sums(const StepPart* __restrict__ part, int64_t nb, int64_t total,
                          double* __restrict__ stats, unsigned long long* __restrict__ ndiff) {
  __shared__ double shs[32];
  __shared__ int shi[32];
  double loss = 0.0;
  int err = 0, diff = 0;
  for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) {
    loss += part[b].loss;
    err += part[b].err;
    diff += part[b].diff;
  }
  loss = block_sum(loss, shs);
  err = block_sum(err, shi);
  diff = block_sum(diff, shi);
  if (threadIdx.x == 0) {
    stats[0] = loss;
    stats[1] = (double)err;
    stats[2] = (double)total;
    *ndiff = (unsigned long long)diff;
  }
}

// v summed over the threads before this one, by warps; *total: over the block.
__device__ __forceinline__ int32_t block_scan(int32_t v, int32_t* __restrict__ sh /* 32 */, int32_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) sh[w] = x;
  __syncthreads();
  int32_t before = 0, all = 0;
  for (int k = 0; k < (int)blockDim.x >> 5; ++k) {
    if (k < w) before += sh[k];
    all += sh[k];
  }
  *total = all;
  return before + x - v;
}

// Exclusive scan of block counts in one block; writes the total to *total.
__global__ void scan_blocks(int32_t* __restrict__ counts, int64_t nb, int64_t* __restrict__ total,
                            const StepPart* __restrict__ part, double* __restrict__ stats,
                            unsigned long long* __restrict__ ndiff) {
  __shared__ int32_t sh[32];
  int64_t carry = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += blockDim.x) {
    const int64_t b = b0 + threadIdx.x;
    const int32_t v = (b < nb) ? counts[b] : 0;
    int32_t sum;
    const int32_t excl = block_scan(v, sh, &sum);
    if (b < nb) counts[b] = (int32_t)(carry + excl);
    carry += sum;
  }
  if (threadIdx.x == 0) *total = carry;
  if (part) step_sums(part, nb, carry, stats, ndiff);
}

// Positions and the list of the flagged points.  SUM: counts are the blocks'
// own, which every block sums up to its place itself (up to SC_SUM of them: a
// launch less), and block 0 writes the total and the step's sums; else they
// are scanned.
constexpr int64_t SC_SUM = 1024;
template <bool SUM>
__global__ void __launch_bounds__(SC_T) scan_write(const uint8_t* __restrict__ active,
                                                   const uint8_t* __restrict__ ref, int64_t n,
                                                   const int32_t* __restrict__ counts,
                                                   int32_t* __restrict__ pos, int32_t* __restrict__ list,
                                                   int64_t* __restrict__ total,
                                                   const StepPart* __restrict__ part,
                                                   double* __restrict__ stats,
                                                   unsigned long long* __restrict__ ndiff) {
  __shared__ int32_t sh[32];
  __shared__ int32_t off_s;
  const int64_t i0 = (int64_t)blockIdx.x * SC_PTS + threadIdx.x * 4;
  int32_t f[4], run = 0, first = 0;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    f[p] = i0 + p < n ? scan_flag(active, ref, i0 + p) : 0;
    run += f[p];
  }
  if (SUM) {
    int32_t c = 0;
    const int64_t end = blockIdx.x ? blockIdx.x : gridDim.x;   // block 0: the total
    for (int64_t b = threadIdx.x; b < end; b += SC_T) c += counts[b];
    c = block_sum(c, sh);
    if (threadIdx.x == 0) off_s = c;
    __syncthreads();
    first = off_s;
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) *total = first;
      if (part) step_sums(part, gridDim.x, first, stats, ndiff);
      first = 0;
    }
  } else {
    first = counts[blockIdx.x];
  }
  int32_t sum;
  int32_t at = first + block_scan(run, sh, &sum);
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int64_t i = i0 + p;
    if (i >= n) break;
    if (pos) pos[i] = at;
    if (f[p]) list[at] = (int32_t)i;   // flagged indices, in order
    at += f[p];
  }
}

// Positions, list and count of the flagged points; with `step`, the step first
// and its sums.  The step's parts take `room` (the compaction's partials,
// written later) while block 0 reads them beside the list's writers, else the
// list's space.
int launch_scan(const uint8_t* active, const uint8_t* ref, int64_t n, int32_t* counts, int32_t* pos,
                int32_t* list, int64_t* total, const StepArgs* step, void* room, cudaStream_t s) {
  const int64_t sb = ceil_div(n, (int64_t)SC_PTS);
  StepPart* part = step ? static_cast<StepPart*>(sb <= SC_SUM ? room : list) : nullptr;
  double* stats = step ? step->stats : nullptr;
  unsigned long long* ndiff = step ? step->ndiff : nullptr;
  if (step) step_points<<<(unsigned)sb, SC_T, 0, s>>>(*step, n, counts, part);
  else scan_count<<<(unsigned)sb, SC_T, 0, s>>>(active, ref, n, counts);
  SPSVM_LAUNCH_CHECK();
  if (sb <= SC_SUM) {
    scan_write<true><<<(unsigned)sb, SC_T, 0, s>>>(active, ref, n, counts, pos, list, total, part, stats, ndiff);
    SPSVM_LAUNCH_CHECK();
    return SPSVM_OK;
  }
  scan_blocks<<<1, 1024, 0, s>>>(counts, sb, total, part, stats, ndiff);
  SPSVM_LAUNCH_CHECK();
  scan_write<false><<<(unsigned)sb, SC_T, 0, s>>>(active, ref, n, counts, pos, list, total, nullptr, nullptr, nullptr);
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

// ---- compaction + masked transposed products ---------------------------
// One block: 32 basis rows (each warp four of them) over a slice of the
// compact columns.  A lane takes two pairs of adjacent compact columns per
// step through the list of active indices, so every lane carries an active
// point whatever their density, a row's reads cover a contiguous stretch of
// K (16 loads in flight per lane) and its writes are whole 128-byte lines.
// The weighted sums are compensated pairs: of every product, its rounding
// included, in short slices (a chain of latencies, where that costs nothing;
// the gradient of a small fit is as accurate as these sums), else of FP32 sums
// of eight terms (of 32: 387 us below as well).  One FP64 reduction per warp.  Bound by HBM: at n = 200,000, 2,048 rows, 43%
// active (1.64 GB read, 0.70 GB written) 0.38 ms, 6.1 TB/s; a thread per point
// of every row, 57% of them idle, with two-byte writes took 3.36 ms.
constexpr int CP_T = 256;
constexpr int CP_WARPS = CP_T / 32;
constexpr int CP_R = 4;                      // basis rows per warp
constexpr int CP_ROWS = CP_WARPS * CP_R;     // basis rows per block
constexpr int CP_Q = 128;                    // compact columns per step
constexpr int CP_CHUNK = 2;                  // steps summed in FP32 (4 terms each)
constexpr int64_t CP_FINE = 2048;            // columns of a short slice
constexpr int64_t CP_MIN_SLICE = 1024;       // points per slice that pay its epilogue

// Columns per slice of the compact matrix for ns active points.
__device__ __forceinline__ int64_t cp_slice(int64_t ns, int64_t slices) {
  return max64(CP_Q, round_up(ceil_div(ns, slices), (int64_t)CP_Q));
}

// Sums of eight values over a warp: lane l ends with the sum of value
// (l >> 2) & 7 (9 exchanges instead of 40).
__device__ __forceinline__ double warp_sum8(double (&v)[8], int lane) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const bool up = (lane & 16) != 0;
    const double give = up ? v[k] : v[k + 4], keep = up ? v[k + 4] : v[k];
    v[k] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const bool up = (lane & 8) != 0;
    const double give = up ? v[k] : v[k + 2], keep = up ? v[k + 2] : v[k];
    v[k] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
  }
  {
    const bool up = (lane & 4) != 0;
    const double give = up ? v[0] : v[1], keep = up ? v[1] : v[0];
    v[0] = keep + __shfl_xor_sync(0xffffffffu, give, 4);
  }
  double s = v[0];
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

// KF: K's format; CF: the compact copy's (FP32 from FP32, or hi / lo planes,
// copied from K's planes or split from an FP32 value).  pair_ok: the lo
// plane starts on an even element, so two columns go in one store.
template <int KF, int CF>
__global__ void __launch_bounds__(CP_T, 3) compact_kernel(
    KView K, int64_t rows, const int32_t* __restrict__ list, const int64_t* __restrict__ ns_dev,
    const float* __restrict__ w1, const float* __restrict__ w2, void* kc_data, int64_t kc_ld,
    int64_t kc_plane, int64_t kc_n, int pair_ok, int64_t slices, double2* __restrict__ part,
    const unsigned long long* __restrict__ kc_cond) {
  const int64_t ns = *ns_dev;
  const int64_t per = cp_slice(ns, slices);
  const int64_t b = (int64_t)blockIdx.y * per;
  if (b >= ns && blockIdx.y > 0) return;
  const int64_t e = min64(ns, b + per);
  if (kc_cond && *kc_cond == 0) kc_data = nullptr;   // the caller keeps the copy it has
  const int lane = threadIdx.x & 31;
  const int64_t j0 = (int64_t)blockIdx.x * CP_ROWS + (threadIdx.x >> 5) * CP_R;
  if (j0 >= rows) return;
  int64_t row[CP_R];   // rows past the last repeat it (and are not written)
#pragma unroll
  for (int r = 0; r < CP_R; ++r) row[r] = min64(j0 + r, rows - 1) * K.ld;
  float f1[CP_R], f2[CP_R], h1[CP_R], h2[CP_R], l1[CP_R], l2[CP_R];
#pragma unroll
  for (int r = 0; r < CP_R; ++r) f1[r] = f2[r] = h1[r] = h2[r] = l1[r] = l2[r] = 0.f;
  int since = 0;
  const bool fine = per <= CP_FINE;
  // the next step's indices are read a step ahead (K's loads wait for them)
  int32_t nxt[4];
  auto indices = [&](int64_t q0) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int64_t q = q0 + 64 * (p >> 1) + 2 * lane + (p & 1);
      nxt[p] = q < e ? list[q] : -1;
    }
  };
  indices(b);
  for (int64_t q0 = b; q0 < e; q0 += CP_Q) {
    int32_t i[4];
    float a[4], c[4];
    bool in[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      in[p] = nxt[p] >= 0;
      i[p] = in[p] ? nxt[p] : 0;
    }
    indices(q0 + CP_Q);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      a[p] = in[p] && w1 ? w1[i[p]] : 0.f;
      c[p] = in[p] && w2 ? w2[i[p]] : 0.f;
    }
    float v[CP_R][4];
    uint32_t raw[CP_R][4];
#pragma unroll
    for (int r = 0; r < CP_R; ++r)
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (KF == SPSVM_FP32) {
          v[r][p] = in[p] ? static_cast<const float*>(K.data)[row[r] + i[p]] : 0.f;
        } else {
          const uint16_t* src = static_cast<const uint16_t*>(K.data) + row[r] + i[p];
          raw[r][p] = in[p] ? (uint32_t)src[0] | ((uint32_t)src[K.plane] << 16) : 0u;
        }
      }
#pragma unroll
    for (int r = 0; r < CP_R; ++r) {
      if (KF != SPSVM_FP32)
#pragma unroll
        for (int p = 0; p < 4; ++p) v[r][p] = bf_lo(raw[r][p]) + bf_hi(raw[r][p]);
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if (fine) {
          const float p1 = __fmul_rn(a[p], v[r][p]), p2 = __fmul_rn(c[p], v[r][p]);
          l1[r] = __fadd_rn(l1[r], __fmaf_rn(a[p], v[r][p], -p1));
          l2[r] = __fadd_rn(l2[r], __fmaf_rn(c[p], v[r][p], -p2));
          pair_add(h1[r], l1[r], p1);
          pair_add(h2[r], l2[r], p2);
        } else {
          f1[r] = fmaf(a[p], v[r][p], f1[r]);
          f2[r] = fmaf(c[p], v[r][p], f2[r]);
        }
      }
      if (kc_data && j0 + r < rows) {
#pragma unroll
        for (int p = 0; p < 4; p += 2) {
          const int64_t off = (j0 + r) * kc_ld + q0 + 64 * (p >> 1) + 2 * lane;
          if (CF == SPSVM_FP32) {
            float* dst = static_cast<float*>(kc_data) + off;
            if (in[p + 1]) *reinterpret_cast<float2*>(dst) = make_float2(v[r][p], v[r][p + 1]);
            else if (in[p]) dst[0] = v[r][p];
          } else {
            __nv_bfloat162 h, l;
            if (KF == SPSVM_FP32) {
              split_bf16(v[r][p], h.x, l.x);
              split_bf16(v[r][p + 1], h.y, l.y);
            } else {
              h.x = __ushort_as_bfloat16((unsigned short)raw[r][p]);
              l.x = __ushort_as_bfloat16((unsigned short)(raw[r][p] >> 16));
              h.y = __ushort_as_bfloat16((unsigned short)raw[r][p + 1]);
              l.y = __ushort_as_bfloat16((unsigned short)(raw[r][p + 1] >> 16));
            }
            __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(kc_data) + off;
            if (in[p + 1] && pair_ok) {
              *reinterpret_cast<__nv_bfloat162*>(dst) = h;
              *reinterpret_cast<__nv_bfloat162*>(dst + kc_plane) = l;
            } else {
              if (in[p]) { dst[0] = h.x; dst[kc_plane] = l.x; }
              if (in[p + 1]) { dst[1] = h.y; dst[kc_plane + 1] = l.y; }
            }
          }
        }
      }
    }
    if (++since == CP_CHUNK) {
#pragma unroll
      for (int r = 0; r < CP_R; ++r) {
        pair_add(h1[r], l1[r], f1[r]);
        pair_add(h2[r], l2[r], f2[r]);
        f1[r] = f2[r] = 0.f;
      }
      since = 0;
    }
  }
  if (kc_data && e == ns) {   // zero columns up to the next multiple of 128
    const int64_t end = min64(kc_n, round_up(ns, (int64_t)128));
    for (int64_t q = ns + lane; q < end; q += 32)
#pragma unroll
      for (int r = 0; r < CP_R; ++r)
        if (j0 + r < rows) {
          const int64_t off = (j0 + r) * kc_ld + q;
          if (CF == SPSVM_FP32) {
            static_cast<float*>(kc_data)[off] = 0.f;
          } else {
            static_cast<__nv_bfloat16*>(kc_data)[off] = __float2bfloat16_rn(0.f);
            static_cast<__nv_bfloat16*>(kc_data)[kc_plane + off] = __float2bfloat16_rn(0.f);
          }
        }
  }
  double s[8];
#pragma unroll
  for (int r = 0; r < CP_R; ++r) {
    pair_add(h1[r], l1[r], f1[r]);
    pair_add(h2[r], l2[r], f2[r]);
    s[2 * r] = pair_value(h1[r], l1[r]);
    s[2 * r + 1] = pair_value(h2[r], l2[r]);
  }
  const double tot = warp_sum8(s, lane);
  const int k = (lane >> 2) & 7;   // value k: row k / 2, sum k % 2
  if ((lane & 3) == 0 && j0 + (k >> 1) < rows)
    reinterpret_cast<double*>(part + (int64_t)blockIdx.y * rows + j0 + (k >> 1))[k & 1] = tot;
}

// Sums of the slices' partials, 32 rows a block, eight threads a row that take
// every eighth slice; with `grad`, the gradient's entries of these rows and,
// in the block that ends last, the three dots (blocks' parts in order).
constexpr int CF_G = 8;
__global__ void __launch_bounds__(32 * CF_G) compact_finish(const double2* __restrict__ part, int64_t slices,
                                                            int64_t rows, double* w1out, double* w2out,
                                                            const int64_t* __restrict__ ns_dev, GradArgs grad,
                                                            double* __restrict__ dpart) {
  __shared__ double2 sh[CF_G][32];
  __shared__ bool last_s;
  const int c = threadIdx.x & 31, q = threadIdx.x >> 5;
  const int64_t j = (int64_t)blockIdx.x * 32 + c;
  const int64_t ns = *ns_dev;
  double r = 0.0, be = 0.0;   // read ahead of the sums
  if (grad.g && q == 0 && j < rows) {
    const int64_t k = grad.J[j];
    r = k < 0 ? 0.0 : (double)grad.o[k] - (grad.b0 ? *grad.b0 : 0.0);
    be = grad.beta[j];
  }
  const int64_t used = max64(1, ceil_div(ns, cp_slice(ns, slices)));
  double a = 0.0, b = 0.0;
  if (j < rows)
    for (int64_t s = q; s < used; s += CF_G) {
      const double2 p = part[s * rows + j];
      a += p.x;
      b += p.y;
    }
  sh[q][c] = make_double2(a, b);
  __syncthreads();
  if (q != 0) return;
#pragma unroll
  for (int k = 1; k < CF_G; ++k) {
    a += sh[k][c].x;
    b += sh[k][c].y;
  }
  double x = 0.0, g = 0.0;
  if (j < rows) {
    if (w1out) w1out[j] = a;
    if (w2out) w2out[j] = b;
    if (grad.g) {
      g = grad.lambda * r + a;
      grad.g[j] = g;
      grad.rhs[j] = -g;
      x = be * r;
    }
  }
  if (!grad.g) return;
  const double d0 = warp_sum(x), d1 = warp_sum(g * g), d2 = warp_sum(j < rows ? b * b : 0.0);
  if (c == 0) {
    double* d = dpart + 3 * blockIdx.x;
    d[0] = d0;
    d[1] = d1;
    d[2] = d2;
    __threadfence();
    last_s = atomicInc(grad.done, gridDim.x - 1) == gridDim.x - 1;
    __threadfence();
  }
  __syncwarp();
  if (!last_s) return;
  double t[3] = {0.0, 0.0, 0.0};
  for (int64_t k = c; k < gridDim.x; k += 32)
#pragma unroll
    for (int e = 0; e < 3; ++e) t[e] += __ldcg(dpart + 3 * k + e);
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    t[e] = warp_sum(t[e]);
    if (c == 0) grad.dots[e] = t[e];
  }
}

// Wt[j][r] = K[j][list[r]] for the k = *k_dev listed points (nothing when
// k > kmax); sign[r] = +1 when list[r] is active, else -1.  Blocks stride
// over the basis rows, threads over the points.
__global__ void diff_gather(KView K, int64_t rows, const int32_t* __restrict__ list,
                            const int32_t* __restrict__ k_dev, int32_t kmax,
                            const uint8_t* __restrict__ active, float* __restrict__ Wt,
                            int64_t ldw, float* __restrict__ sign) {
  const int32_t k = *k_dev;
  if (k > kmax) return;
  if (blockIdx.x == 0)
    for (int r = threadIdx.x; r < k; r += blockDim.x) sign[r] = active[list[r]] ? 1.0f : -1.0f;
  for (int64_t j = blockIdx.x; j < rows; j += gridDim.x)
    for (int r = threadIdx.x; r < k; r += blockDim.x) Wt[j * ldw + r] = K.at(j, list[r]);
}

// *k_dev = (int32) *total
__global__ void store_count(const int64_t* __restrict__ total, int32_t* __restrict__ k_dev) {
  *k_dev = (int32_t)*total;
}

}  // namespace
}  // namespace spsvm

namespace spsvm {
namespace {
// Blocks per tile of points: two, four or eight while SMs would be idle or nearly
// so, and a block keeps rows enough to pay the cluster's barriers: 32 up to a block
// for every other SM, 64 up to three blocks per SM, then 128; the outputs, whose
// epilogue one block in each cluster runs, 64 up to one block per SM, then 192.
// 30,000 points by 1,024 rows: u = K v 28 us, one block a tile 114.  From L2,
// 100,000 by 128: two blocks of 64 rows 7.3, one 7.8, four 10.3 (from HBM 20.7, 25.1
// and 21.8; outputs 17.1, 14.8 and 25.4); 60,000 by 256: two 9.2, four 9.8, one 12.3
// (outputs 17.5, 21.3 and 17.0).
int gv_cluster(int64_t tiles, int64_t rows, bool outputs) {
  const int64_t sms = sm_count();
  int cs = 1;
  while (2 * cs <= GV_CLUSTER && tiles * cs < (outputs ? 2 : 4) * sms) {
    const int64_t after = 2 * cs * tiles;
    const int64_t least = outputs ? (after <= sms ? 64 : 192)
                                  : (2 * after <= sms ? 32 : (after <= 3 * sms ? 64 : 128));
    if (rows < 2 * cs * least) break;
    cs *= 2;
  }
  return cs;
}
template <class Kern, class... Args>
cudaError_t gv_launch(Kern kern, int64_t tiles, int cs, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * cs));
  cfg.blockDim = dim3(GV_T);
  cfg.stream = s;
  if (cs == 1) return cudaLaunchKernelEx(&cfg, kern, args...);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
// The instantiation for K's format.
#define SPSVM_GV_KERNEL(K, NAME, CL)                                      \
  ((K)->format == SPSVM_FP32 ? NAME<SPSVM_FP32, CL>                       \
                             : ((K)->plane % 2 == 0 ? NAME<SPSVM_BF16SPLIT, CL> : NAME<kSplitOdd, CL>))
}  // namespace
}  // namespace spsvm

using namespace spsvm;

extern "C" size_t spsvm_reduce_scratch_bytes(int64_t n) {
  if (n < 0) return 0;
  return (size_t)(ceil_div(n, GV_PTS) * 3 * sizeof(double) + 64);
}

extern "C" int spsvm_outputs(const spsvm_kmat* K, const double* beta, const float* y, float* o,
                             uint8_t* active, double* stats, void* scratch, size_t scratch_bytes,
                             void* stream) {
  SPSVM_TRY(check_kmat(K, "outputs"));
  if (!y || !o) return set_error(SPSVM_ERR_ARG, "outputs: NULL y/o");
  if (K->n == 0) return SPSVM_OK;
  if (stats && (!scratch || scratch_bytes < spsvm_reduce_scratch_bytes(K->n)))
    return set_error(SPSVM_ERR_OOM, "outputs: scratch too small");
  cudaStream_t s = as_stream(stream);
  ProfScope prof(PROF_OUTPUTS, s, beta ? 4.0 * (double)K->rows * K->n : 9.0 * K->n);
  const int64_t blocks = ceil_div(K->n, GV_PTS);
  double* part = stats ? static_cast<double*>(scratch) : nullptr;
  const int cs = beta ? gv_cluster(blocks, K->rows, true) : 1;
  auto kern = cs > 1 ? SPSVM_GV_KERNEL(K, outputs_kernel, true)
                     : (blocks > 6 * (int64_t)sm_count() ? SPSVM_GV_KERNEL(K, outputs_dense_kernel, false)
                                                         : SPSVM_GV_KERNEL(K, outputs_kernel, false));
  SPSVM_CUDA_TRY(gv_launch(kern, blocks, cs, s, view(K), K->rows, K->n, beta, y, o, active, part));
  SPSVM_LAUNCH_CHECK();
  if (stats) {
    sum_triples<<<1, 256, 0, s>>>(part, blocks, stats);
    SPSVM_LAUNCH_CHECK();
  }
  return SPSVM_OK;
}

extern "C" int spsvm_gemv(const spsvm_kmat* K, const double* v, float* u, int32_t accumulate,
                          void* stream) {
  SPSVM_TRY(check_kmat(K, "gemv"));
  if (!v || !u) return set_error(SPSVM_ERR_ARG, "gemv: NULL pointer");
  if (K->n == 0) return SPSVM_OK;
  const int64_t blocks = ceil_div(K->n, GV_PTS);
  ProfScope prof(PROF_GEMV, as_stream(stream), 4.0 * (double)K->rows * K->n);
  const int cs = gv_cluster(blocks, K->rows, false);
  auto kern = cs > 1 ? SPSVM_GV_KERNEL(K, gemv_kernel, true) : SPSVM_GV_KERNEL(K, gemv_kernel, false);
  SPSVM_CUDA_TRY(gv_launch(kern, blocks, cs, as_stream(stream), view(K), K->rows, K->n, v, u, accumulate));
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

namespace {
// Slices of the compact columns: about eight blocks per SM in all, but no
// slice below CP_MIN_SLICE points (its sums end in an FP64 warp reduction), or half
// as many while the blocks have an SM each (1,000 points by 300 rows, all active:
// split form 24.6 us against 36.4, FP32 19.6 against 26.2; past that the other way:
// 400,000 points by 30 rows, all active 72 us against 55).
int64_t compact_slices(int64_t n, int64_t rows) {
  const int64_t row_blocks = max64(1, ceil_div(rows, (int64_t)CP_ROWS));
  const int64_t short_slices = ceil_div(n, CP_MIN_SLICE / 2);
  if (row_blocks * short_slices <= sm_count()) return max64(1, short_slices);
  const int64_t want = ceil_div(8 * (int64_t)sm_count(), row_blocks);
  return max64(1, min64(want, min64(ceil_div(n, CP_MIN_SLICE), 1024)));
}

template <int KF, int CF>
void compact_launch(dim3 grid, const spsvm_kmat* K, const int32_t* list, const int64_t* ns,
                    const float* w1, const float* w2, const spsvm_kmat* Kc, int64_t kc_n,
                    int64_t slices, double2* part, const unsigned long long* cond, cudaStream_t s) {
  compact_kernel<KF, CF><<<grid, CP_T, 0, s>>>(
      view(K), K->rows, list, ns, w1, w2, Kc ? Kc->data : nullptr, Kc ? Kc->ld : 0,
      Kc ? Kc->plane : 0, kc_n, Kc ? (int)(Kc->plane % 2 == 0) : 0, slices, part, cond);
}
}  // namespace

extern "C" size_t spsvm_compact_scratch_bytes(int64_t n, int64_t rows) {
  if (n < 0 || rows < 0) return 0;
  const int64_t scan_blocks_n = ceil_div(n, SC_PTS);
  // partials for the largest split the launcher may pick (bounded by chunks)
  const int64_t ysplit = ceil_div(n, CP_T) < 1024 ? ceil_div(n, CP_T) : 1024;
  return (size_t)(round_up(scan_blocks_n * 4, 256) +
                  round_up((ysplit > 0 ? ysplit : 1) * (rows > 0 ? rows : 1) * 16, 256) +
                  round_up((n > 0 ? n : 1) * 4, 256));   // list of active indices
}

extern "C" int spsvm_compact_active(const spsvm_kmat* K, const uint8_t* active, const float* w1,
                                    const float* w2, double* w1out, double* w2out,
                                    spsvm_kmat* Kc, int64_t* n_active, int32_t* pos,
                                    void* scratch, size_t scratch_bytes, void* stream) {
  return compact_active_impl(K, active, w1, w2, w1out, w2out, Kc, nullptr, n_active, pos, scratch,
                             scratch_bytes, stream);
}

// With kc_cond, K_SJ is written only when *kc_cond (read on the device) is
// nonzero: the fit passes the count of points whose active flag changed, so
// an unchanged active set keeps the copy in hand without a host round trip.
int spsvm::compact_active_impl(const spsvm_kmat* K, const uint8_t* active, const float* w1,
                               const float* w2, double* w1out, double* w2out, spsvm_kmat* Kc,
                               const unsigned long long* kc_cond, int64_t* n_active,
                               int32_t* pos, void* scratch, size_t scratch_bytes, void* stream,
                               const StepArgs* step, const GradArgs* grad) {
  SPSVM_TRY(check_kmat(K, "compact"));
  if (!active || !n_active || !pos) return set_error(SPSVM_ERR_ARG, "compact: NULL pointer");
  if (Kc) {
    SPSVM_TRY(check_kmat(Kc, "compact(out)"));
    // the compact copy keeps K's format, or splits FP32 values into hi / lo planes
    const bool fmt_ok = Kc->format == K->format || (K->format == SPSVM_FP32 && Kc->format == SPSVM_BF16SPLIT);
    if (!fmt_ok || Kc->rows < K->rows || Kc->n < round_up(K->n, 128))
      return set_error(SPSVM_ERR_ARG, "compact: output matrix too small or wrong format");
  }
  if ((w1out && !w1) || (w2out && !w2)) return set_error(SPSVM_ERR_ARG, "compact: missing weights");
  if (!scratch || scratch_bytes < spsvm_compact_scratch_bytes(K->n, K->rows))
    return set_error(SPSVM_ERR_OOM, "compact: scratch too small");
  cudaStream_t s = as_stream(stream);
  ProfScope prof(PROF_COMPACT, s, 4.0 * (double)K->rows * K->n);
  const int64_t n = K->n;
  const int64_t sb = ceil_div(n, SC_PTS);
  int32_t* counts = static_cast<int32_t*>(scratch);
  double2* part = reinterpret_cast<double2*>(static_cast<char*>(scratch) + round_up(sb * 4, 256));
  const int64_t ysplit_max = ceil_div(n, CP_T) < 1024 ? ceil_div(n, CP_T) : 1024;
  int32_t* list = reinterpret_cast<int32_t*>(
      static_cast<char*>(scratch) + round_up(sb * 4, 256) +
      round_up((ysplit_max > 0 ? ysplit_max : 1) * (K->rows > 0 ? K->rows : 1) * 16, 256));
  if (n == 0) {
    SPSVM_CUDA_TRY(cudaMemsetAsync(n_active, 0, sizeof(int64_t), s));
  } else {
    SPSVM_TRY(launch_scan(active, nullptr, n, counts, pos, list, n_active, step, part, s));
  }
  if (K->rows > 0 && n > 0) {
    const int64_t slices = compact_slices(n, K->rows);
    const dim3 grid((unsigned)ceil_div(K->rows, CP_ROWS), (unsigned)slices);
    const int64_t kc_n = Kc ? min64(round_up(n, 128), Kc->n) : 0;
    const bool ksplit = K->format == SPSVM_BF16SPLIT, csplit = Kc && Kc->format == SPSVM_BF16SPLIT;
    if (ksplit)
      compact_launch<SPSVM_BF16SPLIT, SPSVM_BF16SPLIT>(grid, K, list, n_active, w1, w2, Kc, kc_n,
                                                       slices, part, kc_cond, s);
    else if (csplit)
      compact_launch<SPSVM_FP32, SPSVM_BF16SPLIT>(grid, K, list, n_active, w1, w2, Kc, kc_n, slices,
                                                  part, kc_cond, s);
    else
      compact_launch<SPSVM_FP32, SPSVM_FP32>(grid, K, list, n_active, w1, w2, Kc, kc_n, slices, part,
                                             kc_cond, s);
    SPSVM_LAUNCH_CHECK();
    if (w1out || w2out) {
      // (the list has been read: its space takes the blocks' dots)
      compact_finish<<<(unsigned)ceil_div(K->rows, (int64_t)32), 32 * CF_G, 0, s>>>(
          part, slices, K->rows, w1out, w2out, n_active, grad ? *grad : GradArgs{},
          reinterpret_cast<double*>(list));
      SPSVM_LAUNCH_CHECK();
    }
  } else if (K->rows > 0) {
    if (w1out) SPSVM_CUDA_TRY(cudaMemsetAsync(w1out, 0, K->rows * sizeof(double), s));
    if (w2out) SPSVM_CUDA_TRY(cudaMemsetAsync(w2out, 0, K->rows * sizeof(double), s));
  }
  return SPSVM_OK;
}

extern "C" int spsvm_active_diff(const spsvm_kmat* K, const uint8_t* active, const uint8_t* ref,
                                 int32_t kmax, float* Wt, int64_t ldw, float* sign, int32_t* k_dev,
                                 void* scratch, size_t scratch_bytes, void* stream) {
  SPSVM_TRY(check_kmat(K, "active_diff"));
  if (!active || !ref || !k_dev || kmax < 0 || (kmax > 0 && (!Wt || !sign || ldw < kmax)))
    return set_error(SPSVM_ERR_ARG, "active_diff: bad arguments");
  if (!scratch || scratch_bytes < spsvm_compact_scratch_bytes(K->n, 0))
    return set_error(SPSVM_ERR_OOM, "active_diff: scratch too small");
  cudaStream_t s = as_stream(stream);
  const int64_t n = K->n;
  if (n == 0) {
    SPSVM_CUDA_TRY(cudaMemsetAsync(k_dev, 0, sizeof(int32_t), s));
    return SPSVM_OK;
  }
  const int64_t sb = ceil_div(n, SC_PTS);
  int32_t* counts = static_cast<int32_t*>(scratch);
  // the compaction's scratch: counts, partial sums (one slot for no rows), list
  int64_t* total = reinterpret_cast<int64_t*>(static_cast<char*>(scratch) + round_up(sb * 4, 256));
  const int64_t ysplit_max = ceil_div(n, CP_T) < 1024 ? ceil_div(n, CP_T) : 1024;
  int32_t* list = reinterpret_cast<int32_t*>(
      static_cast<char*>(scratch) + round_up(sb * 4, 256) + round_up(ysplit_max * 16, 256));
  SPSVM_TRY(launch_scan(active, ref, n, counts, nullptr, list, total, nullptr, nullptr, s));
  store_count<<<1, 1, 0, s>>>(total, k_dev);
  SPSVM_LAUNCH_CHECK();
  if (kmax > 0 && K->rows > 0) {
    diff_gather<<<(unsigned)min64(K->rows, 4 * (int64_t)sm_count()), 128, 0, s>>>(
        view(K), K->rows, list, k_dev, kmax, active, Wt, ldw, sign);
    SPSVM_LAUNCH_CHECK();
  }
  return SPSVM_OK;
}
