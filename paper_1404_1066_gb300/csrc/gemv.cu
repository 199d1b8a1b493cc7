// HBM-bound passes over the stored kernel matrix K_nJ (basis-major):
//   * o = K_nJ beta with the active set, loss and error count of Eq. 4;
//   * u = K_nJ v (line-search direction);
//   * active-set compaction K_SJ with the masked transposed products
//     K_SJ^T w (gradient and Newton right-hand side of Eq. 4).
// Products are FP32; every 32 terms the running sum is promoted to FP64.
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
// bytes in flight).
template <int FMT>
__device__ __forceinline__ void load2(const KView& K, int64_t j, int64_t i, float k[2]) {
  if (FMT == SPSVM_FP32) {
    const float2 a = *reinterpret_cast<const float2*>(static_cast<const float*>(K.data) + j * K.ld + i);
    k[0] = a.x;
    k[1] = a.y;
  } else {
    const uint16_t* base = static_cast<const uint16_t*>(K.data);
    const uint32_t h = *reinterpret_cast<const uint32_t*>(base + j * K.ld + i);
    const uint32_t l = *reinterpret_cast<const uint32_t*>(base + K.plane + j * K.ld + i);
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
// shared memory.  HBM (or L2) bound: n = 30,000, 1,024 rows (123 MB) 29 us, 116
// with 59 blocks.
constexpr int GV_CLUSTER = 8;
template <int FMT>
__device__ __forceinline__ bool cluster_products(const KView& K, int64_t rows, int64_t n,
                                                 const double* __restrict__ v, int64_t i, float* vs,
                                                 double (*red)[GV_P], double acc[GV_P]) {
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int64_t per = ceil_div(ceil_div(rows, (int64_t)GV_CHUNK), (int64_t)cs) * GV_CHUNK;
  const int64_t j0 = min64(rows, rank * per);
  KView Kr = K;
  if (FMT == SPSVM_FP32) Kr.data = static_cast<const float*>(K.data) + j0 * K.ld;
  else Kr.data = static_cast<const uint16_t*>(K.data) + j0 * K.ld;
  row_products<FMT>(Kr, min64(rows, j0 + per) - j0, n, v + j0, i, vs, acc);
  if (cs == 1) return true;
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

// o = K beta (or given), active flags, per-block loss / errors / |S|.
template <int FMT>
__global__ void __launch_bounds__(GV_T) outputs_kernel(
    KView K, int64_t rows, int64_t n, const double* __restrict__ beta,
    const float* __restrict__ y, float* __restrict__ o, uint8_t* __restrict__ active,
    double* __restrict__ part, int accumulate) {
  __shared__ float vs[GV_BETA];
  __shared__ double sh[32];
  __shared__ double red[GV_T][GV_P];
  const int64_t tile = blockIdx.x / cg::this_cluster().num_blocks();
  const int64_t i = (tile * GV_T + threadIdx.x) * GV_P;
  double acc[GV_P];
  if (beta && !cluster_products<FMT>(K, rows, n, beta, i, vs, red, acc)) return;
  double loss = 0.0, err = 0.0, act = 0.0;
  {
#pragma unroll
    for (int p = 0; p < GV_P; ++p) {
      const int64_t ii = i + p;
      if (ii >= n) break;
      float oi;
      if (beta) {
        oi = accumulate ? (float)((double)o[ii] + acc[p]) : (float)acc[p];
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

template <int FMT>
__global__ void __launch_bounds__(GV_T) gemv_kernel(KView K, int64_t rows, int64_t n,
                                                    const double* __restrict__ v,
                                                    float* __restrict__ u, int accumulate) {
  __shared__ float vs[GV_BETA];
  __shared__ double red[GV_T][GV_P];
  const int64_t i = ((int64_t)(blockIdx.x / cg::this_cluster().num_blocks()) * GV_T + threadIdx.x) * GV_P;
  double acc[GV_P];
  if (!cluster_products<FMT>(K, rows, n, v, i, vs, red, acc)) return;
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

// The scanned flag of point i: active[i], or with ref, active[i] != ref[i].
__device__ __forceinline__ int scan_flag(const uint8_t* __restrict__ active,
                                         const uint8_t* __restrict__ ref, int64_t i) {
  return ref ? (active[i] != ref[i]) : active[i];
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

// Exclusive scan of block counts in one block; writes the total to *total.
__global__ void scan_blocks(int32_t* __restrict__ counts, int64_t nb, int64_t* __restrict__ total) {
  __shared__ int32_t sh[1024];
  __shared__ int64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t b0 = 0; b0 < nb; b0 += blockDim.x) {
    const int64_t b = b0 + threadIdx.x;
    const int32_t v = (b < nb) ? counts[b] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int off = 1; off < (int)blockDim.x; off <<= 1) {
      int32_t add = (threadIdx.x >= (unsigned)off) ? sh[threadIdx.x - off] : 0;
      __syncthreads();
      sh[threadIdx.x] += add;
      __syncthreads();
    }
    const int32_t incl = sh[threadIdx.x];
    if (b < nb) counts[b] = (int32_t)(carry + incl - v);
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry += incl;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void scan_write(const uint8_t* __restrict__ active, const uint8_t* __restrict__ ref,
                           int64_t n, const int32_t* __restrict__ offsets, int32_t* __restrict__ pos,
                           int32_t* __restrict__ list) {
  __shared__ int32_t sh[SC_PTS];
  const int64_t base = (int64_t)blockIdx.x * SC_PTS;
  for (int p = 0; p < 4; ++p) {
    const int64_t i = base + threadIdx.x * 4 + p;
    sh[threadIdx.x * 4 + p] = (i < n) ? scan_flag(active, ref, i) : 0;
  }
  __syncthreads();
  // sequential scan per thread over its 4, then block scan of thread sums
  int32_t local[4], run = 0;
  for (int p = 0; p < 4; ++p) { local[p] = run; run += sh[threadIdx.x * 4 + p]; }
  __shared__ int32_t ts[SC_T];
  ts[threadIdx.x] = run;
  __syncthreads();
  for (int off = 1; off < SC_T; off <<= 1) {
    int32_t add = (threadIdx.x >= (unsigned)off) ? ts[threadIdx.x - off] : 0;
    __syncthreads();
    ts[threadIdx.x] += add;
    __syncthreads();
  }
  const int32_t excl = ts[threadIdx.x] - run + offsets[blockIdx.x];
  for (int p = 0; p < 4; ++p) {
    const int64_t i = base + threadIdx.x * 4 + p;
    if (i < n) {
      if (pos) pos[i] = excl + local[p];
      if (sh[threadIdx.x * 4 + p]) list[excl + local[p]] = (int32_t)i;   // flagged indices, in order
    }
  }
}

// ---- compaction + masked transposed products ---------------------------
// One block: 32 basis rows (each warp four of them) over a slice of the
// compact columns.  A lane takes two pairs of adjacent compact columns per
// step through the list of active indices, so every lane carries an active
// point whatever their density, a row's reads cover a contiguous stretch of
// K (16 loads in flight per lane) and its writes are whole 128-byte lines.
// The weighted sums are FP32 over 32 terms, then a compensated pair, and one
// FP64 reduction per warp.  Bound by HBM: at n = 200,000, 2,048 rows, 43%
// active (1.64 GB read, 0.70 GB written) 0.38 ms, 6.1 TB/s; a thread per point
// of every row, 57% of them idle, with two-byte writes took 3.36 ms.
constexpr int CP_T = 256;
constexpr int CP_WARPS = CP_T / 32;
constexpr int CP_R = 4;                      // basis rows per warp
constexpr int CP_ROWS = CP_WARPS * CP_R;     // basis rows per block
constexpr int CP_Q = 128;                    // compact columns per step
constexpr int CP_CHUNK = 8;                  // steps summed in FP32 (4 terms each)
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
        f1[r] = fmaf(a[p], v[r][p], f1[r]);
        f2[r] = fmaf(c[p], v[r][p], f2[r]);
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

// Sums the slices' partials in order.
__global__ void compact_finish(const double2* __restrict__ part, int64_t slices, int64_t rows,
                               double* w1out, double* w2out, const int64_t* __restrict__ ns_dev) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= rows) return;
  const int64_t ns = *ns_dev;
  const int64_t used = max64(1, ceil_div(ns, cp_slice(ns, slices)));
  double a = 0.0, b = 0.0;
  for (int64_t s = 0; s < used; ++s) {
    const double2 p = part[s * rows + j];
    a += p.x;
    b += p.y;
  }
  if (w1out) w1out[j] = a;
  if (w2out) w2out[j] = b;
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
// Blocks per tile of points: enough for four blocks per SM, each with a chunk
// of rows at least.
int gv_cluster(int64_t tiles, int64_t rows) {
  int cs = 1;
  while (2 * cs <= GV_CLUSTER && tiles * cs < 4 * (int64_t)sm_count() &&
         2 * cs <= ceil_div(rows, (int64_t)GV_CHUNK))
    cs *= 2;
  return cs;
}
template <class Kern, class... Args>
cudaError_t gv_launch(Kern kern, int64_t tiles, int cs, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(tiles * cs));
  cfg.blockDim = dim3(GV_T);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
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
  const int cs = beta ? gv_cluster(blocks, K->rows) : 1;
  SPSVM_CUDA_TRY(gv_launch(K->format == SPSVM_FP32 ? outputs_kernel<SPSVM_FP32> : outputs_kernel<SPSVM_BF16SPLIT>,
                           blocks, cs, s, view(K), K->rows, K->n, beta, y, o, active, part, 0));
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
  SPSVM_CUDA_TRY(gv_launch(K->format == SPSVM_FP32 ? gemv_kernel<SPSVM_FP32> : gemv_kernel<SPSVM_BF16SPLIT>,
                           blocks, gv_cluster(blocks, K->rows), as_stream(stream), view(K), K->rows, K->n,
                           v, u, accumulate));
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

namespace {
// Slices of the compact columns: about eight blocks per SM in all, but no
// slice below CP_MIN_SLICE points (its sums end in an FP64 warp reduction).
int64_t compact_slices(int64_t n, int64_t rows) {
  const int64_t want = ceil_div(8 * (int64_t)sm_count(), max64(1, ceil_div(rows, (int64_t)CP_ROWS)));
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
                               int32_t* pos, void* scratch, size_t scratch_bytes, void* stream) {
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
    scan_count<<<(unsigned)sb, SC_T, 0, s>>>(active, nullptr, n, counts);
    SPSVM_LAUNCH_CHECK();
    scan_blocks<<<1, 1024, 0, s>>>(counts, sb, n_active);
    SPSVM_LAUNCH_CHECK();
    scan_write<<<(unsigned)sb, SC_T, 0, s>>>(active, nullptr, n, counts, pos, list);
    SPSVM_LAUNCH_CHECK();
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
      compact_finish<<<(unsigned)ceil_div(K->rows, 256), 256, 0, s>>>(part, slices, K->rows, w1out,
                                                                      w2out, n_active);
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
  scan_count<<<(unsigned)sb, SC_T, 0, s>>>(active, ref, n, counts);
  SPSVM_LAUNCH_CHECK();
  scan_blocks<<<1, 1024, 0, s>>>(counts, sb, total);
  SPSVM_LAUNCH_CHECK();
  scan_write<<<(unsigned)sb, SC_T, 0, s>>>(active, ref, n, counts, nullptr, list);
  SPSVM_LAUNCH_CHECK();
  store_count<<<1, 1, 0, s>>>(total, k_dev);
  SPSVM_LAUNCH_CHECK();
  if (kmax > 0 && K->rows > 0) {
    diff_gather<<<(unsigned)min64(K->rows, 4 * (int64_t)sm_count()), 128, 0, s>>>(
        view(K), K->rows, list, k_dev, kmax, active, Wt, ldw, sign);
    SPSVM_LAUNCH_CHECK();
  }
  return SPSVM_OK;
}
