// Kernel block and candidate scores in plain FP32 SIMT arithmetic (the
// SPSVM_FP32 form).  RBF kernel of Section 2 through the distance expansion
// ||x - z||^2 = ||x||^2 + ||z||^2 - 2 x^T z; the basis-vector score of
// Section 4 ("Basis vector selection") fused into the same tile loop.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "simt_tile.h"

namespace spsvm {

namespace {

constexpr int64_t PT = 128;   // points per tile

// Tiles of 64 (or 32) basis rows by 128 points: the points run along the
// tile's columns, so a warp's kernel values go out as 256 contiguous bytes of
// a basis row.  FP32 ALU bound for d past about 60: n = 100,000, d = 784, 64
// rows 0.214 ms (47 TFLOP/s, FMA pipe 69% of active cycles); tiles of 4 x 8
// outputs with scalar shared loads took 0.540 ms.
using Wide = simt::Tile<64, 128, 8>;
using Narrow = simt::Tile<32, 128, 4>;

template <class T, class RA, class RB>
__device__ __forceinline__ void rbf_rows(const float* __restrict__ X, int64_t n, int64_t ldx,
                                         const int64_t* __restrict__ idx, int64_t i0, int64_t c0,
                                         int32_t m, RA (&a)[T::LA], RB (&b)[T::LB]) {
#pragma unroll
  for (int u = 0; u < T::LA; ++u) {
    const int64_t c = c0 + T::load_row(u);
    a[u].p = c < m ? X + idx[c] * ldx : nullptr;
  }
#pragma unroll
  for (int u = 0; u < T::LB; ++u) {
    const int64_t i = i0 + T::load_row(u);
    b[u].p = i < n ? X + i * ldx : nullptr;
  }
}

template <class T, bool VEC>
__global__ void __launch_bounds__(T::NT, 3) kernel_block_simt(
    const float* __restrict__ X, int64_t n, int64_t d, int64_t ldx,
    const float* __restrict__ norms, const int64_t* __restrict__ idx, int32_t m,
    float gamma, void* out, int32_t format, int64_t ld, int64_t plane, int64_t row0) {
  __shared__ typename T::Smem sm;
  const int64_t i0 = (int64_t)blockIdx.x * T::TN, c0 = (int64_t)blockIdx.y * T::TM;
  simt::FloatRows<VEC> a[T::LA], b[T::LB];
  rbf_rows<T>(X, n, ldx, idx, i0, c0, m, a, b);
  uint64_t acc[T::RM][4];
  T::product(sm, a, b, 0, d, acc);
  float xn[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int64_t i = i0 + T::col(c);
    xn[c] = i < n ? norms[i] : 0.f;
  }
#pragma unroll
  for (int r = 0; r < T::RM; ++r) {
    const int64_t c = c0 + T::row(r);
    if (c >= m) continue;
    const float zn = norms[idx[c]];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t i = i0 + T::col(4 * h);
      const float2 lo = simt::unpack2(acc[r][2 * h]), hi = simt::unpack2(acc[r][2 * h + 1]);
      const float v[4] = {rbf_from_dot(xn[4 * h], zn, lo.x, gamma), rbf_from_dot(xn[4 * h + 1], zn, lo.y, gamma),
                          rbf_from_dot(xn[4 * h + 2], zn, hi.x, gamma), rbf_from_dot(xn[4 * h + 3], zn, hi.y, gamma)};
      const int64_t off = (row0 + c) * ld + i;
      if (format == SPSVM_FP32 && i + 4 <= n) {
        *reinterpret_cast<float4*>(static_cast<float*>(out) + off) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (i + e < n) kstore(out, format, plane, off + e, v[e]);
      }
    }
  }
}

// Per tile of 128 points: partial sums over i in S of (o_i - y_i) K_ic and
// K_ic^2 for the tile's candidates, written to part[tile][c] as two
// compensated pairs.  A
// thread sums 4 points at a time in FP32; everything wider is summed as
// compensated pairs (an FP64 warp sum per candidate would outweigh the tile's
// product at small d).
template <class T, bool VEC>
__global__ void __launch_bounds__(T::NT, 3) score_partials_simt(
    const float* __restrict__ X, int64_t n, int64_t d, int64_t ldx,
    const float* __restrict__ norms, const float* __restrict__ y,
    const float* __restrict__ o, const int64_t* __restrict__ idx, int32_t kappa,
    float gamma, float4* __restrict__ part) {
  __shared__ typename T::Smem sm;
  const int64_t i0 = (int64_t)blockIdx.x * T::TN, c0 = (int64_t)blockIdx.y * T::TM;
  simt::FloatRows<VEC> a[T::LA], b[T::LB];
  rbf_rows<T>(X, n, ldx, idx, i0, c0, kappa, a, b);
  uint64_t acc[T::RM][4];
  T::product(sm, a, b, 0, d, acc);
  float res[8], act[8], xn[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int64_t i = i0 + T::col(c);
    res[c] = act[c] = xn[c] = 0.f;
    if (i < n) {
      const float oi = o[i], yi = y[i];
      const bool s = yi * oi < 1.0f;
      res[c] = s ? (oi - yi) : 0.f;
      act[c] = s ? 1.f : 0.f;
      xn[c] = norms[i];
    }
  }
  // value 2 r (+ 1): the row's G (H) sum, as a pair
  constexpr int NV = 2 * T::RM;
  float hi[NV], lo[NV];
#pragma unroll
  for (int r = 0; r < T::RM; ++r) {
    const int64_t c = c0 + T::row(r);
    const float zn = c < kappa ? norms[idx[c]] : 0.f;
    float gs[2] = {0.f, 0.f}, hs[2] = {0.f, 0.f};
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const float2 dot = simt::unpack2(acc[r][p]);
      const float v0 = rbf_from_dot(xn[2 * p], zn, dot.x, gamma);
      const float v1 = rbf_from_dot(xn[2 * p + 1], zn, dot.y, gamma);
      gs[p >> 1] = fmaf(res[2 * p + 1], v1, fmaf(res[2 * p], v0, gs[p >> 1]));
      hs[p >> 1] = fmaf(act[2 * p + 1] * v1, v1, fmaf(act[2 * p] * v0, v0, hs[p >> 1]));
    }
    hi[2 * r] = gs[0];
    lo[2 * r] = 0.f;
    pair_add(hi[2 * r], lo[2 * r], gs[1]);
    hi[2 * r + 1] = hs[0];
    lo[2 * r + 1] = 0.f;
    pair_add(hi[2 * r + 1], lo[2 * r + 1], hs[1]);
  }
  // sums over the 16 threads of a row group: each exchange halves the values
  // a thread holds, then (NV < 16) the last lanes combine
  static_assert(T::TX == 16, "16 threads per row group");
  const int tx = T::tx();
  int mine = 0;
#pragma unroll
  for (int step = 0; step < 4; ++step) {
    const int h = 8 >> step, cnt = NV >> (step + 1);
    const bool up = (tx & h) != 0;
    if (cnt > 0) {
#pragma unroll
      for (int k = 0; k < NV / 2; ++k) {
        if (k >= cnt) break;
        const float gh = up ? hi[k] : hi[k + cnt], gl = up ? lo[k] : lo[k + cnt];
        float kh = up ? hi[k + cnt] : hi[k], kl = up ? lo[k + cnt] : lo[k];
        pair_add(kh, kl, __shfl_xor_sync(0xffffffffu, gh, h));
        hi[k] = kh;
        lo[k] = kl + __shfl_xor_sync(0xffffffffu, gl, h);
      }
      mine += up ? cnt : 0;
    } else {
      // both lanes end with the same pair: the lower lane's value first
      const float oh = __shfl_xor_sync(0xffffffffu, hi[0], h), ol = __shfl_xor_sync(0xffffffffu, lo[0], h);
      float kh = up ? oh : hi[0], kl = up ? ol : lo[0];
      pair_add(kh, kl, up ? hi[0] : oh);
      hi[0] = kh;
      lo[0] = kl + (up ? lo[0] : ol);
    }
  }
  const int64_t c = c0 + T::row(mine >> 1);
  if (c < kappa && (NV == 16 || (tx & 1) == 0))
    reinterpret_cast<float2*>(part + (int64_t)blockIdx.x * kappa + c)[mine & 1] = make_float2(hi[0], lo[0]);
}

// The 32-row tile where it wastes fewer rows, or where 64-row tiles would leave
// SMs with one block or none (d = 784, 64 rows: n = 20,000 75 us against 83;
// n = 30,000 110 against 85).
bool use_narrow(int64_t n, int64_t m) {
  return m <= 32 || 4 * ceil_div(n, PT) * ceil_div(m, (int64_t)64) < 5 * (int64_t)sm_count();
}

// g_k = lambda o[c] + sum_tiles G, h_k = lambda + sum_tiles H, delta = g^2/(2h),
// two candidates a block (a whole sector a partial), 256 threads over the
// partials of each, sums as compensated pairs.  256 candidates: 76 partials
// (split form, n = 500,000) 5 us; 3,907, one block a candidate in FP64, 12.
constexpr int SF_C = 2, SF_T = 512;
__global__ void __launch_bounds__(SF_T) score_finish(const float4* __restrict__ part, int64_t tiles,
                                                     int32_t kappa, const float* __restrict__ o,
                                                     const int64_t* __restrict__ idx, double lambda,
                                                     double* g, double* h, double* delta) {
  __shared__ float4 sh[SF_T / 32][SF_C];
  const int c = threadIdx.x % SF_C, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int k = blockIdx.x * SF_C + c;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (k < kappa) {
    constexpr int STEP = SF_T / SF_C, U = 16;
    for (int64_t t = threadIdx.x / SF_C; t < tiles; t += U * STEP) {
      float4 p[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        p[u] = t + u * STEP < tiles ? part[(t + u * STEP) * kappa + k] : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        pair_add(s.x, s.y, make_float2(p[u].x, p[u].y));
        pair_add(s.z, s.w, make_float2(p[u].z, p[u].w));
      }
    }
  }
#pragma unroll
  for (int x = SF_C; x < 32; x <<= 1) {
    const float a = __shfl_xor_sync(0xffffffffu, s.x, x), b = __shfl_xor_sync(0xffffffffu, s.y, x);
    const float d = __shfl_xor_sync(0xffffffffu, s.z, x), e = __shfl_xor_sync(0xffffffffu, s.w, x);
    pair_add(s.x, s.y, make_float2(a, b));
    pair_add(s.z, s.w, make_float2(d, e));
  }
  if (lane < SF_C) sh[w][c] = s;
  __syncthreads();
  if (threadIdx.x >= SF_C || k >= kappa) return;
  for (int q = 1; q < SF_T / 32; ++q) {
    pair_add(s.x, s.y, make_float2(sh[q][c].x, sh[q][c].y));
    pair_add(s.z, s.w, make_float2(sh[q][c].z, sh[q][c].w));
  }
  const double gg = lambda * (double)o[idx[k]] + pair_value(s.x, s.y);
  const double hh = lambda + pair_value(s.z, s.w);
  g[k] = gg;
  h[k] = hh;
  delta[k] = gg * gg / (2.0 * hh);
}

}  // namespace

int launch_kernel_block_simt(const spsvm_points* p, const int64_t* idx, int32_t m,
                             float gamma, spsvm_kmat* out, int64_t row0, cudaStream_t s) {
  if (m == 0 || p->n == 0) return SPSVM_OK;
  auto launch = [&](auto tile, auto vec) {
    using T = decltype(tile);
    const dim3 grid((unsigned)ceil_div(p->n, PT), (unsigned)ceil_div(m, T::TM));
    kernel_block_simt<T, decltype(vec)::value><<<grid, T::NT, 0, s>>>(
        p->X, p->n, p->d, p->ldx, p->norms, idx, m, gamma, out->data, out->format, out->ld,
        out->plane, row0);
  };
  const bool vec = simt::rows_aligned(p->X, p->ldx);
  if (use_narrow(p->n, m)) vec ? launch(Narrow{}, std::true_type{}) : launch(Narrow{}, std::false_type{});
  else vec ? launch(Wide{}, std::true_type{}) : launch(Wide{}, std::false_type{});
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

static void launch_score_simt(const spsvm_points* p, const float* y, const float* o,
                              const int64_t* idx, int32_t kappa, float gamma, float4* part,
                              cudaStream_t s) {
  auto launch = [&](auto tile, auto vec) {
    using T = decltype(tile);
    const dim3 grid((unsigned)ceil_div(p->n, PT), (unsigned)ceil_div(kappa, T::TM));
    score_partials_simt<T, decltype(vec)::value><<<grid, T::NT, 0, s>>>(
        p->X, p->n, p->d, p->ldx, p->norms, y, o, idx, kappa, gamma, part);
  };
  const bool vec = simt::rows_aligned(p->X, p->ldx);
  if (use_narrow(p->n, kappa)) vec ? launch(Narrow{}, std::true_type{}) : launch(Narrow{}, std::false_type{});
  else vec ? launch(Wide{}, std::true_type{}) : launch(Wide{}, std::false_type{});
}

}  // namespace spsvm

using namespace spsvm;

extern "C" size_t spsvm_kernel_block_scratch_bytes(int64_t m, int64_t d, int32_t precision) {
  if (m < 0 || d < 1 || precision != SPSVM_BF16SPLIT) return 0;
  return kernel_block_tc_scratch(m, round_up(d, 64));
}

extern "C" int spsvm_kernel_block(const spsvm_points* p, const int64_t* idx, int32_t m,
                                  float gamma, int32_t precision, spsvm_kmat* out,
                                  int64_t row0, void* scratch, size_t scratch_bytes,
                                  void* stream) {
  if (!p || !p->X || !p->norms || !idx) return set_error(SPSVM_ERR_ARG, "kernel_block: NULL pointer");
  SPSVM_TRY(check_kmat(out, "kernel_block"));
  if (m < 0 || row0 < 0 || row0 + m > out->rows || out->n != p->n || !(gamma > 0.f))
    return set_error(SPSVM_ERR_ARG, "kernel_block: m=%d row0=%lld rows=%lld n=%lld/%lld gamma=%g",
                     m, (long long)row0, (long long)out->rows, (long long)out->n,
                     (long long)p->n, (double)gamma);
  // algorithmic work: 2 n m d multiply-adds, times the six products of the split form
  ProfScope prof(PROF_KERNEL_BLOCK, as_stream(stream),
                 (precision == SPSVM_BF16SPLIT ? 12.0 : 2.0) * (double)p->n * m * (double)p->d);
  if (precision == SPSVM_BF16SPLIT) {
    if (!p->hi || !p->mid || !p->lo)
      return set_error(SPSVM_ERR_ARG, "kernel_block: BF16SPLIT needs the split planes of the points");
    return launch_kernel_block_tc(p, idx, m, gamma, out, row0, scratch, scratch_bytes,
                                  as_stream(stream));
  }
  if (precision != SPSVM_FP32) return set_error(SPSVM_ERR_ARG, "kernel_block: bad precision");
  return launch_kernel_block_simt(p, idx, m, gamma, out, row0, as_stream(stream));
}

namespace spsvm {
int launch_score_tc(const spsvm_points* p, const float* y, const float* o, const int64_t* idx,
                    int32_t kappa, float gamma, float4* part, int64_t* parts, void* zbuf,
                    size_t zbytes, cudaStream_t s);
int64_t score_tc_parts(int64_t n);
namespace {
// partial sums per candidate (of each tile of 128 points in FP32, at most as
// many in the tensor-core form), then room for the gathered candidate rows
size_t score_part_bytes(int64_t n, int32_t kappa) {
  const int64_t tiles = std::max<int64_t>(ceil_div(n, PT), score_tc_parts(n));
  return (size_t)round_up(tiles * (int64_t)kappa * (int64_t)sizeof(float4), 256);
}
}  // namespace
}  // namespace spsvm

extern "C" size_t spsvm_score_scratch_bytes(int64_t n, int64_t d, int32_t kappa) {
  if (n < 0 || kappa < 0 || d < 1) return 0;
  return score_part_bytes(n, kappa) + kernel_block_tc_scratch(kappa, round_up(d, 64));
}

extern "C" int spsvm_score_candidates(const spsvm_points* p, const float* y, const float* o,
                                      const int64_t* idx, int32_t kappa, float gamma,
                                      double lambda, int32_t precision, double* g, double* h,
                                      double* delta, void* scratch, size_t scratch_bytes,
                                      void* stream) {
  if (!p || !p->X || !p->norms || !y || !o || !idx || !g || !h || !delta)
    return set_error(SPSVM_ERR_ARG, "score_candidates: NULL pointer");
  if (kappa < 0 || p->n < 1 || !(gamma > 0.f) || !(lambda > 0.0))
    return set_error(SPSVM_ERR_ARG, "score_candidates: bad arguments");
  if (kappa == 0) return SPSVM_OK;
  const size_t need = spsvm_score_scratch_bytes(p->n, p->d, kappa);
  if (scratch_bytes < need || !scratch)
    return set_error(SPSVM_ERR_OOM, "score_candidates: scratch %zu < %zu", scratch_bytes, need);
  cudaStream_t s = as_stream(stream);
  ProfScope prof(PROF_SCORE, s, (precision == SPSVM_BF16SPLIT ? 12.0 : 2.0) * (double)p->n * kappa * (double)p->d);
  float4* part = static_cast<float4*>(scratch);
  int64_t parts = ceil_div(p->n, PT);
  if (precision == SPSVM_BF16SPLIT) {
    if (!p->hi || !p->mid || !p->lo)
      return set_error(SPSVM_ERR_ARG, "score_candidates: BF16SPLIT needs split planes");
    const size_t pb = score_part_bytes(p->n, kappa);
    SPSVM_TRY(launch_score_tc(p, y, o, idx, kappa, gamma, part, &parts, static_cast<char*>(scratch) + pb,
                              scratch_bytes - pb, s));
  } else if (precision == SPSVM_FP32) {
    launch_score_simt(p, y, o, idx, kappa, gamma, part, s);
    SPSVM_LAUNCH_CHECK();
  } else {
    return set_error(SPSVM_ERR_ARG, "score_candidates: bad precision");
  }
  score_finish<<<(unsigned)ceil_div(kappa, SF_C), SF_T, 0, s>>>(part, parts, kappa, o, idx, lambda, g, h, delta);
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free candidate scoring.  Some callers must not allocate device
// memory at all: a serving loop that has handed the whole HBM budget to a
// pool it does not own, a host framework whose allocator owns every device
// byte, or code running where cudaMalloc would synchronise the device at a
// moment it must not.  For them the score's per-tile partial sums live in a
// fixed array in this library's device memory instead of caller scratch.
// ---------------------------------------------------------------------------
#include <cuda.h>

#include <mutex>

namespace spsvm {
namespace {
// 16 MiB: enough for n = 500,000 points and 256 candidates in either form
// (16.2 MB of per-tile partial sums and gathered candidate rows).
constexpr size_t kScoreScratchMax = size_t(16) << 20;
// Held by every GPU that loads this library until the process exits.
__device__ __align__(256) unsigned char g_score_scratch[kScoreScratchMax];
std::mutex g_score_scratch_mu;
// the array's device address per device, with the context it was looked up
// in (a context torn down and made again, e.g. by cudaDeviceReset, may load
// the module at another address: the set-up then runs again)
void* g_score_scratch_ptr[64] = {};
CUcontext g_score_scratch_ctx[64] = {};

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
CtxGetCurrentFn ctx_get_current() {
  static const CtxGetCurrentFn fn = []() {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<CtxGetCurrentFn>(f);
    cudaGetLastError();
    return (CtxGetCurrentFn) nullptr;
  }();
  return fn;
}
}  // namespace
}  // namespace spsvm

extern "C" int spsvm_score_candidates_noalloc(const spsvm_points* p, const float* y,
                                              const float* o, const int64_t* idx, int32_t kappa,
                                              float gamma, double lambda, int32_t precision,
                                              double* g, double* h, double* delta, void* stream) {
  if (!p || kappa < 0 || p->n < 1)
    return set_error(SPSVM_ERR_ARG, "score_candidates_noalloc: bad arguments");
  const size_t need = spsvm_score_scratch_bytes(p->n, p->d, kappa);
  if (need > kScoreScratchMax)
    return set_error(SPSVM_ERR_ARG,
                     "score_candidates_noalloc: n=%lld, d=%lld, kappa=%d need %zu bytes of "
                     "scratch, more than the fixed %zu-byte array; use spsvm_score_candidates",
                     (long long)p->n, (long long)p->d, kappa, need, kScoreScratchMax);
  int dev = 0;
  SPSVM_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return set_error(SPSVM_ERR_ARG, "score_candidates_noalloc: device %d", dev);
  void* ptr = nullptr;
  {
    // set-up on the first call on this device (current), and again when the
    // device's context is not the one of the last set-up: look up the
    // array's device address
    CUcontext ctx = nullptr;
    if (auto fn = ctx_get_current()) fn(&ctx);
    std::lock_guard<std::mutex> lk(g_score_scratch_mu);
    if (!g_score_scratch_ptr[dev] || g_score_scratch_ctx[dev] != ctx) {
      void* a = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&a, g_score_scratch);
      if (e != cudaSuccess || !a)
        return set_error(SPSVM_ERR_CUDA, "score_candidates_noalloc: cudaGetSymbolAddress: %s",
                         cudaGetErrorString(e));
      g_score_scratch_ptr[dev] = a;
      g_score_scratch_ctx[dev] = ctx;
    }
    ptr = g_score_scratch_ptr[dev];
  }
  return spsvm_score_candidates(p, y, o, idx, kappa, gamma, lambda, precision, g, h, delta, ptr,
                                kScoreScratchMax, stream);
}
