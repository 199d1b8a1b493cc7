// Exact line search along the Newton direction d (Section 4's Newton
// reoptimisation of Eq. 4; f is convex and piecewise quadratic along a
// line).  phi'(t) = a0 + a1 t - sum_i v_i max(0, m_i - t v_i) is piecewise
// linear and nondecreasing; each pass evaluates it on 33 points over the
// current bracket and notes which of the 32 cells hold breakpoints m_i / v_i,
// so that the root is solved exactly on a cell free of breakpoints.
// The first pass is dense around t = 1, where Newton steps end; a later one
// puts its points around the secant estimate of the root, as close as the
// change of slope between neighbouring cells allows, with the cell's ends as
// the outer points, so the bracket shrinks by hundreds a pass.  The whole
// search is one launch: all CTAs make a pass and write their partial sums,
// and after one grid barrier every CTA adds up the same partials in the same
// order and takes the same decision.
//
// Bound by latency: a pass is a loop over the points, a barrier and the sum.
// n = 30,000 25 us, n = 500,000 41 us; with a uniform grid on the bracket
// (32-fold a pass), counts by shared atomics with FP64 divisions and two
// barriers over 304 CTAs a pass it took 103 us and 150.
#include "internal.h"

namespace spsvm {

namespace {

constexpr int LP = 33;          // grid points per pass
constexpr int LC = LP - 1;      // cells
constexpr int LV = LP + 2;      // summed values: phi' sums, a0, a1
constexpr int LT = 512;
constexpr int LW = LT / 32;
constexpr int kPerCta = 4 * LT; // points that pay another CTA in the barrier
constexpr int kMaxPasses = 64;  // the search needs at most 1 + 12 + 13
constexpr int kOne = 16;        // the first grid's point at t = 1

// The points of every grid are FP32 numbers: the sums are taken there, so a
// point rounded for them alone would shift the root by up to 2^-24.
__constant__ float kFirstGrid[LP] = {
    0.0f,   0.25f,  0.5f,   0.65f, 0.75f, 0.82f,  0.87f, 0.91f, 0.94f, 0.96f, 0.97f,
    0.98f,  0.986f, 0.991f, 0.995f, 0.998f, 1.0f, 1.002f, 1.005f, 1.009f, 1.014f, 1.02f,
    1.03f,  1.04f,  1.06f,  1.09f, 1.13f, 1.18f,  1.25f, 1.35f, 1.5f,  1.75f, 2.0f};

// Result of the search (CTA 0 writes it).
struct LsState {
  double t;
  int32_t err;
};

// Scratch after the state and the barrier words: two buffers (passes take
// them in turn: a CTA is at most one pass ahead) of the CTAs' partials,
// value-major: LV pairs and the mask of the cells with breakpoints.
constexpr size_t kLsHead = 256;                       // state, barrier

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of all CTAs of a cooperative launch: each adds one to a counter that
// only grows, and waits for `target` of them (one hop from the last arrival
// to the waiters).  Gives up after about a second and returns true.
__device__ bool grid_barrier(unsigned* count, unsigned target) {
  __shared__ int to_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    int to = 0;
    for (uint32_t it = 0; ld_acquire_u32(count) < target; ++it) {
      if (it >= (1u << 22)) {
        to = 1;
        break;
      }
      if (it >= 32) __nanosleep(64);
    }
    to_s = to;
  }
  __syncthreads();
  return to_s != 0;
}

__device__ __forceinline__ void pair_of(double x, float& hi, float& lo) {
  hi = (float)x;
  lo = (float)(x - (double)hi);
}

// One point (m, v) against the grid: F_k += v max(0, m - T_k v), and the cell
// that strictly holds its breakpoint m / v into the mask (one on a grid point
// splits nothing).  The breakpoint is placed by its FP32 quotient: one within
// a few rounding errors of a grid point may count in either cell.
__device__ __forceinline__ void ls_point(float m, float v, const float (&tk)[LP], const float* T,
                                         float (&F)[LP], unsigned& cells) {
  if (v == 0.0f) return;
#pragma unroll
  for (int k = 0; k < LP; ++k) F[k] = fmaf(v, fmaxf(0.0f, fmaf(-tk[k], v, m)), F[k]);
  const float b = __fdividef(m, v);
  if (!(b > tk[0] && b < tk[LC])) return;
  int c = 0;
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1)
    if (b > T[c + h]) c += h;
  if (b < T[c + 1]) cells |= 1u << c;
}

// One pass of this CTA over its points for the grid T: partial sums in
// redF[warp][k] (FP32 over four lanes, then compensated pairs), the cells that hold breakpoints in
// redC[warp].  The thread's first LK points (m, v) are in registers, the rest
// are read LK at a time.
constexpr int LK = 4;
__device__ void ls_pass(const float* __restrict__ o, const float* __restrict__ u,
                        const float* __restrict__ y, int64_t n, const float* T, const float (&km)[LK],
                        const float (&kv)[LK], float2 (*redF)[LV], unsigned* redC) {
  float tk[LP], F[LP];
#pragma unroll
  for (int k = 0; k < LP; ++k) {
    tk[k] = T[k];
    F[k] = 0.f;
  }
  unsigned cells = 0;
#pragma unroll
  for (int p = 0; p < LK; ++p) ls_point(km[p], kv[p], tk, T, F, cells);
  const int64_t step = (int64_t)gridDim.x * LT;
  for (int64_t i = (int64_t)blockIdx.x * LT + threadIdx.x + LK * step; i < n; i += LK * step) {
    float m[LK], v[LK];
#pragma unroll
    for (int p = 0; p < LK; ++p) {
      const bool in = i + p * step < n;
      const float yi = in ? y[i + p * step] : 0.f;
      m[p] = in ? 1.0f - yi * o[i + p * step] : 0.f;
      v[p] = in ? yi * u[i + p * step] : 0.f;
    }
#pragma unroll
    for (int p = 0; p < LK; ++p) ls_point(m[p], v[p], tk, T, F, cells);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  cells = __reduce_or_sync(0xffffffffu, cells);
  // warp sums: grid points 0..31 by the column-sum exchange (lane k ends with
  // point k), point 32 by a plain reduction.  In pairs from four lanes on: at t =
  // 1 the terms have one sign, and FP32 sums over the warp's 128 of them left t
  // farther from 64 bits than one point a thread did (n = 5,000, mean of 160
  // directions: 8.2e-10 and 6.2e-10; this 5.8e-10).
  const float2 f32 = warp_column_sum(F[LP - 1]);
  float v32[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) v32[k] = F[k];
  redF[w][lane] = warp_column_sums(v32, lane);
  if (lane == 0) {
    redF[w][LP - 1] = f32;
    redC[w] = cells;
  }
}

__global__ void __launch_bounds__(LT, 1) ls_search(const float* __restrict__ o,
                                                   const float* __restrict__ u,
                                                   const float* __restrict__ y, int64_t n,
                                                   const double* __restrict__ d,
                                                   const int64_t* __restrict__ J, int32_t m,
                                                   double lambda, char* __restrict__ work,
                                                   LsState* __restrict__ st, unsigned* __restrict__ bar,
                                                   const double* __restrict__ b0,
                                                   double* __restrict__ t_dev,
                                                   int32_t* __restrict__ err_dev) {
  __shared__ double T[LP];
  __shared__ float Tf[LP];
  __shared__ float2 redF[LW][LV];
  __shared__ float2 redA[LW][2];
  __shared__ unsigned redC[LW];
  __shared__ float2 Fs[LV];
  __shared__ unsigned cells_s;
  __shared__ int done_s;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const unsigned nb = gridDim.x;
  float2* PF0 = reinterpret_cast<float2*>(work + kLsHead);
  unsigned* PC0 = reinterpret_cast<unsigned*>(PF0 + (size_t)2 * LV * nb);
  // warp 0 of every CTA carries the search state across passes (all CTAs
  // see the same sums and take the same decisions)
  double a0 = 0.0, a1 = 0.0, tt = 0.0;
  int phase = 0, grow = 0, depth = 0, err = 0;
  bool aimed = false;   // the grid is dense around an estimate, not even
  if (t < LP) T[t] = kFirstGrid[t];
  float km[LK], kv[LK];
#pragma unroll
  for (int p = 0; p < LK; ++p) {
    const int64_t i = (int64_t)blockIdx.x * LT + t + (int64_t)p * nb * LT;
    const float yi = i < n ? y[i] : 0.f;
    km[p] = i < n ? 1.0f - yi * o[i] : 0.f;
    kv[p] = i < n ? yi * u[i] : 0.f;
  }
  for (int pass = 0; pass < kMaxPasses; ++pass) {
    __syncthreads();
    if (t < LP) Tf[t] = (float)T[t];
    __syncthreads();
    ls_pass(o, u, y, n, Tf, km, kv, redF, redC);
    float2* PF = PF0 + (size_t)(pass & 1) * LV * nb;
    unsigned* PC = PC0 + (size_t)(pass & 1) * nb;
    if (pass == 0) {
      // a0 = lambda d^T K_JJ beta, a1 = lambda d^T K_JJ d: (K_JJ beta)_k = o
      // at basis point k (minus the bias b0 = beta_0 when slot 0, point
      // index -1, holds it; that slot has no regulariser row)
      const double bb = b0 ? *b0 : 0.0, db = b0 ? d[0] : 0.0;
      double s0 = 0.0, s1 = 0.0;
      for (int64_t k = (int64_t)blockIdx.x * LT + t; k < m; k += (int64_t)nb * LT) {
        const int64_t j = J[k];
        if (j < 0) continue;
        s0 += d[k] * ((double)o[j] - bb);
        s1 += d[k] * ((double)u[j] - db);
      }
      float h[2], l[2];
      pair_of(s0, h[0], l[0]);
      pair_of(s1, h[1], l[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int x = 16; x > 0; x >>= 1) {
          const float oh = __shfl_xor_sync(0xffffffffu, h[q], x), ol = __shfl_xor_sync(0xffffffffu, l[q], x);
          pair_add(h[q], l[q], make_float2(oh, ol));
        }
        if (lane == 0) redA[w][q] = make_float2(h[q], l[q]);
      }
    }
    __syncthreads();
    if (t < LV && (t < LP || pass == 0)) {
      float h = 0.f, l = 0.f;
      for (int q = 0; q < LW; ++q) {
        if (t < LP) pair_add(h, l, redF[q][t]);
        else pair_add(h, l, redA[q][t - LP]);
      }
      PF[(size_t)t * nb + blockIdx.x] = make_float2(h, l);
    } else if (t == 64) {
      unsigned c = 0;
      for (int q = 0; q < LW; ++q) c |= redC[q];
      PC[blockIdx.x] = c;
    }
    if (nb > 1) {
      if (grid_barrier(bar, nb * (unsigned)(pass + 1))) {
        err = 1;
        break;
      }
    } else {
      __syncthreads();
    }
    // the sums over the CTAs: warp w takes values w, w + LW, w + 2 LW (their
    // loads together), the last warp also the cells
    static_assert(LV <= 3 * LW, "three values a warp");
    {
      float h[3], l[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) h[q] = l[q] = 0.f;
      for (unsigned b = lane; b < nb; b += 32) {
        float2 x[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int v = w + q * LW;
          x[q] = v < LP || (v < LV && pass == 0) ? __ldcg(&PF[(size_t)v * nb + b]) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) pair_add(h[q], l[q], x[q]);
      }
      if (w == LW - 1) {
        unsigned c = 0;
        for (unsigned b = lane; b < nb; b += 32) c |= __ldcg(&PC[b]);
        c = __reduce_or_sync(0xffffffffu, c);
        if (lane == 0) cells_s = c;
      }
#pragma unroll
      for (int x = 16; x > 0; x >>= 1)
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float oh = __shfl_xor_sync(0xffffffffu, h[q], x), ol = __shfl_xor_sync(0xffffffffu, l[q], x);
          pair_add(h[q], l[q], make_float2(oh, ol));
        }
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (w + q * LW < LV) Fs[w + q * LW] = make_float2(h[q], l[q]);
      }
    }
    __syncthreads();
    if (w == 0) {
      if (pass == 0) {
        a0 = lambda * pair_value(Fs[LP].x, Fs[LP].y);
        a1 = lambda * pair_value(Fs[LP + 1].x, Fs[LP + 1].y);
      }
      // lane k: phi' at point k and at point k + 1
      const double tk = T[lane], tn = T[lane + 1];
      const double dk = a0 + a1 * tk - pair_value(Fs[lane].x, Fs[lane].y);
      const double dlast = a0 + a1 * T[LC] - pair_value(Fs[LC].x, Fs[LC].y);
      double dn = __shfl_down_sync(0xffffffffu, dk, 1);
      if (lane == 31) dn = dlast;
      int done = 0;
      bool next = false;
      // lane k: the slope of cell k
      const float slope = (float)(dn - dk) / (float)(tn - tk);
      if (phase == 0) {
        const double d0 = __shfl_sync(0xffffffffu, dk, 0), d1 = __shfl_sync(0xffffffffu, dk, kOne);
        if (!(d0 < 0.0)) {
          tt = 0.0;
          done = 1;
        } else if (fabs(d1) <= 1e-6 * fabs(d0)) {
          tt = 1.0;
          done = 1;
        } else {
          phase = 1;
        }
      }
      if (!done && phase == 1) {   // grow the bracket until phi' >= 0 at its right end
        if (dlast < 0.0 && grow < 12) {
          ++grow;
          next = true;
        } else if (dlast < 0.0) {
          tt = T[LC];   // phi still decreasing: take the far end (bounded)
          done = 1;
        } else {
          phase = 2;
        }
      }
      __syncwarp();
      // points 0 and LC the ends lo and hi, 1 .. LC - 1 even over [A, B],
      // rounded to FP32 (lo and hi are)
      auto grid = [&](double lo, double hi, double A, double B) {
        T[lane] = lane == 0 ? lo : (double)(float)(A + (B - A) * (1.0 / (LC - 2)) * (lane - 1));
        if (lane == 31) T[31] = (double)(float)B;
        if (lane == 0) T[LC] = hi;
        aimed = A > lo || B < hi;
      };
      if (next) {
        // [hi, 8 hi], around where the last cell's slope meets zero
        const double lo = T[LC], hi = 8.0 * lo;
        const float run = (float)-dlast / __shfl_sync(0xffffffffu, slope, LC - 1);
        const double step = run > 0.0f && run < 1e30f ? (double)run : 0.0;
        __syncwarp();
        // (past it as a rule: points leave the active set on the way)
        if (step > 0.0 && lo + 2.5 * step < hi) grid(lo, hi, lo + 0.75 * step, lo + 2.5 * step);
        else grid(lo, hi, lo, hi);
      } else if (!done) {   // the cell holding the root
        const unsigned up = __ballot_sync(0xffffffffu, !(dn < 0.0));
        const int k = up ? __ffs(up) - 1 : LC - 1;
        const double tl = __shfl_sync(0xffffffffu, tk, k), tr = __shfl_sync(0xffffffffu, tn, k);
        const double fl = __shfl_sync(0xffffffffu, dk, k), fr = __shfl_sync(0xffffffffu, dn, k);
        const double h = tr - tl, rise = fr - fl;
        double root = tl;
        if (rise > 0.0) {
          // -fl / rise by an FP32 quotient and one FP64 correction (an FP64
          // division takes a thousand cycles here)
          const float inv = 1.0f / (float)rise;
          double q = (double)((float)-fl * inv);
          q += (-fl - q * rise) * (double)inv;
          root = tl + q * h;
        }
        if (!(root > tl)) root = tl;
        if (root > tr) root = tr;
        if (!((cells_s >> k) & 1u) || depth >= 12 || !(rise > 0.0) || h <= 2e-7 * tr || pass == kMaxPasses - 1) {
          tt = root;
          done = 1;
        } else {
          // slopes of the neighbouring cells bound the secant's error; a root
          // outside the points it set gets an even grid over its cell
          const float mid = (float)rise / (float)h;
          float sl = __shfl_sync(0xffffffffu, slope, k > 0 ? k - 1 : k);
          float sr = __shfl_sync(0xffffffffu, slope, k < LC - 1 ? k + 1 : k);
          if (!(fabsf(sl) < 1e30f)) sl = 0.0f;   // an empty cell says nothing
          if (!(fabsf(sr) < 1e30f)) sr = 2.0f * mid;
          float rel = fabsf(sr - sl) / mid;
          rel = rel < 1.0f / 256 ? 1.0f / 256 : (rel < 1.0f ? rel : 1.0f);
          const double wd = 0.5 * h * rel;
          if (aimed && (k == 0 || k == LC - 1)) grid(tl, tr, tl, tr);
          else grid(tl, tr, fmax(tl, root - wd), fmin(tr, root + wd));
          ++depth;
        }
      }
      if (lane == 0) done_s = done;
    }
    __syncthreads();
    if (done_s) break;
  }
  if (blockIdx.x == 0 && t == 0) {
    st->t = err ? 0.0 : tt;
    st->err = err;
    if (t_dev) *t_dev = err ? 0.0 : tt;
    if (err_dev) *err_dev = err;
  }
}

// CTAs of a search over n points: at most one per SM (they must all be
// resident for the barrier).
int ls_grid(int64_t n) {
  const int64_t want = ceil_div(n, (int64_t)kPerCta);
  return (int)max64(1, min64(want, (int64_t)sm_count()));
}

}  // namespace
}  // namespace spsvm

using namespace spsvm;

extern "C" size_t spsvm_line_scratch_bytes(int64_t n) {
  (void)n;
  return kLsHead + (size_t)(2 * sm_count()) * (LV * sizeof(float2) + sizeof(unsigned));
}

extern "C" int spsvm_line_search(const float* o, const float* u, const float* y, int64_t n,
                                 const double* d, const int64_t* J, int32_t m, double lambda,
                                 double* t_host, double* t_dev, void* scratch,
                                 size_t scratch_bytes, void* stream) {
  return spsvm::line_search_impl(o, u, y, n, d, J, m, lambda, t_host, t_dev, scratch, scratch_bytes,
                                 stream, nullptr);
}

namespace {
// Enqueues the search (the result in the scratch's state, and in t_dev and
// err_dev when given).
int ls_launch(const float* o, const float* u, const float* y, int64_t n, const double* d,
              const int64_t* J, int32_t m, double lambda, double* t_dev, int32_t* err_dev,
              void* scratch, size_t scratch_bytes, cudaStream_t s, const double* b0) {
  if (!scratch || scratch_bytes < spsvm_line_scratch_bytes(n))
    return set_error(SPSVM_ERR_OOM, "line_search: scratch too small");
  ProfScope prof(PROF_LINE, s, 12.0 * (double)n);
  const int grid = ls_grid(n);
  LsState* st = static_cast<LsState*>(scratch);
  unsigned* bar = reinterpret_cast<unsigned*>(static_cast<char*>(scratch) + 128);
  char* work = static_cast<char*>(scratch);
  void* args[] = {(void*)&o, (void*)&u, (void*)&y, (void*)&n, (void*)&d, (void*)&J, (void*)&m,
                  (void*)&lambda, (void*)&work, (void*)&st, (void*)&bar, (void*)&b0,
                  (void*)&t_dev, (void*)&err_dev};
  if (grid > 1) {
    SPSVM_CUDA_TRY(cudaMemsetAsync(scratch, 0, kLsHead, s));
    SPSVM_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)ls_search, dim3(grid), dim3(LT), args, 0, s));
  } else {
    SPSVM_CUDA_TRY(cudaLaunchKernel((const void*)ls_search, dim3(1), dim3(LT), args, 0, s));
  }
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}
}  // namespace

int spsvm::line_search_impl(const float* o, const float* u, const float* y, int64_t n,
                            const double* d, const int64_t* J, int32_t m, double lambda,
                            double* t_host, double* t_dev, void* scratch, size_t scratch_bytes,
                            void* stream, const double* b0) {
  if (!o || !u || !y || !d || !J || !t_host || n < 0 || m < 0)
    return set_error(SPSVM_ERR_ARG, "line_search: bad arguments");
  cudaStream_t s = as_stream(stream);
  SPSVM_TRY(ls_launch(o, u, y, n, d, J, m, lambda, t_dev, nullptr, scratch, scratch_bytes, s, b0));
  LsState h{};
  const ReadChunk c{&h, scratch, sizeof(h)};
  SPSVM_TRY(read_plain(s, &c, 1));
  if (h.err) return set_error(SPSVM_ERR_TIMEOUT, "line_search: grid barrier timed out");
  *t_host = h.t;
  return SPSVM_OK;
}

int spsvm::line_search_async(const float* o, const float* u, const float* y, int64_t n,
                             const double* d, const int64_t* J, int32_t m, double lambda,
                             double* t_dev, int32_t* err_dev, void* scratch, size_t scratch_bytes,
                             void* stream, const double* b0) {
  if (!o || !u || !y || !d || !J || !t_dev || !err_dev || n < 0 || m < 0)
    return set_error(SPSVM_ERR_ARG, "line_search: bad arguments");
  return ls_launch(o, u, y, n, d, J, m, lambda, t_dev, err_dev, scratch, scratch_bytes,
                   as_stream(stream), b0);
}
