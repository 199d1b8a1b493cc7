// Triangular solves and refinement of the mixed Newton solve (Section 4's
// reoptimisation).  A chain of 64-row blocks costs a hand-off between CTAs
// per block (2 us; 131 us per solve at m = 4,096), so diagonal
// blocks of up to 1,024 rows are inverted first (work that fills the GPU, once
// per factor), and a solve is a handful of matrix-vector products over the
// whole grid with a barrier after each.
#include "refine.h"
#include "simt_tile.h"

namespace spsvm {

namespace {

// ---- block inverses --------------------------------------------------------
constexpr int IB = 64;       // blocks inverted directly
constexpr int IP = IB + 4;   // shared row pitch, 16-byte aligned
constexpr int IT = 256;

// Inverse X of one 64 x 64 lower block: its four 16 x 16 diagonal blocks by
// one lane per column, then 16 -> 32 -> 64 by X21 = -X22 (L21 X11).  Latency
// bound: 7 us; row by row with a barrier per row it took 23.
__global__ void __launch_bounds__(IT) inverse64(float* __restrict__ L, int64_t ldl, int64_t m,
                                                float* __restrict__ W, float* __restrict__ WT,
                                                int64_t NI) {
  __shared__ __align__(16) float Ls[IB][IP], X[IB][IP], P[IB / 2][IP];
  const int64_t r0 = (int64_t)blockIdx.x * IB;
  const int nb = (int)min64(IB, m - r0);
  const int t = threadIdx.x, w = t >> 5, lane = t & 31;
  {
    // row t / 4, 16 columns: the lower triangle, the identity past m
    const int r = t >> 2, c0 = 16 * (t & 3);
    float4 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      v[q] = r < nb && r0 + c0 + 4 * q < ldl   // (a row's pitch is a multiple of 4)
                 ? *reinterpret_cast<const float4*>(L + (r0 + r) * ldl + r0 + c0 + 4 * q)
                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float e[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + 4 * q + j;
        Ls[r][c] = r < nb ? (c <= r ? e[j] : 0.f) : (r == c ? 1.f : 0.f);
        X[r][c] = 0.f;
      }
    }
  }
  __syncthreads();
  if (w < 4 && lane < 16) {
    const int o = 16 * w;
    float x[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) x[i] = i == lane ? 1.f : 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      x[k] *= 1.0f / Ls[o + k][o + k];
#pragma unroll
      for (int i = k + 1; i < 16; ++i) x[i] = fmaf(-Ls[o + i][o + k], x[k], x[i]);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) X[o + i][o + lane] = x[i];
  }
  __syncthreads();
  {
    // 16 -> 32: block p, output (i, j .. j + 1)
    const int p = t >> 7, i = (t & 127) >> 3, j = 2 * (t & 7), o = 32 * p;
    float s0 = 0.f, s1 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float l = Ls[o + 16 + i][o + k];
      s0 = fmaf(l, X[o + k][o + j], s0);
      s1 = fmaf(l, X[o + k][o + j + 1], s1);
    }
    P[16 * p + i][j] = s0;
    P[16 * p + i][j + 1] = s1;
    __syncthreads();
    s0 = s1 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const float l = X[o + 16 + i][o + 16 + k];
      s0 = fmaf(l, P[16 * p + k][j], s0);
      s1 = fmaf(l, P[16 * p + k][j + 1], s1);
    }
    X[o + 16 + i][o + j] = -s0;
    X[o + 16 + i][o + j + 1] = -s1;
  }
  __syncthreads();
  {
    // 32 -> 64: output (i, j .. j + 3)
    const int i = t >> 3, j = 4 * (t & 7);
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    auto product = [&](const float* row, const float (*B)[IP], int off) {
#pragma unroll
      for (int e = 0; e < 4; ++e) s[e] = 0.f;
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const float4 b = *reinterpret_cast<const float4*>(&B[off + k][j]);
        const float l = row[k];
        s[0] = fmaf(l, b.x, s[0]);
        s[1] = fmaf(l, b.y, s[1]);
        s[2] = fmaf(l, b.z, s[2]);
        s[3] = fmaf(l, b.w, s[3]);
      }
    };
    product(&Ls[32 + i][0], X, 0);
    *reinterpret_cast<float4*>(&P[i][j]) = make_float4(s[0], s[1], s[2], s[3]);
    __syncthreads();
    product(&X[32 + i][32], P, 0);
    *reinterpret_cast<float4*>(&X[32 + i][j]) = make_float4(-s[0], -s[1], -s[2], -s[3]);
  }
  __syncthreads();
  const int64_t lo = r0 % NI;
  float* Wb = W + (r0 / NI) * NI * NI + lo * NI + lo;
  float* WTb = WT + (r0 / NI) * NI * NI + lo * NI + lo;
#pragma unroll
  for (int u = 0; u < IB * IB / IT; ++u) {
    const int e = t + IT * u, i = e / IB, j = e % IB;   // rows and columns past m are zero
    Wb[i * NI + j] = i < nb && j < nb ? X[i][j] : 0.f;
    const float xt = j < nb && i < nb ? X[j][i] : 0.f;  // (row i of the transpose)
    WTb[i * NI + j] = xt;
    if (j > i && j < nb) L[(r0 + i) * ldl + r0 + j] = xt;
  }
}

// Inverses of 256-row blocks, eight columns a CTA kept in shared memory: row
// tile i (64 rows) is X_i = -inv(L_ii) sum_{j < i} L_ij X_j.  Threads 4 r ..
// 4 r + 3 share row r's contraction.  Latency bound, m = 512 13 us, m = 4,096 23; past 256 rows
// the chain of tiles loses to merging (one block of 1,024 rows this way 109
// us, 512 rows 35).
constexpr int SB = 256;      // rows per block
constexpr int CC = 8;        // columns per CTA
// Shared row of entry k of a column: rotated within its line of four, so that
// the four threads of a row (four k apart) read four different bank groups.
__device__ __forceinline__ int xrow(int k) { return (k & ~3) | ((k + (k >> 2)) & 3); }
__global__ void __launch_bounds__(IT) inverse_columns(const float* __restrict__ L, int64_t ldl, int64_t m,
                                                      float* __restrict__ W, float* __restrict__ WT,
                                                      int64_t NI) {
  __shared__ __align__(16) float X[SB][CC], R[IB][CC];
  const int64_t base = (int64_t)blockIdx.y * SB;
  const int nk = (int)min64(SB, m - base), c0 = (int)blockIdx.x * CC;
  // rows and columns of W count from the block of NI rows
  W += base % NI;
  WT += base % NI;
  const int nt = (nk + IB - 1) / IB, i0 = c0 / IB;
  if (i0 >= nt - 1) return;   // the last tile's columns: done by inverse64
  const int t = threadIdx.x, r = t >> 2, q = t & 3;
  for (int e = t; e < IB * CC; e += IT)
    X[xrow(IB * i0 + e / CC)][e % CC] = W[(base + IB * i0 + e / CC) * NI + c0 + e % CC];
  __syncthreads();
  for (int i = i0 + 1; i < nt; ++i) {
    const int64_t row = base + IB * i + r;
    const bool in = row < m;
    const float* Lr = L + row * ldl + base;
    float4 inv[4];   // the row of inv(L_ii) (zeros past m), columns 4 q + 16 s ..
#pragma unroll
    for (int s = 0; s < 4; ++s)
      inv[s] = *reinterpret_cast<const float4*>(W + row * NI + IB * i + 4 * q + 16 * s);
    float acc[CC];
#pragma unroll
    for (int c = 0; c < CC; ++c) acc[c] = 0.f;
    auto add = [&](float (&f)[CC], const float4& a, const float (*B)[CC], int k0) {
      const float e[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float* b = &B[xrow(k0 + k)][0];
        const float4 b0 = *reinterpret_cast<const float4*>(b);
        const float4 b1 = *reinterpret_cast<const float4*>(b + 4);
        f[0] = fmaf(e[k], b0.x, f[0]); f[1] = fmaf(e[k], b0.y, f[1]);
        f[2] = fmaf(e[k], b0.z, f[2]); f[3] = fmaf(e[k], b0.w, f[3]);
        f[4] = fmaf(e[k], b1.x, f[4]); f[5] = fmaf(e[k], b1.y, f[5]);
        f[6] = fmaf(e[k], b1.z, f[6]); f[7] = fmaf(e[k], b1.w, f[7]);
      }
    };
    auto sum4 = [&](float (&f)[CC]) {   // over the row's four threads
#pragma unroll
      for (int c = 0; c < CC; ++c) {
        f[c] += __shfl_xor_sync(0xffffffffu, f[c], 1);
        f[c] += __shfl_xor_sync(0xffffffffu, f[c], 2);
      }
    };
    // 128 entries of the row at a time, the next ones read while these are used
    float4 a[8], n[8];
    auto fetch = [&](float4 (&f)[8], int k) {
#pragma unroll
      for (int u = 0; u < 8; ++u)
        f[u] = in && k + 16 * u < IB * i ? *reinterpret_cast<const float4*>(Lr + k + 16 * u)
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    fetch(a, IB * i0 + 4 * q);
    for (int k = IB * i0 + 4 * q; k < IB * i; k += 128) {
      fetch(n, k + 128);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (k + 16 * u < IB * i) add(acc, a[u], X, k + 16 * u);
#pragma unroll
      for (int u = 0; u < 8; ++u) a[u] = n[u];
    }
    sum4(acc);
    *reinterpret_cast<float2*>(&R[xrow(r)][2 * q]) =
        q == 0 ? make_float2(acc[0], acc[1])
               : (q == 1 ? make_float2(acc[2], acc[3])
                         : (q == 2 ? make_float2(acc[4], acc[5]) : make_float2(acc[6], acc[7])));
    __syncthreads();
    float o[CC];
#pragma unroll
    for (int c = 0; c < CC; ++c) o[c] = 0.f;
#pragma unroll
    for (int s = 0; s < 4; ++s) add(o, inv[s], R, 4 * q + 16 * s);
    sum4(o);
    const float2 x = q == 0 ? make_float2(-o[0], -o[1])
                            : (q == 1 ? make_float2(-o[2], -o[3])
                                      : (q == 2 ? make_float2(-o[4], -o[5]) : make_float2(-o[6], -o[7])));
    *reinterpret_cast<float2*>(&X[xrow(IB * i + r)][2 * q]) = x;
    *reinterpret_cast<float2*>(W + row * NI + c0 + 2 * q) = x;
    __syncthreads();   // (and R is free again)
    const int c = t >> 5, rr = t & 31;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      WT[(base + c0 + c) * NI + IB * i + rr + 32 * u] = X[xrow(IB * i + rr + 32 * u)][c];
  }
}

// Merging pairs of s-row inverses: T = L21 W11, then W21 = -W22 T, 64 x 64
// tiles with the contraction over four groups of threads.  Both products read
// rows along the contraction: T is kept transposed (T^T = W11^T L21^T), and
// W21 goes out both ways.  s = 512, m = 4,096 (256 tiles) 27 and 30 us; few
// tiles (m = 1,024) 19 us each, bound by their own chain.
using MT = simt::Tile<64, 64, 4, 4>;
using MRows = simt::FloatRows<true>;

// grid: (tiles of L21's rows, tiles of W11's columns, pairs)
__global__ void __launch_bounds__(MT::THREADS, 1) merge_first(const float* __restrict__ L, int64_t ldl,
                                                              int64_t m, const float* __restrict__ WT,
                                                              float* __restrict__ T, int64_t NI, int64_t s) {
  extern __shared__ __align__(16) unsigned char dyn[];
  MT::Smem* sm = reinterpret_cast<MT::Smem*>(dyn);
  const int64_t r0 = (int64_t)blockIdx.z * 2 * s, i0 = (int64_t)blockIdx.x * 64, j0 = (int64_t)blockIdx.y * 64;
  if (r0 + s + i0 >= m) return;
  const float* wt = WT + (r0 / NI) * NI * NI + (r0 % NI) * (NI + 1);
  MRows a[MT::LA], b[MT::LB];
#pragma unroll
  for (int u = 0; u < MT::LA; ++u) a[u].p = wt + (j0 + MT::load_row(u)) * NI;
#pragma unroll
  for (int u = 0; u < MT::LB; ++u) {
    const int64_t i = r0 + s + i0 + MT::load_row(u);
    b[u].p = i < m ? L + i * ldl + r0 : nullptr;
  }
  uint64_t acc[MT::RM][4];
  float v[8];
  MT::block_k(sm, a, b, j0, s, acc);   // W11 is lower: its column j starts at row j
  MT::combine(sm, acc, v);
  float* out = T + (int64_t)blockIdx.z * s * s + (j0 + MT::row(MT::group())) * s + i0;
  *reinterpret_cast<float4*>(out + MT::col(0)) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(out + MT::col(4)) = make_float4(v[4], v[5], v[6], v[7]);
}

// grid: (tiles of W11's columns, tiles of W22's rows, pairs)
__global__ void __launch_bounds__(MT::THREADS, 1) merge_second(int64_t m, const float* __restrict__ T,
                                                               float* __restrict__ W, float* __restrict__ WT,
                                                               int64_t NI, int64_t s) {
  extern __shared__ __align__(16) unsigned char dyn[];
  MT::Smem* sm = reinterpret_cast<MT::Smem*>(dyn);
  const int64_t r0 = (int64_t)blockIdx.z * 2 * s, i0 = (int64_t)blockIdx.y * 64, j0 = (int64_t)blockIdx.x * 64;
  if (r0 + s + i0 >= m) return;
  float* w = W + (r0 / NI) * NI * NI + (r0 % NI) * (NI + 1);
  float* wt = WT + (r0 / NI) * NI * NI + (r0 % NI) * (NI + 1);
  MRows a[MT::LA], b[MT::LB];
#pragma unroll
  for (int u = 0; u < MT::LA; ++u) a[u].p = w + (s + i0 + MT::load_row(u)) * NI + s;
#pragma unroll
  for (int u = 0; u < MT::LB; ++u) b[u].p = T + (int64_t)blockIdx.z * s * s + (j0 + MT::load_row(u)) * s;
  uint64_t acc[MT::RM][4];
  float v[8];
  MT::block_k(sm, a, b, 0, i0 + 64, acc);   // W22 is lower
  MT::combine(sm, acc, v);
  const int i = MT::row(MT::group());
  float* out = w + (s + i0 + i) * NI + j0;
  *reinterpret_cast<float4*>(out + MT::col(0)) = make_float4(-v[0], -v[1], -v[2], -v[3]);
  *reinterpret_cast<float4*>(out + MT::col(4)) = make_float4(-v[4], -v[5], -v[6], -v[7]);
  float (*tr)[65] = reinterpret_cast<float (*)[65]>(dyn);   // (combine has left the stages free)
#pragma unroll
  for (int c = 0; c < 8; ++c) tr[MT::col(c)][i] = -v[c];
  __syncthreads();
  for (int e = threadIdx.x; e < 64 * 64; e += MT::THREADS)
    wt[(j0 + e / 64) * NI + s + i0 + e % 64] = tr[e / 64][e % 64];
}

// ---- refinement --------------------------------------------------------------
constexpr int RT = 512;
constexpr int RW = RT / 32;
constexpr int RX = 4096;     // entries of x staged in shared memory

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of the grid (a counter that only grows, zeroed before the launch);
// true when the wait gave up.
__device__ bool refine_barrier(unsigned* count, unsigned& target, int code, const WaitCtx& wc) {
  __shared__ int to_s;
  target += gridDim.x;
  __syncthreads();
  if (threadIdx.x == 0) {
    int to = 0;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
    const uint32_t lim = wait_limit(wc, 1u << 22);
    for (uint32_t it = 0; ld_acquire_u32(count) < target; ++it) {
      if (it >= lim) {
        wait_gave_up(wc, code);
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

// Dot product of a row's elements [c0, c1) (multiples of 4; the row 16-byte
// aligned) with s, over the warp.
__device__ __forceinline__ float row_dot(const float* __restrict__ row, const float* s, int c0, int c1,
                                         int lane) {
  float f[4] = {0.f, 0.f, 0.f, 0.f};
  for (int c = c0 + 4 * lane; c < c1; c += 512) {
    float4 a[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      a[q] = c + 128 * q < c1 ? *reinterpret_cast<const float4*>(row + c + 128 * q)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (c + 128 * q >= c1) break;
      const float4 b = *reinterpret_cast<const float4*>(s + c + 128 * q);
      f[q] = fmaf(a[q].x, b.x, fmaf(a[q].y, b.y, fmaf(a[q].z, b.z, fmaf(a[q].w, b.w, f[q]))));
    }
  }
  return warp_sum((f[0] + f[1]) + (f[2] + f[3]));
}

// Maxima of |a| are taken over the encodings, which order NaN above infinity: a
// vector with a NaN has a NaN for its maximum.
__device__ __forceinline__ unsigned long long bits_of(double a) {
  return (unsigned long long)__double_as_longlong(fabs(a));
}
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long q = __shfl_xor_sync(0xffffffffu, v, o);
    v = q > v ? q : v;
  }
  return v;
}

// One launch for the whole refinement: x = 0, v = (float) b, then steps of z =
// L^{-1} v, (the low-rank correction of z,) x += L^{-T} z, r = b - (H + shift
// I) x in FP64, v = (float) r, until the normwise backward error ||r|| / (||H +
// shift I|| ||x|| + ||b||) is at most tol, or the residual stops halving (from
// the third step: the first two are the FP32 solve and its first correction).
// A triangular solve takes the diagonal blocks in turn: the block's entries by
// its explicit inverse, then its share of the others, rows (forward) or
// columns (backward) over all warps.  Every CTA reduces the CTAs' maxima and
// takes the same decision.  All CTAs are resident (cooperative launch); the
// barriers are bounded.  Bound by the barriers and, from m = 4,096, by the
// FP64 residual (27 us a step at GB300's FP64 rate): three steps take 47 us at m
// = 1,024 and 107 at 4,096, where twelve launches with a chain of 64-row
// blocks took 250 and 930.
__global__ void __launch_bounds__(RT, 1) refine_kernel(RefineArgs a, int64_t NI, int vec, WaitCtx wc) {
  __shared__ __align__(16) float sv[kInvMax];
  __shared__ __align__(16) double sx[RX];
  __shared__ unsigned long long mx[RW][2];
  __shared__ float part[RW][16];
  __shared__ int stop_s;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t m = a.m, G = gridDim.x, cta = blockIdx.x;
  const int64_t B = ceil_div(m, NI);
  const int64_t gw = cta * RW + w, GW = G * RW;     // warp of the grid
  const int64_t rp = ceil_div(m, G), c0 = min64(m, cta * rp), c1 = min64(m, c0 + rp);   // own rows
  unsigned target = 0;
  if (a.finfo && *a.finfo != 0) {   // the factor broke down
    if (cta == 0 && t == 0) a.state->stop = 4;
    return;
  }
  // block maxima of two values into this CTA's slots o, o + 1
  auto put_max = [&](unsigned long long p, unsigned long long q, int o) {
    p = warp_max_bits(p);
    q = warp_max_bits(q);
    if (lane == 0) {
      mx[w][0] = p;
      mx[w][1] = q;
    }
    __syncthreads();
    if (t < 2) {
      unsigned long long v = 0;
      for (int k = 0; k < RW; ++k) v = mx[k][t] > v ? mx[k][t] : v;
      a.red[cta * 4 + o + t] = __longlong_as_double((long long)v);
    }
    __syncthreads();
  };
  // entries [base, base + cnt) of a vector other CTAs wrote, zeros up to the
  // next multiple of 64
  auto stage = [&](const float* src, int64_t base, int cnt) {
    __syncthreads();
    for (int e = t; e < (int)round_up(cnt, 64); e += RT) sv[e] = e < cnt ? __ldcg(src + base + e) : 0.f;
    __syncthreads();
  };
  {
    unsigned long long hm = 0, bm = 0;
    for (int64_t i = c0 + t; i < c1; i += RT) {
      const double bi = a.b[i];
      a.v[i] = f64_to_f32_rn(bi);
      a.x[i] = 0.0;
      const unsigned long long h = bits_of(a.rowsum[i]), bb = bits_of(bi);
      hm = h > hm ? h : hm;
      bm = bb > bm ? bb : bm;
    }
    put_max(hm, bm, 2);
  }
  if (refine_barrier(a.bar, target, 221, wc)) return;
  double be = 0.0, rprev = 0.0;
  int stop = 0, it = 0;
  for (; it < a.max_iter && !stop; ++it) {
    // ---- z = L^{-1} v
    for (int64_t k = 0; k < B; ++k) {
      const int64_t base = k * NI;
      const int nk = (int)min64(NI, m - base);
      stage(a.v, base, nk);
      for (int64_t r = gw; r < nk; r += GW) {
        const float s = row_dot(a.W + (base + r) * NI, sv, 0, (int)(r / 64 + 1) * 64, lane);
        if (lane == 0) __stcg(a.z + base + r, s);
      }
      if (refine_barrier(a.bar, target, 221, wc)) return;
      if (k + 1 == B) break;
      stage(a.z, base, nk);
      for (int64_t i = base + nk + gw; i < m; i += GW) {
        const float s = row_dot(a.L + i * a.ldl + base, sv, 0, nk, lane);
        if (lane == 0) __stcg(a.v + i, __ldcg(a.v + i) - s);
      }
      if (refine_barrier(a.bar, target, 221, wc)) return;
    }
    if (a.V) {   // z -= V C^{-1} (V^T z): partial dots of own rows, then own rows
      for (int c = t; c < a.k; c += RT) {
        float s = 0.f;
        for (int64_t i = c0; i < c1; ++i) s = fmaf(a.V[i * a.ldv + c], __ldcg(a.z + i), s);
        __stcg(a.sp + cta * a.ldv + c, s);
      }
      if (refine_barrier(a.bar, target, 221, wc)) return;
      float* ss = sv;
      float* ws = sv + SPSVM_LOWRANK_KMAX;
      for (int c = t; c < a.k; c += RT) {
        float h = 0.f, l = 0.f;
        for (int64_t q = 0; q < G; ++q) pair_add(h, l, __ldcg(a.sp + q * a.ldv + c));
        ss[c] = __fadd_rn(h, l);
      }
      __syncthreads();
      for (int c = t; c < a.k; c += RT) {
        float s = 0.f;
        for (int e = 0; e < a.k; ++e) s = fmaf(a.Ci[c * a.ldv + e], ss[e], s);
        ws[c] = s;
      }
      __syncthreads();
      for (int64_t i = c0 + w; i < c1; i += RW) {
        float s = 0.f;
        for (int c = lane; c < a.k; c += 32) s = fmaf(a.V[i * a.ldv + c], ws[c], s);
        s = warp_sum(s);
        if (lane == 0) __stcg(a.z + i, __ldcg(a.z + i) - s);
      }
      if (refine_barrier(a.bar, target, 221, wc)) return;
    }
    // ---- x += L^{-T} z
    for (int64_t k = B - 1; k >= 0; --k) {
      const int64_t base = k * NI;
      const int nk = (int)min64(NI, m - base);
      stage(a.z, base, nk);
      for (int64_t r = gw; r < nk; r += GW) {
        const float s = row_dot(a.WT + (base + r) * NI, sv, (int)(r / 64) * 64, (int)round_up(nk, 64), lane);
        if (lane == 0) {
          __stcg(a.xs + base + r, s);
          __stcg(a.x + base + r, __ldcg(a.x + base + r) + (double)s);
        }
      }
      if (refine_barrier(a.bar, target, 222, wc)) return;
      if (k == 0) break;
      stage(a.xs, base, nk);
      // 16 earlier columns at a time: half-warp t / 16 takes every 32nd row
      for (int64_t tile = cta; tile < base / 16; tile += G) {
        const int c = t & 15;
        const float* col = a.L + base * a.ldl + 16 * tile + c;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        for (int r = t >> 4; r < nk; r += 16 * (RT / 16)) {
          float l[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int rq = r + q * (RT / 16);
            l[q] = rq < nk ? col[rq * a.ldl] : 0.f;
          }
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const int rq = r + q * (RT / 16);
            if (rq < nk) s[q & 3] = fmaf(l[q], sv[rq], s[q & 3]);
          }
        }
        float f = (s[0] + s[1]) + (s[2] + s[3]);
        f += __shfl_xor_sync(0xffffffffu, f, 16);
        if (lane < 16) part[w][lane] = f;
        __syncthreads();
        if (t < 16) {
          float z = 0.f;
#pragma unroll
          for (int q = 0; q < RW; ++q) z += part[q][t];
          __stcg(a.z + 16 * tile + t, __ldcg(a.z + 16 * tile + t) - z);
        }
        __syncthreads();
      }
      if (refine_barrier(a.bar, target, 222, wc)) return;
    }
    // ---- r = b - (H + shift I) x, one warp per row
    unsigned long long rm = 0, xm = 0;
    const bool staged = m <= RX;
    if (staged) {
      for (int64_t e = t; e < m; e += RT) sx[e] = __ldcg(a.x + e);
      __syncthreads();
    }
    for (int64_t i = c0 + w; i < c1; i += RW) {
      const double* __restrict__ Hi = a.H + i * a.ldh;
      double s[4] = {0.0, 0.0, 0.0, 0.0};
      if (vec) {
        const double2* __restrict__ H2 = reinterpret_cast<const double2*>(Hi);
        const double2* x2 = staged ? reinterpret_cast<const double2*>(sx) : reinterpret_cast<const double2*>(a.x);
        const int64_t half = m >> 1;
        for (int64_t c = lane; c < half; c += 256) {
          double2 h[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) h[q] = c + 32 * q < half ? H2[c + 32 * q] : make_double2(0.0, 0.0);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if (c + 32 * q >= half) break;
            const double2 xv = staged ? x2[c + 32 * q] : __ldcg(x2 + c + 32 * q);
            s[q & 3] = fma(h[q].y, xv.y, fma(h[q].x, xv.x, s[q & 3]));
          }
        }
        if ((m & 1) && lane == 0) s[0] = fma(Hi[m - 1], __ldcg(a.x + m - 1), s[0]);
      } else {
        for (int64_t c = lane; c < m; c += 128) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (c + 32 * q < m) s[q] = fma(Hi[c + 32 * q], __ldcg(a.x + c + 32 * q), s[q]);
        }
      }
      const double sum = warp_sum((s[0] + s[1]) + (s[2] + s[3]));
      if (lane == 0) {
        const double xi = __ldcg(a.x + i);
        const double ri = a.b[i] - sum - a.shift * xi;
        __stcg(a.v + i, f64_to_f32_rn(ri));
        const unsigned long long rb = bits_of(ri), xb = bits_of(xi);
        rm = rb > rm ? rb : rm;
        xm = xb > xm ? xb : xm;
      }
    }
    put_max(rm, xm, 0);
    if (refine_barrier(a.bar, target, 222, wc)) return;
    // ---- the backward error and the decision, the same in every CTA
    if (w == 0) {
      unsigned long long q[4] = {0ull, 0ull, 0ull, 0ull};
      for (int64_t e = lane; e < G; e += 32)
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const unsigned long long v = (unsigned long long)__double_as_longlong(__ldcg(a.red + 4 * e + p));
          q[p] = v > q[p] ? v : q[p];
        }
#pragma unroll
      for (int p = 0; p < 4; ++p) q[p] = warp_max_bits(q[p]);
      const double rn = __longlong_as_double((long long)q[0]), xn = __longlong_as_double((long long)q[1]);
      const double hn = __longlong_as_double((long long)q[2]), bn = __longlong_as_double((long long)q[3]);
      const double denom = hn * xn + bn;
      be = rn == 0.0 && denom == 0.0 ? 0.0 : rn / denom;
      int s = 0;
      if (!(rn < INFINITY) || !(denom < INFINITY)) s = 3;   // a NaN or an infinity anywhere
      else if (be <= a.tol) s = 1;
      else if (it >= 2 && rn > 0.5 * rprev) s = 2;
      rprev = rn;
      if (lane == 0) stop_s = s;
    }
    __syncthreads();
    stop = stop_s;
  }
  if (cta == 0 && t == 0) {
    a.state->stop = stop;
    a.state->iters = it;
    a.state->be = be;
  }
}

}  // namespace

int launch_block_inverse(float* L, int64_t ldl, int64_t m, float* W, float* WT, float* T, cudaStream_t s) {
  const int64_t NI = inv_size(m);
  inverse64<<<(unsigned)ceil_div(m, (int64_t)IB), IT, 0, s>>>(L, ldl, m, W, WT, NI);
  SPSVM_LAUNCH_CHECK();
  if (m > IB) {
    const dim3 grid((unsigned)(min64(NI, SB) / CC), (unsigned)ceil_div(m, (int64_t)SB));
    inverse_columns<<<grid, IT, 0, s>>>(L, ldl, m, W, WT, NI);
    SPSVM_LAUNCH_CHECK();
  }
  const int smem = (int)(MT::KG * sizeof(MT::Smem));
  for (int64_t h = SB; h < NI && h < m; h *= 2) {
    SPSVM_CUDA_TRY(cudaFuncSetAttribute(merge_first, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    SPSVM_CUDA_TRY(cudaFuncSetAttribute(merge_second, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // pairs whose second half has rows; tiles of rows past m return at once
    const int64_t pairs = ceil_div(m - h, 2 * h);
    const int64_t rows = ceil_div(min64(h, m - h), (int64_t)64);   // of the widest second half
    merge_first<<<dim3((unsigned)rows, (unsigned)(h / 64), (unsigned)pairs), MT::THREADS, smem, s>>>(
        L, ldl, m, WT, T, NI, h);
    SPSVM_LAUNCH_CHECK();
    merge_second<<<dim3((unsigned)(h / 64), (unsigned)rows, (unsigned)pairs), MT::THREADS, smem, s>>>(
        m, T, W, WT, NI, h);
    SPSVM_LAUNCH_CHECK();
  }
  return SPSVM_OK;
}

int launch_refine(const RefineArgs& a0, cudaStream_t s) {
  RefineArgs a = a0;
  int64_t NI = inv_size(a.m);
  WaitCtx wc;
  SPSVM_TRY(wait_ctx(s, &wc));
  const int grid = (int)max64(1, min64(ceil_div(a.m, kRefineRows), (int64_t)sm_count()));
  int vec = a.ldh % 2 == 0 && (reinterpret_cast<uintptr_t>(a.H) & 15) == 0 &&
            (reinterpret_cast<uintptr_t>(a.x) & 15) == 0;
  void* args[] = {&a, &NI, &vec, &wc};
  SPSVM_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)refine_kernel, dim3(grid), dim3(RT), args, 0, s));
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

}  // namespace spsvm
