// FP32 tile product shared by the SPSVM_FP32 kernels: D[a][b] = sum_k A[a][k]
// B[b][k] over rows stored with k contiguous, one multiply-add per term in
// the order of k.
#pragma once
#include "internal.h"

namespace spsvm {
namespace simt {

// acc += a * b on two FP32 lanes (each an IEEE fused multiply-add): the
// packed instruction takes one issue slot for two multiply-adds, which leaves
// the other slots to the shared-memory loads.
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ uint64_t dup2(float a) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Four consecutive elements k .. k + 3 of a row (zeros at and past d, and for
// a null row).  VEC: every row starts 16-byte aligned.
template <bool VEC>
__device__ __forceinline__ float4 row4(const float* __restrict__ row, int64_t k, int64_t d) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!row) return v;
  if (VEC && k + 4 <= d) return *reinterpret_cast<const float4*>(row + k);
  if (k < d) v.x = row[k];
  if (k + 1 < d) v.y = row[k + 1];
  if (k + 2 < d) v.z = row[k + 2];
  if (k + 3 < d) v.w = row[k + 3];
  return v;
}
// Rows read through a float pointer, or as BF16 hi / lo planes.
template <bool VEC>
struct FloatRows {
  const float* p;
  __device__ __forceinline__ bool null() const { return !p; }
  __device__ __forceinline__ float4 load(int64_t k, int64_t d) const { return row4<VEC>(p, k, d); }
};
struct PlaneRows {
  const __nv_bfloat16* hi;
  int64_t plane;
  __device__ __forceinline__ float4 load(int64_t k, int64_t d) const {
    float v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      v[e] = hi && k + e < d ? __bfloat162float(hi[k + e]) + __bfloat162float(hi[plane + k + e]) : 0.f;
    return make_float4(v[0], v[1], v[2], v[3]);
  }
};

// TM x TN outputs by (TM / RM) x (TN / 8) threads, each RM x 8 of them in two
// (RM 8) or one groups of 4 rows and two groups of 4 columns, 16 k per stage
// in two shared-memory stages.  An element (row, k) is staged k-major at
// column row ^ 8 (k / 4 % 4), so both the transposing stores and the 16-byte
// reads are free of bank conflicts.  RM 8: 32 packed multiply-adds (64 issue
// cycles of a sub-partition) per 4 16-byte shared loads and 8 duplications.
// KG: groups of threads in a block that each run the product over their share
// of k on stages of their own (block_k, combine).
template <int TM_, int TN_, int RM_, int KG_ = 1>
struct Tile {
  static constexpr int TM = TM_, TN = TN_, RM = RM_, KG = KG_, RN = 8, TK = 16;
  static constexpr int TX = TN / RN, TY = TM / RM, NT = TX * TY, THREADS = NT * KG;
  static constexpr int LA = TM * TK / 4 / NT, LB = TN * TK / 4 / NT;   // 16-byte loads a thread
  static_assert(LA * NT * 4 == TM * TK && LB * NT * 4 == TN * TK, "tile loads");
  static_assert(TM % 32 == 0 && TN % 32 == 0 && (RM == 4 || RM == 8), "tile shape");
  struct Smem {
    alignas(16) float A[2][TK][TM];
    alignas(16) float B[2][TK][TN];
  };
  // Thread within its group, and the group.
  static __device__ __forceinline__ int tid() { return KG == 1 ? (int)threadIdx.x : (int)threadIdx.x % NT; }
  static __device__ __forceinline__ int group() { return KG == 1 ? 0 : (int)threadIdx.x / NT; }
  static __device__ __forceinline__ void sync() {
    if (KG == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + group()), "n"(NT) : "memory");
  }
  // Row of the thread's u-th staged element (its k is 4 (t % 4)).
  static __device__ __forceinline__ int load_row(int u) { return (tid() + NT * u) >> 2; }
  static __device__ __forceinline__ int tx() { return tid() % TX; }
  static __device__ __forceinline__ int ty() { return tid() / TX; }
  // Tile row / column of accumulator r / c of a thread.
  static __device__ __forceinline__ int row(int r) { return 4 * ty() + (r & 3) + (r >> 2) * (TM / 2); }
  static __device__ __forceinline__ int col(int c) { return 4 * tx() + (c & 3) + (c >> 2) * (TN / 2); }

  template <int L, int W>
  static __device__ __forceinline__ void stage(float (*S)[W], const float4 (&v)[L]) {
    const int k4 = tid() & 3;
#pragma unroll
    for (int u = 0; u < L; ++u) {
      const int col = load_row(u) ^ (8 * k4);
      S[4 * k4 + 0][col] = v[u].x;
      S[4 * k4 + 1][col] = v[u].y;
      S[4 * k4 + 2][col] = v[u].z;
      S[4 * k4 + 3][col] = v[u].w;
    }
  }

  // acc[r][c / 2] (packed pairs of columns) = the sums over k in [k0, k1) of
  // rows a[], b[] (this thread's staged rows).  All threads; starts with the
  // stages free and ends with a barrier.  step(acc) runs after every TK terms
  // but the last ones, and may move the sums so far elsewhere.
  struct NoStep {
    __device__ __forceinline__ void operator()(uint64_t (&)[RM][RN / 2]) const {}
  };
  template <class RA, class RB, class Step = NoStep>
  static __device__ __forceinline__ void product(Smem& sm, const RA (&a)[LA], const RB (&b)[LB],
                                                 int64_t k0, int64_t k1, uint64_t (&acc)[RM][RN / 2],
                                                 Step step = Step()) {
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int c = 0; c < RN / 2; ++c) acc[r][c] = 0ull;
    const int x4 = 4 * tx(), y4 = 4 * ty();
    const int kq = 4 * (tid() & 3);
    float4 va[LA], vb[LB];
    auto fetch = [&](int64_t k) {
#pragma unroll
      for (int u = 0; u < LA; ++u) va[u] = a[u].load(k + kq, k1);
#pragma unroll
      for (int u = 0; u < LB; ++u) vb[u] = b[u].load(k + kq, k1);
    };
    // one chunk: the next one is fetched while stage s is used, then staged
    auto chunk = [&](int64_t k, int s) {
      const bool more = k + TK < k1;
      if (more) fetch(k + TK);
#pragma unroll
      for (int kk = 0; kk < TK; ++kk) {
        const int sw = 8 * (kk >> 2);
        float av[RM];
        uint64_t bv[RN / 2];
#pragma unroll
        for (int h = 0; h < RM / 4; ++h) {
          const float4 f = *reinterpret_cast<const float4*>(&sm.A[s][kk][(h * (TM / 2) + y4) ^ sw]);
          av[4 * h] = f.x; av[4 * h + 1] = f.y; av[4 * h + 2] = f.z; av[4 * h + 3] = f.w;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const ulonglong2 f = *reinterpret_cast<const ulonglong2*>(&sm.B[s][kk][(h * (TN / 2) + x4) ^ sw]);
          bv[2 * h] = f.x; bv[2 * h + 1] = f.y;
        }
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          const uint64_t ar = dup2(av[r]);
#pragma unroll
          for (int c = 0; c < RN / 2; ++c) fma2(acc[r][c], ar, bv[c]);
        }
      }
      if (more) {
        stage<LA, TM>(sm.A[s ^ 1], va);
        stage<LB, TN>(sm.B[s ^ 1], vb);
        step(acc);
      }
      sync();
    };
    fetch(k0);
    stage<LA, TM>(sm.A[0], va);
    stage<LB, TN>(sm.B[0], vb);
    sync();
    for (int64_t k = k0; k < k1; k += 2 * TK) {
      chunk(k, 0);
      if (k + TK < k1) chunk(k + TK, 1);
    }
  }

  // product over [k0, k1) by the whole block: group g takes the g-th share
  // (share, a multiple of TK, or the chunks evenly).  combine then leaves
  // thread (group g, t) with the 8 sums of row r = g of thread t's outputs,
  // added over the groups in order (KG == RM; sm: the groups' stages);
  // combine_cols with all rows of its columns 2 g, 2 g + 1 (KG == RN / 2).
  // All threads; both end with a barrier.
  template <class RA, class RB>
  static __device__ __forceinline__ void block_k(Smem* sm, const RA (&a)[LA], const RB (&b)[LB],
                                                 int64_t k0, int64_t k1, uint64_t (&acc)[RM][RN / 2]) {
    block_k(sm, a, b, k0, k1, ceil_div(ceil_div(k1 - k0, (int64_t)TK), (int64_t)KG) * TK, acc);
  }
  template <class RA, class RB>
  static __device__ __forceinline__ void block_k(Smem* sm, const RA (&a)[LA], const RB (&b)[LB],
                                                 int64_t k0, int64_t k1, int64_t share,
                                                 uint64_t (&acc)[RM][RN / 2]) {
    const int64_t g0 = min64(k1, k0 + group() * share);
    product(sm[group()], a, b, g0, min64(k1, g0 + share), acc);
  }
  static __device__ __forceinline__ void combine(Smem* sm, const uint64_t (&acc)[RM][RN / 2], float (&v)[RN]) {
    static_assert(KG == RM && sizeof(Smem) >= sizeof(float) * RM * NT * RN, "one row per group");
    ulonglong2* mine = reinterpret_cast<ulonglong2*>(&sm[group()]);
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        mine[(r * 2 + h) * NT + tid()] = make_ulonglong2(acc[r][2 * h], acc[r][2 * h + 1]);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < RN; ++c) v[c] = 0.f;
#pragma unroll
    for (int g = 0; g < KG; ++g) {
      const float4* p = reinterpret_cast<const float4*>(&sm[g]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 f = p[(group() * 2 + h) * NT + tid()];
        v[4 * h] += f.x; v[4 * h + 1] += f.y; v[4 * h + 2] += f.z; v[4 * h + 3] += f.w;
      }
    }
    __syncthreads();
  }
  static __device__ __forceinline__ void combine_cols(Smem* sm, const uint64_t (&acc)[RM][RN / 2],
                                                      uint64_t (&v)[RM]) {
    static_assert(KG == RN / 2 && sizeof(Smem) >= sizeof(float) * RM * NT * RN, "a pair of columns per group");
    uint64_t* mine = reinterpret_cast<uint64_t*>(&sm[group()]);
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int p = 0; p < RN / 2; ++p) mine[(r * (RN / 2) + p) * NT + tid()] = acc[r][p];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      v[r] = reinterpret_cast<const uint64_t*>(&sm[0])[(r * (RN / 2) + group()) * NT + tid()];
#pragma unroll
      for (int g = 1; g < KG; ++g)
        v[r] = add2(v[r], reinterpret_cast<const uint64_t*>(&sm[g])[(r * (RN / 2) + group()) * NT + tid()]);
    }
    __syncthreads();
  }
};

// Whether rows of pitch ld from base can be read 16 bytes at a time.
inline bool rows_aligned(const float* base, int64_t ld) {
  return (ld % 4) == 0 && (reinterpret_cast<uintptr_t>(base) & 15) == 0;
}

}  // namespace simt
}  // namespace spsvm
