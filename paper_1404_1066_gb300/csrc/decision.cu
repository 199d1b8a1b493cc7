// Decision values f(q) = sum_j beta_j k(q, b_j) (Section 4: the classifier
// h(x) = w^T phi(x) with w restricted to the basis J), tile by tile, never
// storing the query-by-basis kernel block.  SPSVM_FP32: FP32 SIMT dot
// products, beta_j k(q, b_j) summed as compensated FP32 pairs over a tile of 64
// basis rows and in FP64 over the tiles.  SPSVM_BF16SPLIT: the tensor-core kernel block engine with
// the basis rows and the queries split into three BF16 planes each, FP32 sums
// of beta_j k over 32 basis rows per partial, the partials summed as a
// compensated pair in a fixed order.
#include <cooperative_groups.h>

#include <type_traits>

#include "internal.h"
#include "simt_tile.h"

namespace cg = cooperative_groups;

namespace spsvm {

int64_t decision_tc_parts(int64_t m);
int launch_decision_tc(const spsvm_points* q, const void* zplanes, size_t zbytes, int64_t m,
                       const float* znorm, const double* beta, float gamma, float* dpart,
                       int64_t ldp, cudaStream_t s);

namespace {

// Basis rows by queries.  The wide tile where there are queries enough to fill
// the SMs; else 32 queries, half the rows per thread and the features
// split over four groups of threads: the loop over features is then
// a latency chain of one warp per sub-partition, which the groups shorten, and
// blocks that fit an SM twice let every cluster of a small request start at
// once (with one block per SM not all clusters of 8 found room).
using Wide = simt::Tile<64, 128, 8>;
using Small = simt::Tile<64, 32, 4, 4>;
constexpr int kMaxCluster = 8;

__global__ void row_norms_kernel(const float* __restrict__ A, int64_t m, int64_t d, int64_t lda,
                                 float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= m) return;
  float h = 0.f, l = 0.f;
#pragma unroll 8
  for (int64_t k = lane; k < d; k += 32) pair_add_sq(h, l, A[i * lda + k]);
  const float s = warp_pair_sum(h, l);
  if (lane == 0) out[i] = s;
}

// A query's value has the same bits in every request: each sum below has one
// order, whatever the tile and the cluster.
//   * A dot product is the sum, in order, of those over up to four shares of the
//     features (whole steps of 16, at least two): the small tile's
//     groups take one each, the wide tile keeps the sums so far in shared memory.
//   * beta_j k over a tile of 64 basis rows: four rows at a time in order, the 16
//     sums of four joined by fours (q and q + 8 of two neighbours), these in order.
//   * A query's tiles fall in kLanes lanes, tile t in lane t % kLanes; a lane's
//     tiles are added in order, then the lanes.  A cluster's blocks take whole
//     lanes, and rank 0 adds them through distributed shared memory.
constexpr int kLanes = kMaxCluster;
// (32 features at least: of 64, one query by 4,096 rows, d = 128 took 80 us
// instead of 69; of 16, 100,000 queries by 512 rows, d = 64 368 instead of 346)
__host__ __device__ inline int64_t feature_share(int64_t d) {
  return max64(2, ceil_div(ceil_div(d, (int64_t)16), (int64_t)4)) * 16;
}

// Sums of beta_j k.  In pairs (beta_j in two FP32 terms: an FP64 multiply-add and
// conversion per kernel value, at 1/64 of the FP32 rate, cost more than the dot
// products at small d), or in FP64 for the tiles with a beta_j outside the range
// where the pairs keep 2^-46 of it.
struct PairSum {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float bh, float bl, double, float k) {
    const float x = __fmul_rn(bh, k);
    l = __fadd_rn(l, __fmaf_rn(bl, k, __fmaf_rn(bh, k, -x)));
    pair_add(h, l, x);
  }
  __device__ __forceinline__ void join(PairSum o) {   // a.join(b) == b.join(a)
    l = __fadd_rn(l, o.l);
    pair_add(h, l, o.h);
  }
  __device__ __forceinline__ PairSum shfl_xor(int x) const {
    PairSum o;
    o.h = __shfl_xor_sync(0xffffffffu, h, x);
    o.l = __shfl_xor_sync(0xffffffffu, l, x);
    return o;
  }
  __device__ __forceinline__ double value() const { return pair_value(h, l); }
};
struct WideSum {
  double s = 0.0;
  __device__ __forceinline__ void add(float, float, double b, float k) { s += b * (double)k; }
  __device__ __forceinline__ void join(WideSum o) { s += o.s; }
  __device__ __forceinline__ WideSum shfl_xor(int x) const {
    WideSum o;
    o.s = __shfl_xor_sync(0xffffffffu, s, x);
    return o;
  }
  __device__ __forceinline__ double value() const { return s; }
};
__device__ __forceinline__ bool beyond_pairs(double b) {
  const double a = fabs(b);
  return b != 0.0 && !(a >= 0x1p-80 && a <= 0x1p90);
}

// FP32 ALU bound for many queries, latency of the feature loop for few: 1,000
// queries, 512 basis rows, d = 784 0.037 ms, where 8 blocks of 128 queries took
// 0.66 ms.  The one order costs the wide tile 3 to 9%: 30,000 queries by 4,096
// rows, d = 128 1.11 ms, 1.02 with sums in whatever order a block meets them.
template <class T, bool VB, bool VQ>
__global__ void __launch_bounds__(T::THREADS, T::KG == 1 ? 3 : 2) decision_simt(
    const float* __restrict__ B, int64_t m, int64_t ldb, const float* __restrict__ bnorm,
    const double* __restrict__ beta, const float* __restrict__ Q, int64_t nq, int64_t ldq,
    int64_t d, float gamma, float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char dyn[];
  typename T::Smem* sm = reinterpret_cast<typename T::Smem*>(dyn);
  constexpr int W = T::THREADS / 32;
  constexpr int RED = T::KG == 1 ? 4 : 16;   // partial sums of a tile per query
  __shared__ float qn[T::TN], bn[T::TM], bh[T::TM], bl[T::TM];
  __shared__ double bd[T::TM];
  // [lane][query]: PairSum, or (widel[lane]) WideSum
  __shared__ __align__(8) unsigned char totals[kLanes * T::TN * 8];
  __shared__ int widel[kLanes], widet[2];   // widet: per warp that loads a tile's coefficients
  static_assert(T::TM == 64 && T::TY * T::RM == 64 && T::THREADS >= T::TN, "64 rows a tile, a thread per query");
  static_assert(sizeof(typename T::Smem) >= sizeof(double) * RED * T::TN, "partial sums fit the stages");
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t q0 = (int64_t)(blockIdx.x / cs) * T::TN;
  cl.sync();   // every block of the cluster is resident before its shared memory is written
  // query norms: the rows split over the cluster's warps, each written to every block
  for (int r = rank * W + w; r < T::TN; r += cs * W) {
    float h = 0.f, l = 0.f;
    if (q0 + r < nq) {
#pragma unroll 8
      for (int64_t k = lane; k < d; k += 32) pair_add_sq(h, l, Q[(q0 + r) * ldq + k]);
    }
    const float s = warp_pair_sum(h, l);
    if (lane < cs) *cl.map_shared_rank(&qn[r], lane) = s;
  }
  cl.sync();
  simt::FloatRows<VB> a[T::LA];
  simt::FloatRows<VQ> b[T::LB];
#pragma unroll
  for (int u = 0; u < T::LB; ++u) {
    const int64_t q = q0 + T::load_row(u);
    b[u].p = q < nq ? Q + q * ldq : nullptr;
  }
  const int64_t share = feature_share(d), tiles = ceil_div(m, (int64_t)T::TM);
  // sum += the sum over the tile at b0 of query q0 + t (threads below TN), from
  // the dot products of this thread's rows and columns
  auto add_tile = [&](auto& sum, int64_t b0, auto dots) {
    using S = std::remove_reference_t<decltype(sum)>;
    S* red = reinterpret_cast<S*>(dyn);   // [RED][TN]
    // four rows from T::row(r0) on, all columns at once (independent chains)
    auto four = [&](int r0, auto& v, auto col) {
#pragma unroll
      for (int r = r0; r < r0 + 4; ++r) {
        const int j = T::row(r);
        if (b0 + j >= m) continue;
        const float zn = bn[j], jh = bh[j], jl = bl[j];
        const double jd = std::is_same<S, WideSum>::value ? bd[j] : 0.0;
#pragma unroll
        for (int c = 0; c < (int)(sizeof(v) / sizeof(S)); ++c)
          v[c].add(jh, jl, jd, rbf_from_dot(qn[col(c)], zn, dots(r, c), gamma));
      }
    };
    if constexpr (T::KG == 1) {
      auto col = [](int c) { return T::col(c); };
      S s[8], u[8];
      four(0, s, col);
      four(4, u, col);
#pragma unroll
      for (int c = 0; c < 8; ++c) s[c].join(u[c]);
#pragma unroll
      for (int c = 0; c < 8; ++c) s[c].join(s[c].shfl_xor(T::TX));   // the neighbour's
      if (lane < T::TX)
#pragma unroll
        for (int c = 0; c < 8; ++c) red[w * T::TN + T::col(c)] = s[c];
    } else {
      auto col = [](int e) { return 4 * T::tx() + ((2 * T::group() + e) & 3) + (T::group() >> 1) * (T::TN / 2); };
      S s[2];
      four(0, s, col);
#pragma unroll
      for (int e = 0; e < 2; ++e) red[T::ty() * T::TN + col(e)] = s[e];
    }
    __syncthreads();
    if (t < T::TN) {
      S s;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if constexpr (T::KG == 1) {
          s.join(red[p * T::TN + t]);
        } else {
          S x = red[2 * p * T::TN + t], y = red[(2 * p + 1) * T::TN + t];
          x.join(red[(2 * p + 8) * T::TN + t]);
          y.join(red[(2 * p + 9) * T::TN + t]);
          x.join(y);
          s.join(x);
        }
      }
      sum.join(s);
    }
  };
  for (int ln = rank; ln < kLanes; ln += cs) {
    PairSum sum;        // of query q0 + t over the lane's tiles
    WideSum wide;       // and over those with a beta_j beyond the pairs
    bool any = false;   // there was one
    for (int64_t tile = ln; tile < tiles; tile += kLanes) {
      const int64_t b0 = tile * T::TM;
      __syncthreads();   // the last tile's norms, coefficients and sums have been read
      if (t < T::TM) {
        const int64_t j = b0 + t;
        const double bj = j < m ? beta[j] : 0.0;
        bn[t] = j < m ? bnorm[j] : 0.f;
        bd[t] = bj;
        bh[t] = (float)bj;
        bl[t] = (float)(bj - (double)bh[t]);
        const bool beyond = __any_sync(0xffffffffu, beyond_pairs(bj));
        if (lane == 0) widet[w] = beyond;
      }
#pragma unroll
      for (int u = 0; u < T::LA; ++u) {
        const int64_t j = b0 + T::load_row(u);
        a[u].p = j < m ? B + j * ldb : nullptr;
      }
      uint64_t acc[T::RM][4];
      if constexpr (T::KG > 1) {
        T::block_k(sm, a, b, 0, d, share, acc);
        uint64_t v[4];
        T::combine_cols(sm, acc, v);
        auto dots = [&](int r, int e) {
          const float2 x = simt::unpack2(v[r]);
          return e ? x.y : x.x;
        };
        if (widet[0] | widet[1]) {
          add_tile(wide, b0, dots);
          any = true;
        } else {
          add_tile(sum, b0, dots);
        }
      } else {
        // the sums of a whole share are added to those kept
        ulonglong2* keep = reinterpret_cast<ulonglong2*>(dyn + sizeof(typename T::Smem)) + t;
        const int steps = (int)(share / T::TK);
        int left = steps;
        bool kept = false;
        auto add_kept = [&](uint64_t (&f)[T::RM][4]) {
#pragma unroll
          for (int i = 0; i < T::RM * 2; ++i) {
            const ulonglong2 o = keep[i * T::THREADS];
            f[i / 2][2 * (i & 1)] = simt::add2(o.x, f[i / 2][2 * (i & 1)]);
            f[i / 2][2 * (i & 1) + 1] = simt::add2(o.y, f[i / 2][2 * (i & 1) + 1]);
          }
        };
        T::product(*sm, a, b, 0, d, acc, [&](uint64_t (&f)[T::RM][4]) {
          if (--left > 0) return;
          left = steps;
          if (kept) add_kept(f);
          kept = true;
#pragma unroll
          for (int i = 0; i < T::RM * 2; ++i) {
            keep[i * T::THREADS] = make_ulonglong2(f[i / 2][2 * (i & 1)], f[i / 2][2 * (i & 1) + 1]);
            f[i / 2][2 * (i & 1)] = f[i / 2][2 * (i & 1) + 1] = 0ull;
          }
        });
        if (kept) add_kept(acc);
        auto dots = [&](int r, int c) {
          const float2 x = simt::unpack2(acc[r][c / 2]);
          return c & 1 ? x.y : x.x;
        };
        if (widet[0] | widet[1]) {
          add_tile(wide, b0, dots);
          any = true;
        } else {
          add_tile(sum, b0, dots);
        }
      }
    }
    if (t < T::TN) {
      if (any) wide.s += sum.value();
      if (any) reinterpret_cast<WideSum*>(totals)[ln * T::TN + t] = wide;
      else reinterpret_cast<PairSum*>(totals)[ln * T::TN + t] = sum;
      if (t == 0) widel[ln] = any;
    }
  }
  cl.sync();
  if (rank == 0 && t < T::TN && q0 + t < nq) {
    PairSum p;
    WideSum v;
#pragma unroll
    for (int ln = 0; ln < kLanes; ++ln) {
      const int r = ln % cs;
      if (*cl.map_shared_rank(&widel[ln], r))
        v.join(cl.map_shared_rank(reinterpret_cast<WideSum*>(totals), r)[ln * T::TN + t]);
      else
        p.join(cl.map_shared_rank(reinterpret_cast<PairSum*>(totals), r)[ln * T::TN + t]);
    }
    out[q0 + t] = (float)(p.value() + v.s);
  }
  cl.sync();   // no block leaves while rank 0 reads its sums
}

template <class T>
int launch_decision_simt(int cs, const float* B, int64_t m, int64_t ldb, const float* bnorm,
                         const double* beta, const float* Q, int64_t nq, int64_t ldq, int64_t d,
                         float gamma, float* out, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(ceil_div(nq, T::TN) * cs));
  cfg.blockDim = dim3(T::THREADS);
  cfg.dynamicSmemBytes = T::KG * sizeof(typename T::Smem);
  if (T::KG == 1 && d > feature_share(d)) cfg.dynamicSmemBytes += sizeof(float) * T::TM * T::TN;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const bool vb = simt::rows_aligned(B, ldb), vq = simt::rows_aligned(Q, ldq);
  auto kern = vb ? (vq ? decision_simt<T, true, true> : decision_simt<T, true, false>)
                 : (vq ? decision_simt<T, false, true> : decision_simt<T, false, false>);
  SPSVM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)cfg.dynamicSmemBytes));
  SPSVM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, B, m, ldb, bnorm, beta, Q, nq, ldq, d, gamma, out));
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

// out[i] = sum over the P partials of column i as compensated pairs: each of
// 8 groups of threads sums every 8th partial of 32 columns, the groups are
// added in order.  L2 bound: 32,768 columns of 128 partials
// 9 us; one thread a column in FP64 took 24.
constexpr int DF_G = 8;
__global__ void __launch_bounds__(32 * DF_G) decision_finish(const float* __restrict__ part, int64_t P,
                                                             int64_t ldp, int64_t nq,
                                                             float* __restrict__ out) {
  __shared__ float2 sh[DF_G][32];
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int64_t i = (int64_t)blockIdx.x * 32 + c;
  float h = 0.f, l = 0.f;
  if (i < nq) {
    for (int64_t p = g; p < P; p += 8 * DF_G) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p + u * DF_G < P ? part[(p + u * DF_G) * ldp + i] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) pair_add(h, l, v[u]);
    }
  }
  sh[g][c] = make_float2(h, l);
  __syncthreads();
  if (g != 0 || i >= nq) return;
#pragma unroll
  for (int u = 1; u < DF_G; ++u) {
    l = __fadd_rn(l, sh[u][c].y);
    pair_add(h, l, sh[u][c].x);
  }
  out[i] = (float)pair_value(h, l);
}

// Queries per pass of the tensor-core form (bounds the scratch).
constexpr int64_t kDecideChunk = 32768;

struct DecideLayout {
  int64_t ldh, qc, parts;
  size_t off_zn, off_z, z_bytes, off_qn, off_q, q_plane, off_part, total;
};

DecideLayout decide_layout(int64_t nq, int64_t m, int64_t d) {
  DecideLayout L;
  auto al = [](size_t b) { return (size_t)round_up((int64_t)b, 256); };
  L.ldh = round_up(d, 64);
  L.qc = round_up(min64(max64(nq, 1), kDecideChunk), 128);
  L.parts = decision_tc_parts(m);
  size_t o = 0;
  L.off_zn = o;
  o += al((size_t)m * 4);
  L.off_z = o;
  L.z_bytes = (size_t)m * L.ldh * 6;
  o += al(L.z_bytes);
  L.off_qn = o;
  o += al((size_t)L.qc * 4);
  L.off_q = o;
  L.q_plane = (size_t)L.qc * L.ldh * 2;
  o += al(3 * L.q_plane);
  L.off_part = o;
  o += al((size_t)L.parts * L.qc * 4);
  L.total = o;
  return L;
}

}  // namespace
}  // namespace spsvm

using namespace spsvm;

extern "C" size_t spsvm_decision_scratch_bytes(int64_t nq, int64_t m, int64_t d, int32_t precision) {
  if (m < 0 || d < 1) return 0;
  if (precision == SPSVM_BF16SPLIT) return decide_layout(nq, m, d).total;
  return (size_t)round_up(m * 4 + 16, 256);
}

extern "C" int spsvm_decision(const float* B, int64_t m, int64_t ldb, const double* beta,
                              const float* Q, int64_t nq, int64_t ldq, int64_t d, float gamma,
                              int32_t precision, float* out, void* scratch, size_t scratch_bytes,
                              void* stream) {
  if (!B || !beta || !Q || !out || m < 0 || nq < 0 || d < 1 || ldb < d || ldq < d || !(gamma > 0.f))
    return set_error(SPSVM_ERR_ARG, "decision: bad arguments");
  if (precision != SPSVM_FP32 && precision != SPSVM_BF16SPLIT)
    return set_error(SPSVM_ERR_ARG, "decision: bad precision");
  if (nq == 0) return SPSVM_OK;
  if (!scratch || scratch_bytes < spsvm_decision_scratch_bytes(nq, m, d, precision))
    return set_error(SPSVM_ERR_OOM, "decision: scratch too small");
  cudaStream_t s = as_stream(stream);
  if (precision == SPSVM_BF16SPLIT) {
    // algorithmic work: 2 nq m d multiply-adds, times the six plane products
    ProfScope prof(PROF_DECISION, s, 12.0 * (double)nq * m * (double)d);
    if (m == 0) {
      SPSVM_CUDA_TRY(cudaMemsetAsync(out, 0, (size_t)nq * 4, s));
      return SPSVM_OK;
    }
    const DecideLayout L = decide_layout(nq, m, d);
    char* w = static_cast<char*>(scratch);
    // the basis rows' norms and planes (rows past m read as zeros)
    uint16_t* zp = reinterpret_cast<uint16_t*>(w + L.off_z);
    spsvm_points zb{B, m, d, ldb, reinterpret_cast<float*>(w + L.off_zn), zp, zp + 2 * m * L.ldh,
                    L.ldh, zp + m * L.ldh};
    SPSVM_TRY(spsvm_prepare_points(&zb, SPSVM_BF16SPLIT, stream));
    uint16_t* qp = reinterpret_cast<uint16_t*>(w + L.off_q);
    float* part = reinterpret_cast<float*>(w + L.off_part);
    for (int64_t q0 = 0; q0 < nq; q0 += L.qc) {
      const int64_t cnt = min64(L.qc, nq - q0);
      spsvm_points qb{Q + q0 * ldq, cnt, d, ldq, reinterpret_cast<float*>(w + L.off_qn), qp,
                      qp + 2 * L.qc * L.ldh, L.ldh, qp + L.qc * L.ldh};
      SPSVM_TRY(spsvm_prepare_points(&qb, SPSVM_BF16SPLIT, stream));
      SPSVM_TRY(launch_decision_tc(&qb, zp, L.z_bytes, m, zb.norms, beta, gamma, part, L.qc, s));
      decision_finish<<<(unsigned)ceil_div(cnt, (int64_t)32), 32 * DF_G, 0, s>>>(part, L.parts, L.qc,
                                                                                cnt, out + q0);
      SPSVM_LAUNCH_CHECK();
    }
    return SPSVM_OK;
  }
  ProfScope prof(PROF_DECISION, s, 2.0 * (double)nq * m * (double)d);
  float* bnorm = static_cast<float*>(scratch);
  if (m > 0) {
    row_norms_kernel<<<(unsigned)ceil_div(m, 8), 256, 0, s>>>(B, m, d, ldb, bnorm);
    SPSVM_LAUNCH_CHECK();
  }
  // up to three blocks per SM: first more blocks per query tile (basis rows
  // split over a cluster); the small tile where that still leaves SMs with one
  // block or none (512 rows, d = 784: 2,000 queries 70 us against 93; 4,000
  // queries 120 against 96)
  const int64_t want = 3 * (int64_t)sm_count(), tiles = ceil_div(nq, (int64_t)Wide::TN);
  const int64_t basis_tiles = ceil_div(m, (int64_t)Wide::TM);
  auto cluster = [&](int64_t query_tiles) {
    int cs = 1;
    while (2 * cs <= kMaxCluster && 2 * cs <= basis_tiles && query_tiles * cs < want) cs *= 2;
    return cs;
  };
  const int cs = cluster(tiles);
  if (4 * tiles * cs >= 5 * (int64_t)sm_count())
    return launch_decision_simt<Wide>(cs, B, m, ldb, bnorm, beta, Q, nq, ldq, d, gamma, out, s);
  return launch_decision_simt<Small>(cluster(ceil_div(nq, (int64_t)Small::TN)), B, m, ldb, bnorm, beta,
                                     Q, nq, ldq, d, gamma, out, s);
}
