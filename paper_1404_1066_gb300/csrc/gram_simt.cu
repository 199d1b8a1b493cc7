// Masked Gram matrix H = lambda K_JJ + K_SJ^T K_SJ (the generalised Hessian
// of Eq. 4 on the active set S) in FP32 SIMT arithmetic, with FP32 sums per
// 2,048 points added up as compensated pairs.  Also the FP64 finishing pass
// shared by both arithmetic forms.
#include "internal.h"
#include "gram.h"
#include "simt_tile.h"

namespace spsvm {

namespace {

constexpr int64_t kChunk = 2048;     // points per FP32 sum
// Up to this many rows the small tile (m = 512, ns = 20,000: 175 us against 214;
// m = 700: 318 against 304).
constexpr int64_t kSmallBasis = 512;

// Rows a by columns b of the upper triangle.  The wide tile, and for small
// matrices, whose blocks leave the chain over their points exposed, one with
// the points split over four groups of threads.
using Wide = simt::Tile<64, 128, 8>;
using Small = simt::Tile<64, 64, 4, 4>;

__device__ __forceinline__ void set_row(simt::FloatRows<true>& r, const KView& K, int64_t j, int64_t m) {
  r.p = j < m ? static_cast<const float*>(K.data) + j * K.ld : nullptr;
}
__device__ __forceinline__ void set_row(simt::PlaneRows& r, const KView& K, int64_t j, int64_t m) {
  r.hi = j < m ? static_cast<const __nv_bfloat16*>(K.data) + j * K.ld : nullptr;
  r.plane = K.plane;
}

// Column tiles of row tile ta start at the one that holds its diagonal.
template <class T>
__host__ __device__ __forceinline__ int64_t first_col(int64_t ta) { return ta * T::TM / T::TN; }
template <class T>
int64_t upper_tiles(int64_t m) {   // tiles (ta, tb) with tb >= first_col(ta)
  const int64_t A = ceil_div(m, (int64_t)T::TM), B = ceil_div(m, (int64_t)T::TN);
  constexpr int64_t R = T::TN / T::TM;   // row tiles per column tile
  const int64_t f = A / R, g = A % R;    // sum over ta of ta / R
  return A * B - (R * (f * (f - 1) / 2) + g * f);
}

// part[split][a][b] = the split's points' products, for tiles of the upper
// triangle.  The active points are split evenly over the blocks (their number
// is read on the device), FP32 sums per 2,048 points.  FP32 ALU bound:
// ns = 18,000, m = 1,024 0.43 ms (44 TFLOP/s); 64 x 64 tiles of 4 x 4 outputs
// with scalar shared loads over three slices took 1.77 ms.
template <class T, class Rows>
__global__ void __launch_bounds__(T::THREADS, T::KG == 1 ? 3 : 1) gram_simt_kernel(
    KView Kc, int64_t m, const int64_t* __restrict__ ns_dev, int64_t splits,
    float2* __restrict__ part, int64_t ldp) {
  extern __shared__ __align__(16) unsigned char dyn[];
  typename T::Smem* sm = reinterpret_cast<typename T::Smem*>(dyn);
  const int64_t ns = *ns_dev;
  const int64_t per = gram_split_points(ns, splits, kGramQuantumSimt);
  const int64_t p_begin = (int64_t)blockIdx.y * per;
  if (blockIdx.y > 0 && p_begin >= ns) return;   // the finish skips the empty splits
  const int64_t p_end = min64(ns, p_begin + per);
  const int64_t nB = ceil_div(m, (int64_t)T::TN);
  int64_t ta = 0, rem = blockIdx.x;
  while (rem >= nB - first_col<T>(ta)) {
    rem -= nB - first_col<T>(ta);
    ++ta;
  }
  const int64_t a0 = ta * T::TM, b0 = (first_col<T>(ta) + rem) * T::TN;
  Rows a[T::LA], b[T::LB];
#pragma unroll
  for (int u = 0; u < T::LA; ++u) set_row(a[u], Kc, a0 + T::load_row(u), m);
#pragma unroll
  for (int u = 0; u < T::LB; ++u) set_row(b[u], Kc, b0 + T::load_row(u), m);
  float2* P = part + (int64_t)blockIdx.y * ldp * ldp;
  int64_t s0 = p_begin;
  do {
    uint64_t acc[T::RM][4];
    T::block_k(sm, a, b, s0, min64(p_end, s0 + kChunk), acc);
    auto put = [&](int r, const float (&v)[8]) {
      const int64_t ra = a0 + T::row(r);
      if (ra >= m) return;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int64_t cb = b0 + T::col(c);
        if (cb >= m) continue;
        float2* dst = P + ra * ldp + cb;
        float2 sum = make_float2(v[c], 0.f);
        if (s0 != p_begin) {
          sum = *dst;
          pair_add(sum.x, sum.y, v[c]);
        }
        *dst = sum;
      }
    };
    if constexpr (T::KG > 1) {
      float v[8];
      T::combine(sm, acc, v);
      put(T::group(), v);
    } else {
#pragma unroll
      for (int r = 0; r < T::RM; ++r) {
        float v[8];
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float2 x = simt::unpack2(acc[r][p]);
          v[2 * p] = x.x;
          v[2 * p + 1] = x.y;
        }
        put(r, v);
      }
    }
    s0 += kChunk;
  } while (s0 < p_end);
}

}  // namespace

// Splits that fill the SMs: the small tile's block has one to itself; the wide
// tile's share it by threes (m = 1,500, ns = 30,000: 2.05 blocks per SM took
// 2.14 ms).
int64_t gram_simt_splits(int64_t m, int64_t ns_max) {
  const int64_t sms = sm_count();
  if (m <= kSmallBasis) return gram_splits(max64(1, upper_tiles<Small>(m)), sms, 1, 0.9, ns_max, kGramQuantumSimt);
  const int64_t tiles = upper_tiles<Wide>(m);
  return gram_splits(tiles, sms, ceil_div(5 * sms, 2 * tiles), 0.93, ns_max, kGramQuantumSimt);
}

int launch_gram_simt(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t m, float2* part,
                     int64_t ldp, int64_t splits, cudaStream_t s) {
  auto launch = [&](auto tile, auto rows) {
    using T = decltype(tile);
    const dim3 grid((unsigned)upper_tiles<T>(m), (unsigned)splits);
    auto kern = gram_simt_kernel<T, decltype(rows)>;
    const int smem = (int)(T::KG * sizeof(typename T::Smem));
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
      return;   // reported by the launch check
    kern<<<grid, T::THREADS, smem, s>>>(view(Kc), m, ns_dev, splits, part, ldp);
  };
  using F = simt::FloatRows<true>;   // a stored matrix's rows are 16-byte aligned
  using P = simt::PlaneRows;
  const bool planes = Kc->format != SPSVM_FP32;
  if (m <= kSmallBasis) planes ? launch(Small{}, P{}) : launch(Small{}, F{});
  else planes ? launch(Wide{}, P{}) : launch(Wide{}, F{});
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

// K_JJ[a][b] = (K[b][J[a]] + K[a][J[b]]) / 2 (the stored values made
// symmetric; exact in FP64) for the rows and columns from row0 on.  A fit
// keeps K_JJ in its workspace and extends it once per round, so the Gram
// finish reads it coalesced.  One block per 32 x 32 tile (ta <= tb): each
// scattered kernel value is read once, eight in flight a thread, and both
// halves are written along their rows.  Bound by the scattered sectors: m =
// 2,048 85 us (a thread per entry, two reads each: 155 us).
constexpr int FT = 32;
__global__ void __launch_bounds__(FT * 8) kjj_fill_kernel(KView K, const int64_t* __restrict__ J, int64_t m,
                                                          int64_t row0, double* __restrict__ kjj,
                                                          int64_t ldk) {
  __shared__ float B[FT][FT + 1];
  __shared__ double V[FT][FT + 1];
  // tiles of column block tb: ta = 0 .. tb, from the block that holds row0
  const int64_t t0 = row0 / FT;
  int64_t rem = blockIdx.x, tb = t0;
  while (rem > tb) rem -= ++tb;   // (column block tb has tb + 1 tiles)
  const int64_t ta = rem, a0 = ta * FT, b0 = tb * FT;
  const int c = threadIdx.x, y = threadIdx.y;
  const int64_t Jb = b0 + c < m ? J[b0 + c] : -1, Ja = a0 + c < m ? J[a0 + c] : -1;
  float va[4], vb[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = y + 8 * u;
    // the bias slot (point index -1) has no regulariser row or column
    va[u] = a0 + r < m && Jb >= 0 ? K.at(a0 + r, Jb) : 0.f;
    vb[u] = ta != tb && b0 + r < m && Ja >= 0 ? K.at(b0 + r, Ja) : 0.f;
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) B[y + 8 * u][c] = ta != tb ? vb[u] : va[u];
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = y + 8 * u;
    const int64_t a = a0 + r, b = b0 + c;
    double v = 0.0;
    if (a < m && b < m && Jb >= 0 && J[a] >= 0) v = 0.5 * ((double)B[c][r] + (double)va[u]);
    V[r][c] = v;
    if (a < m && b < m && (a >= row0 || b >= row0)) kjj[a * ldk + b] = v;
  }
  if (ta == tb) return;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = y + 8 * u;
    const int64_t b = b0 + r, a = a0 + c;
    if (a < m && b < m && (a >= row0 || b >= row0)) kjj[b * ldk + a] = V[c][r];
  }
}

// H[a][b] = H[b][a] = lambda K_JJ[a][b] + sum_s part[s][min(a,b)][max(a,b)]
// over 32 x 32 upper tiles (the partials are compensated FP32 pairs: an FP64 add
// has 1/64 of their rate): the partials, K_JJ and both halves of H move through
// shared memory so that every global access is coalesced.  Bound by the latency
// of the partials while the blocks leave SMs to spare (then eight splits are in
// flight a thread: 62 splits at m = 64 take 14 us more than one, 66 with one in
// flight), else by HBM (two, which leaves registers for six blocks an SM).
template <int KS>
__global__ void __launch_bounds__(FT * 8, KS == 8 ? 2 : 6) gram_finish_kernel(const float2* __restrict__ part,
                                                             GramPlan plan,
                                                             const int64_t* __restrict__ ns_dev,
                                                             int64_t quantum, int64_t ldp,
                                                             const double* __restrict__ kjj,
                                                             int64_t ldk, int64_t m, double lambda,
                                                             double* __restrict__ H, int64_t ldh) {
  __shared__ double P[FT][FT + 1];
  __shared__ double Kt[FT][FT + 1];
  const int64_t T = ceil_div(m, (int64_t)FT);
  int64_t rem = blockIdx.x, ta = 0;
  while (rem >= T - ta) {
    rem -= T - ta;
    ++ta;
  }
  const int64_t tb = ta + rem;
  const int64_t a0 = ta * FT, b0 = tb * FT;
  const int64_t ns = *ns_dev;   // the splits that hold points
  const int64_t splits = max64(1, ceil_div(ns, gram_split_points(ns, plan.splits(ns), quantum)));
  const int c = threadIdx.x;
  const int64_t b = b0 + c;
  // the thread's four rows of KS splits are read together (zeros past the last),
  // and added in order
  float h[FT / 8], l[FT / 8];
  const float2* src[FT / 8];
#pragma unroll
  for (int u = 0; u < FT / 8; ++u) {
    const int64_t a = a0 + threadIdx.y + 8 * u;
    h[u] = l[u] = 0.f;
    src[u] = a < m && b < m ? part + a * ldp + b : nullptr;
  }
  for (int64_t k0 = 0; k0 < splits; k0 += KS) {
    float2 v[KS][FT / 8];
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int u = 0; u < FT / 8; ++u)
        v[k][u] = src[u] && k0 + k < splits ? src[u][(k0 + k) * ldp * ldp] : make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < KS; ++k)
#pragma unroll
      for (int u = 0; u < FT / 8; ++u) pair_add(h[u], l[u], v[k][u]);
  }
#pragma unroll
  for (int u = 0; u < FT / 8; ++u) {
    const int r = threadIdx.y + 8 * u;
    P[r][c] = pair_value(h[u], l[u]);
    Kt[r][c] = a0 + r < m && b < m ? kjj[(a0 + r) * ldk + b] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < FT; r += 8) {
    const int64_t a = a0 + r;
    if (a < m && b < m) {
      // the partial of the upper triangle for both orientations
      const double pv = (ta == tb && r > c) ? P[c][r] : P[r][c];
      H[a * ldh + b] = lambda * Kt[r][c] + pv;
    }
  }
  if (ta != tb) {   // mirror tile: H[b0 + r][a0 + c] from the transposed values
    const int64_t a = a0 + c;
    for (int r = threadIdx.y; r < FT; r += 8) {
      const int64_t bb = b0 + r;
      if (a < m && bb < m) H[bb * ldh + a] = lambda * Kt[c][r] + P[c][r];
    }
  }
}

int launch_gram_finish(const float2* part, const GramPlan& plan, const int64_t* ns_dev, int64_t quantum, int64_t ldp,
                       const double* kjj, int64_t ldk, int64_t m, double lambda, double* H, int64_t ldh,
                       cudaStream_t s) {
  const int64_t T = ceil_div(m, (int64_t)FT);
  const int64_t blocks = T * (T + 1) / 2;
  auto kern = blocks <= sm_count() ? gram_finish_kernel<8> : gram_finish_kernel<2>;
  kern<<<(unsigned)blocks, dim3(FT, 8), 0, s>>>(part, plan, ns_dev, quantum, ldp, kjj, ldk, m, lambda, H, ldh);
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

size_t gram_part_bytes(int64_t m, int64_t ns) {
  if (m < 0 || ns < 0) return 0;
  const int64_t ldp = round_up(m > 0 ? m : 1, 64);
  int64_t splits = gram_simt_splits(m, ns);
  const int64_t tc = gram_tc_plan(m, ns).most();
  if (tc > splits) splits = tc;
  return (size_t)(splits * ldp * ldp * (int64_t)sizeof(float2));
}

int kjj_fill(const spsvm_kmat* K, const int64_t* J, int64_t m, int64_t row0, double* kjj,
             int64_t ldk, cudaStream_t s) {
  if (m <= row0) return SPSVM_OK;
  const int64_t t0 = row0 / FT, t1 = ceil_div(m, (int64_t)FT);   // column blocks [t0, t1), tb + 1 tiles each
  const int64_t tiles = t1 * (t1 + 1) / 2 - t0 * (t0 + 1) / 2;
  kjj_fill_kernel<<<(unsigned)tiles, dim3(FT, 8), 0, s>>>(view(K), J, m, row0, kjj, ldk);
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

}  // namespace spsvm

using namespace spsvm;

extern "C" size_t spsvm_gram_scratch_bytes(int64_t m, int64_t ns) {
  if (m < 0 || ns < 0) return 0;
  const int64_t ldp = round_up(m > 0 ? m : 1, 64);
  // the partial sums, then K_JJ gathered from K (a fit keeps its own)
  return gram_part_bytes(m, ns) + (size_t)(ldp * ldp * (int64_t)sizeof(double));
}

namespace spsvm {
int gram_impl(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t ns_max, const spsvm_kmat* K,
              const int64_t* J, double lambda, int32_t precision, double* H, int64_t ldh,
              void* scratch, size_t scratch_bytes, cudaStream_t s, int64_t ns_hint,
              const double* kjj, int64_t ldk) {
  SPSVM_TRY(check_kmat(Kc, "gram(Kc)"));
  SPSVM_TRY(check_kmat(K, "gram(K)"));
  if (!ns_dev || !J || !H) return set_error(SPSVM_ERR_ARG, "gram: NULL pointer");
  const int64_t m = K->rows;
  if (Kc->rows < m || ldh < m || ns_max < 0 || ns_max > Kc->n || !(lambda > 0.0))
    return set_error(SPSVM_ERR_ARG, "gram: bad shapes m=%lld Kc.rows=%lld ldh=%lld ns_max=%lld",
                     (long long)m, (long long)Kc->rows, (long long)ldh, (long long)ns_max);
  if (m == 0) return SPSVM_OK;
  const size_t need = kjj ? gram_part_bytes(m, ns_max) : spsvm_gram_scratch_bytes(m, ns_max);
  if (!scratch || scratch_bytes < need) return set_error(SPSVM_ERR_OOM, "gram: scratch too small");
  // algorithmic work: one multiply-add per active point per unique entry,
  // times the four plane products of the BF16SPLIT form
  ProfScope prof(PROF_GRAM, s,
                 (precision == SPSVM_BF16SPLIT ? 4.0 : 1.0) * (double)(ns_hint >= 0 ? ns_hint : ns_max) * (double)m * (double)(m + 1));
  const int64_t ldp = round_up(m, 64);
  float2* part = static_cast<float2*>(scratch);
  if (!kjj) {   // gather K_JJ into the scratch behind the partial sums
    double* kj = reinterpret_cast<double*>(static_cast<char*>(scratch) + gram_part_bytes(m, ns_max));
    SPSVM_TRY(kjj_fill(K, J, m, 0, kj, ldp, s));
    kjj = kj;
    ldk = ldp;
  }
  GramPlan plan{0, 1};
  if (precision == SPSVM_BF16SPLIT) {
    if (Kc->format != SPSVM_BF16SPLIT) return set_error(SPSVM_ERR_ARG, "gram: BF16SPLIT needs split planes");
    plan = gram_tc_plan(m, ns_max);
    SPSVM_TRY(launch_gram_tc(Kc, ns_dev, ns_max, ns_hint, m, part, ldp, plan, s));
  } else if (precision == SPSVM_FP32) {
    plan.s_pair = gram_simt_splits(m, ns_max);
    SPSVM_TRY(launch_gram_simt(Kc, ns_dev, m, part, ldp, plan.s_pair, s));
  } else {
    return set_error(SPSVM_ERR_ARG, "gram: bad precision");
  }
  return launch_gram_finish(part, plan, ns_dev,
                            precision == SPSVM_FP32 ? kGramQuantumSimt : kGramQuantumTc, ldp, kjj, ldk,
                            m, lambda, H, ldh, s);
}
}  // namespace spsvm

extern "C" int spsvm_gram(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t ns_max,
                          const spsvm_kmat* K, const int64_t* J, double lambda, int32_t precision,
                          double* H, int64_t ldh, void* scratch, size_t scratch_bytes,
                          void* stream) {
  return gram_impl(Kc, ns_dev, ns_max, K, J, lambda, precision, H, ldh, scratch, scratch_bytes,
                   as_stream(stream), -1, nullptr, 0);
}
