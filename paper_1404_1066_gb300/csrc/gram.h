// Shared declarations of the Gram-matrix (masked SYRK) launchers.
#pragma once
#include "internal.h"

namespace spsvm {

// Points per tensor-core accumulation of the split form.
constexpr int64_t GRAM_SLICE = 8192;

// Both forms split the active points evenly over at most kGramMaxSplits
// partial matrices (or, where a wave of blocks takes more, one for each slice of
// GRAM_SLICE points: matrices of few tiles on many points, m = 64, ns = 200,000
// in split form 93 us, 239 with 16) of at least a quantum of points: in
// the FP32 form about what a partial matrix costs to write and add, in the split
// form a slice.
// Their number is read on the device, so the last splits may be empty (they
// are neither written nor read).
constexpr int64_t kGramQuantumSimt = 128;
constexpr int64_t kGramQuantumTc = GRAM_SLICE;
constexpr int64_t kGramMaxSplits = 16;
__host__ __device__ __forceinline__ int64_t gram_split_points(int64_t ns, int64_t splits, int64_t quantum) {
  return max64(quantum, round_up(ceil_div(ns, splits), (int64_t)128));
}

inline int64_t gram_most_splits(int64_t tiles, int64_t slots, int64_t ns_max) {
  return max64(kGramMaxSplits, min64(slots / max64(1, tiles), ceil_div(ns_max, GRAM_SLICE)));
}

// The fewest splits, from `least`, that fill whole waves of `slots` blocks to
// `good`, else those that fill them best.
inline int64_t gram_splits(int64_t tiles, int64_t slots, int64_t least, double good, int64_t ns_max,
                           int64_t quantum) {
  const int64_t most = max64(1, min64(gram_most_splits(tiles, slots, ns_max), ceil_div(ns_max, quantum)));
  int64_t best = min64(max64(1, least), most);
  double be = 0.0;
  for (int64_t s = best; s <= most; ++s) {
    const double e = (double)(tiles * s) / (double)(slots * ceil_div(tiles * s, slots));
    if (e > be) {
      be = e;
      best = s;
    }
    if (e >= good) break;
  }
  return best;
}

int64_t gram_simt_splits(int64_t m, int64_t ns_max);
int launch_gram_simt(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t m, float2* part,
                     int64_t ldp, int64_t splits, cudaStream_t s);

// ns_hint: *ns_dev when the host knows it, else -1.  kjj: the symmetric K_JJ (FP64, row pitch ldk) if the caller keeps one, else
// NULL (gathered from K into the scratch behind the partial sums).
int gram_impl(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t ns_max, const spsvm_kmat* K,
              const int64_t* J, double lambda, int32_t precision, double* H, int64_t ldh,
              void* scratch, size_t scratch_bytes, cudaStream_t s, int64_t ns_hint,
              const double* kjj, int64_t ldk);

// Scratch of the partial sums alone (with a caller-kept K_JJ).
size_t gram_part_bytes(int64_t m, int64_t ns);

// K_JJ entries in the rows and columns row0 .. m-1 (see gram_simt.cu).
int kjj_fill(const spsvm_kmat* K, const int64_t* J, int64_t m, int64_t row0, double* kjj,
             int64_t ldk, cudaStream_t s);

// The split form's two kernels: single CTAs on 128 x 128 tiles while one wave
// of them holds every slice of the ns points separately, else pairs on 256 x
// 256 tiles.  s_single (0: never), s_pair: the splits of each.
struct GramPlan {
  int64_t s_single, s_pair;
  __host__ __device__ __forceinline__ bool single(int64_t ns) const {
    return ceil_div(ns, kGramQuantumTc) <= s_single && s_single > 0;
  }
  __host__ __device__ __forceinline__ int64_t splits(int64_t ns) const { return single(ns) ? s_single : s_pair; }
  int64_t most() const { return max64(s_single, s_pair); }
};
GramPlan gram_tc_plan(int64_t m, int64_t ns_max);
int launch_gram_tc(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t ns_max, int64_t ns_hint,
                   int64_t m, float2* part, int64_t ldp, const GramPlan& plan, cudaStream_t s);

}  // namespace spsvm
