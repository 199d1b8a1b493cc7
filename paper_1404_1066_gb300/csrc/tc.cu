// tcgen05 (sm_103a) tensor-core kernels of the SPSVM_BF16SPLIT form.
//
//   * kernel block / candidate scores / decision values (RBF kernel of
//     Section 2 through the distance expansion; the basis-vector score of
//     Section 4; the classifier h(x) = w^T phi(x) on the basis): points X
//     (TMA, 128 rows per tile) times gathered basis / candidate rows, each
//     FP32 value split into three BF16 terms hi + mid + lo (exact) and
//     multiplied as six products, with a fused epilogue
//     exp(-gamma max(0, |x|^2 + |z|^2 - 2 x.z)) that stores the kernel
//     values (FP32), or reduces the score sums or the beta-weighted decision
//     sums without storing them;
//   * masked Gram matrix K_SJ^T K_SJ (the Hessian term of Eq. 4 on the
//     active set): the compact copy split as hi + lo (lo = bf16(x - hi)) and
//     all four plane products, warp-specialised TMA producer / MMA issuer /
//     epilogue over 256 x 256 upper-triangular tiles of CTA pairs with two
//     TMEM accumulators, FP32 partial sums per 8,192 points added up as
//     compensated pairs.
#include <cudaTypedefs.h>

#include <type_traits>

#include "gram.h"
#include "internal.h"
#include "simt_tile.h"
#include "tc_ptx.h"

namespace spsvm {

namespace {

using namespace tc;
using simt::dup2;
using simt::fma2;
using simt::mul2;
using simt::pack2;
using simt::unpack2;

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
  const uint32_t a = smem_u32(p);
  return p + ((1024u - (a & 1023u)) & 1023u);
}

// ---------------------------------------------------------------------------
// The end of a block after a wait that gave up.  A block must not end, nor free
// its TMEM, with copies or MMAs of its own in flight; without a give-up the
// producers' last wait (for the slots to be consumed) and the epilogue's see to
// that.  The words lie in shared memory, the same in both CTAs of a pair.
// ---------------------------------------------------------------------------
struct Leave {
  uint32_t gave;      // nonzero: a wait gave up
  uint32_t left[2];   // slots that each CTA's producer has issued loads for
};
template <bool PAIR>
__device__ __forceinline__ void leave_word(uint32_t* w, uint32_t v) {
  if constexpr (PAIR) {
    st_cluster(map_rank(w, 0), v);
    st_cluster(map_rank(w, 1), v);
  } else {
    *(volatile uint32_t*)w = v;
  }
}
// Waits (for a second or so each) for all copies and MMAs issued.  Called by all
// threads after a barrier behind the roles and before another one.  bytes: what
// one CTA loads per slot; drain: expects the 32 lanes of warp 1 of the even CTA.
// Where a pair's producers stopped at different slots, the even one's barrier
// expects exactly the copies that were issued.
template <bool PAIR, int SLOTS>
__device__ __noinline__ void settle(uint64_t* full, uint64_t* drain, const Leave* lv, uint32_t bytes,
                                    uint32_t rank, int* st) {
  if (threadIdx.x == 0 && rank == 0) {
    const uint32_t q0 = lv->left[0], q1 = PAIR ? lv->left[1] : q0;
    const uint32_t top = q0 > q1 ? q0 : q1;
    for (uint32_t r = top > SLOTS ? top - SLOTS : 0; r < top; ++r) {
      uint64_t* bar = &full[r % SLOTS];
      if (r >= q0) mbar_expect_tx(bar, bytes);
      else if (r >= q1) mbar_complete_tx(bar, bytes);
      mbar_wait(bar, (r / SLOTS) & 1, st, 28, 0);
    }
  }
  if (threadIdx.x >> 5 == 1) {
    if (rank == 0) {
      if constexpr (PAIR) mma_commit_pair(drain);
      else mma_commit(drain);
    }
    mbar_wait(drain, 0, st, 29, 0);
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Kernel block / scores / decision values, persistent and warp-specialised:
// products x.z over tiles of rows (MMA M) by columns (MMA N), both operands
// streamed by TMA, each FP32 value as three planes (x = hi + mid + lo, exact)
// and multiplied as the six products hi hi, hi mid, mid hi, mid mid, hi lo, lo
// hi (the three dropped ones are below 2^-24 of |x z|), hi hi into one TMEM
// accumulator and the rest into a second (the FP32 accumulation's rounding
// grows with the MMAs a sum takes, and only the few large-term ones then
// count).  Epilogue modes:
//   STORE   rows the points, columns the basis: the FP32 kernel values (a warp
//           stores 32 consecutive points of a basis row);
//   SCORE   rows the candidates, columns the points: the score sums, a
//           thread's own over its columns of all of the CTA's tiles, or per
//           tile where tiles are few (kernel values not stored);
//   DECIDE  rows the queries, columns the basis: sums of beta K over 32.
// Basis and candidate rows are gathered into contiguous planes beforehand.
//
// Warp 0 issues the TMA loads, warp 1 the MMAs into one of two tile buffers,
// the other warps drain the other (TMEM lane = row; four lane quarters by
// groups of 32 columns).  A slot of the shared-memory ring holds 64 columns of K
// of both operands, in one plane (a pair, whose chunk starts as soon as its hi
// planes are there) or in all three.  With more than 128 rows two CTAs work as a pair (PAIR,
// cta_group::2) on 256 rows, each staging 128 rows and half of the columns,
// the even one issuing the MMAs for both: a 128 x 128 MMA of one CTA reads its
// operands from shared memory at the full 128 bytes a cycle, with loads of 64
// bytes a cycle on top, the pair reads 96 and loads 47.  Up to 64 columns take
// a tile of 64 (N), at 128 half of the products would be padding.
//
// MMAs on the same plane of the rows stand together, so the rows are read from
// shared memory three times a step instead of six.  Arrivals of a pair are
// relaxed (a release waits for the epilogue's global stores).
// 32,768 queries by 4,096 basis rows, d = 128: 117 us, 1.77 PFLOP/s in the six
// products (154 us in 128 x 128 tiles of single CTAs with the queries as
// columns, where each sum over a warp's rows took 31 exchanges).  Scores of 256
// candidates, n = 500,000: 130 us (157).  Kernel block of 64 rows, n = 500,000:
// 76 us, 512 MB at 6.7 TB/s (90 us in tiles of 128 basis rows).
// ---------------------------------------------------------------------------
enum KbMode { KB_STORE_F32 = 0, KB_SCORE = 2, KB_DECIDE = 3 };

constexpr int PK_M = 128;                                  // rows per CTA
constexpr int PK_KC = 64;                                  // K elements per slot (128-byte rows)
constexpr int PK_WP = 32;                                  // columns per epilogue warp
// RA: rows of A that a CTA stages (64: the MMAs' other rows are whatever lies
// behind, and are not read back)
template <bool PAIR, int N, int RA>
struct Kb {
  static constexpr int CTAS = PAIR ? 2 : 1;
  // Planes per slot.  A single CTA waits once for all three: with a wait for
  // each, the MMAs of a chunk started late (20,000 points by 128 candidates,
  // d = 500: 27.8 us so, 31.6 plane by plane)
  static constexpr int PPS = PAIR ? 1 : 3;
  static constexpr int M = CTAS * PK_M;                    // rows of a tile
  static constexpr int ROWS_B = N / CTAS;                  // columns staged per CTA
  static constexpr int GROUPS = N / PK_WP;
  static constexpr int EPI_WARPS = 4 * GROUPS;
  static constexpr int THREADS = 32 * (2 + EPI_WARPS);
  static constexpr int PLANE_A = RA * PK_KC * 2;
  static constexpr int PLANE = PLANE_A + ROWS_B * PK_KC * 2;   // of both operands
  static constexpr int SLOT = PPS * PLANE;
  static constexpr int SLOTS = 192 * 1024 / SLOT;
  static constexpr int RED_OFF = SLOTS * SLOT;             // SCORE: the groups' sums
  static constexpr int BAR_OFF = RED_OFF + (GROUPS - 1) * 128 * 16;
  static constexpr int STAGE_OFF = BAR_OFF + 512;          // per epilogue warp: 3 x 32 floats
  static constexpr int SMEM = STAGE_OFF + EPI_WARPS * 3 * PK_WP * 4 + 1024;   // + alignment slack
  static_assert(SMEM <= 227 * 1024, "kernel block shared memory");
  static_assert(8 * (2 * SLOTS + 13) + 12 + sizeof(Leave) <= 512, "barriers");
  static_assert(SLOTS * PPS >= 6, "two chunks in flight");
  static_assert(PLANE >= PK_M * PK_KC * 2, "the rows that the MMAs read lie in the slot");
};

// Tile order: groups of PK_GROUP consecutive column tiles (STORE: row blocks,
// so that a basis row's values reach DRAM in runs of PK_GROUP x 1 KB), each
// group swept over all row blocks (column tiles) with the group's own index
// varying fastest.  The CTAs in flight share tiles of both operands through L2.
constexpr int64_t PK_GROUP = 32;
template <int MODE, typename I>
__device__ __forceinline__ void tile_coords_as(I t, I nCB, I nPT, int& cb, int64_t& pt) {
  constexpr I G = (I)PK_GROUP;
  const I grouped = MODE == KB_STORE_F32 ? nCB : nPT, other = MODE == KB_STORE_F32 ? nPT : nCB;
  const I per = other * G;
  const I g = t / per, r = t - g * per;
  const I g0 = g * G;
  const I gw = grouped - g0 < G ? grouped - g0 : G;   // the last group may be narrower
  const I a = r / gw, b = g0 + (r - a * gw);
  cb = (int)(MODE == KB_STORE_F32 ? b : a);
  pt = (int64_t)(MODE == KB_STORE_F32 ? a : b);
}
// (64-bit divisions would take as long as a tile's epilogue)
template <int MODE>
__device__ __forceinline__ void tile_coords(int64_t t, int64_t nCB, int64_t nPT, int& cb, int64_t& pt) {
  if (nCB * nPT < (int64_t)1 << 26) tile_coords_as<MODE, uint32_t>((uint32_t)t, (uint32_t)nCB, (uint32_t)nPT, cb, pt);
  else tile_coords_as<MODE, int64_t>(t, nCB, nPT, cb, pt);
}

template <int MODE, bool PAIR, int N, int RA>
__global__ void __launch_bounds__(Kb<PAIR, N, RA>::THREADS, 1) kblock_tc_kernel(
    const __grid_constant__ CUtensorMap map_ahi, const __grid_constant__ CUtensorMap map_amid,
    const __grid_constant__ CUtensorMap map_alo, const __grid_constant__ CUtensorMap map_bhi,
    const __grid_constant__ CUtensorMap map_bmid, const __grid_constant__ CUtensorMap map_blo,
    int64_t ldh, int64_t ncols, int64_t nrows, int box_a,
    const float* __restrict__ colnorm, const float* __restrict__ rownorm,
    const int64_t* __restrict__ idx, float gamma, float* __restrict__ out, int64_t ld,
    const float* __restrict__ y,
    const float* __restrict__ o, float4* __restrict__ part, int per_tile, const double* __restrict__ beta,
    float* __restrict__ dpart, int64_t ldp, WaitCtx wc) {
  constexpr bool SCORE = MODE == KB_SCORE;
  constexpr bool STORE = MODE == KB_STORE_F32;
  constexpr bool DECIDE = MODE == KB_DECIDE;
  using TL = Kb<PAIR, N, RA>;
  constexpr int SLOTS = TL::SLOTS, KC = PK_KC, PPS = TL::PPS, GROUPS = TL::GROUPS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + TL::BAR_OFF);
  uint64_t* empty = full + SLOTS;
  uint64_t* tfull = empty + SLOTS;
  uint64_t* tempty = tfull + 2;
  uint64_t* redf = tempty + 2;   // per lane quarter: the groups' sums written
  uint64_t* rede = redf + 4;     // per lane quarter: the groups' sums consumed
  uint64_t* drain = rede + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  uint32_t* bad = tmem_slot + 1;   // [2], PAIR: a wait had given up before, as each CTA saw it
  Leave* leave = reinterpret_cast<Leave*>(bad + 2);
  float4* red = reinterpret_cast<float4*>(smem + TL::RED_OFF);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const int64_t unit = PAIR ? blockIdx.x >> 1 : blockIdx.x, units = PAIR ? gridDim.x >> 1 : gridDim.x;
  if (!PAIR && __syncthreads_or(tid == 0 && *(volatile int*)wc.st != 0)) return;
  const int64_t nCB = ceil_div(nrows, (int64_t)TL::M);
  const int64_t nPT = ceil_div(ncols, (int64_t)N);
  const int64_t T = nCB * nPT;
  const int nK = (int)(ldh / KC);
  constexpr uint32_t IDESC = idesc_bf16_f32(TL::M, N);

  if (tid == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], TL::CTAS * TL::EPI_WARPS);   // one arrival per epilogue warp
    }
    for (int qd = 0; qd < 4; ++qd) {
      mbar_init(&redf[qd], 32 * (GROUPS - 1));
      mbar_init(&rede[qd], 32);
    }
    mbar_init(drain, 32);
    *leave = Leave{0u, {0u, 0u}};
    fence_barrier_init();
    prefetch_tmap(&map_ahi);
    prefetch_tmap(&map_amid);
    prefetch_tmap(&map_alo);
    prefetch_tmap(&map_bhi);
    prefetch_tmap(&map_bmid);
    prefetch_tmap(&map_blo);
  }
  bool live = true;
  if constexpr (PAIR) {
    __syncwarp();
    cluster_sync();   // both CTAs run, and their barriers are initialised
    if (tid == 0) {
      const uint32_t st = *(volatile int*)wc.st != 0 ? 1u : 0u;
      st_cluster(map_rank(&bad[rank], 0), st);
      st_cluster(map_rank(&bad[rank], 1), st);
    }
    __syncwarp();
    if (warp == 0) tmem_alloc_pair(tmem_slot, 4 * N);
    fence_before_sync();
    cluster_sync();
    live = bad[0] == 0 && bad[1] == 0;   // the same in both CTAs
  } else {
    if (warp == 0) tmem_alloc(tmem_slot, 4 * N);
    fence_before_sync();
    __syncthreads();
  }
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  auto note = [&](bool ok) {   // every wait's outcome goes through this
    if (!ok) leave_word<PAIR>(&leave->gave, 1u);
    return ok;
  };
  // for a barrier that threads or MMAs of the other CTA may complete; the
  // producer's acquires, what follows it writes over what the MMAs read
  auto wait = [&](uint64_t* bar, uint32_t parity, int code) {
    return note(PAIR ? mbar_wait_cluster<false>(bar, parity, wc.st, code, wc.lim)
                     : mbar_wait(bar, parity, wc.st, code, wc.lim));
  };
  auto wait_free = [&](uint64_t* bar, uint32_t parity, int code) {
    return note(PAIR ? mbar_wait_cluster<true>(bar, parity, wc.st, code, wc.lim)
                     : mbar_wait(bar, parity, wc.st, code, wc.lim));
  };

  const uint32_t slot_bytes = (uint32_t)(TL::SLOT - PPS * (RA - box_a) * 128);   // of one CTA
  if (!live) {
  } else if (warp == 0) {
    if (lane == 0) {
      // ---- TMA producer (of a pair: both CTAs' loads complete on the even one's barrier)
      int64_t q = 0;
      bool ok = true;
      const CUtensorMap* ma[3] = {&map_ahi, &map_amid, &map_alo};
      const CUtensorMap* mb[3] = {&map_bhi, &map_bmid, &map_blo};
      for (int64_t t = unit; t < T && ok; t += units) {
        int cb;
        int64_t pt;
        tile_coords<MODE>(t, nCB, nPT, cb, pt);
        const int ra = cb * TL::M + (int)rank * PK_M, rb = (int)(pt * N) + (int)rank * TL::ROWS_B;
        for (int kc = 0; kc < nK && ok; ++kc) {
#pragma unroll
          for (int p = 0; p < 3; p += PPS, ++q) {
            const int s = (int)(q % SLOTS);
            if (!wait_free(&empty[s], (uint32_t)((q / SLOTS) & 1) ^ 1u, 21)) {
              ok = false;
              break;
            }
            if (rank == 0) mbar_expect_tx(&full[s], TL::CTAS * slot_bytes);
#pragma unroll
            for (int e = 0; e < PPS; ++e) {
              uint8_t* st = smem + s * TL::SLOT + e * TL::PLANE;
              if constexpr (PAIR) {
                const uint32_t bar = map_rank(&full[s], 0);
                tma_load_2d_pair(st, ma[p + e], kc * KC, ra, bar);
                tma_load_2d_pair(st + TL::PLANE_A, mb[p + e], kc * KC, rb, bar);
              } else {
                tma_load_2d(st, ma[p + e], kc * KC, ra, &full[s]);
                tma_load_2d(st + TL::PLANE_A, mb[p + e], kc * KC, rb, &full[s]);
              }
            }
          }
        }
      }
      // the last slots consumed: their copies and the MMAs' arrivals here are done
      for (int64_t r = (q > SLOTS ? q - SLOTS : 0); r < q && ok; ++r)
        ok = wait_free(&empty[r % SLOTS], (uint32_t)((r / SLOTS) & 1), 22);
      leave_word<PAIR>(&leave->left[rank], (uint32_t)q);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---- MMA issuer: the whole warp runs the loop, one lane issues; a wait
      // counts as run out for all lanes when it has for one
      auto mma = [&](auto use, uint32_t d, uint32_t a, uint32_t b, uint32_t accumulate) {
        constexpr int A = decltype(use)::value;
        if constexpr (PAIR) mma_bf16_pair<A>(d, desc_sw128(a), desc_sw128(b), IDESC, accumulate);
        else mma_bf16<A>(d, desc_sw128(a), desc_sw128(b), IDESC, accumulate);
      };
      const std::integral_constant<int, A_DISCARD> once;
      const std::integral_constant<int, A_FILL> fill;
      const std::integral_constant<int, A_USE> use;
      const std::integral_constant<int, A_LASTUSE> last;
      auto commit = [&](uint64_t* bar) {
        if constexpr (PAIR) mma_commit_pair(bar);
        else mma_commit(bar);
      };
      int64_t q = 0, j = 0;
      bool ok = true;
      for (int64_t t = unit; t < T && ok; t += units, ++j) {
        const int acc = (int)(j & 1);
        if (!__all_sync(~0u, wait(&tempty[acc], (uint32_t)((j >> 1) & 1) ^ 1u, 23))) break;
        fence_after_sync();
        // hi hi products in one accumulator, the five smaller ones (2^-8 and
        // below) in another: the FP32 accumulation's rounding then grows with
        // the few large-term MMAs only
        const uint32_t d_big = tmem + acc * 2 * N;
        const uint32_t d_small = d_big + N;
        for (int kc = 0; kc < nK && ok; ++kc) {
          uint32_t a[3], b[3];
          int slot[3];
#pragma unroll
          for (int p = 0; p < 3; p += PPS, ++q) {
            slot[p] = (int)(q % SLOTS);
#pragma unroll
            for (int e = 0; e < PPS; ++e) {
              a[p + e] = smem_u32(smem + slot[p] * TL::SLOT) + e * TL::PLANE;
              b[p + e] = a[p + e] + TL::PLANE_A;
            }
            if (!__all_sync(~0u, note(mbar_wait(&full[slot[p]], (uint32_t)((q / SLOTS) & 1), wc.st, 24, wc.lim)))) {
              ok = false;
              break;
            }
          }
          if (!ok) break;
          fence_after_sync();
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < KC / 16; ++k) {
              const uint32_t koff = k * 32, first = (kc | k) != 0 ? 1u : 0u;
              mma(fill, d_big, a[0] + koff, b[0] + koff, first);
              mma(use, d_small, a[0] + koff, b[1] + koff, first);
              mma(last, d_small, a[0] + koff, b[2] + koff, 1u);
              mma(fill, d_small, a[1] + koff, b[0] + koff, 1u);
              mma(last, d_small, a[1] + koff, b[1] + koff, 1u);
              mma(once, d_small, a[2] + koff, b[0] + koff, 1u);
            }
            for (int p = 0; p < 3; p += PPS) commit(&empty[slot[p]]);
            if (kc == nK - 1) commit(&tfull[acc]);
          }
          __syncwarp();
        }
      }
    }
  } else {
    // ---- epilogue: warp w drains lane quarter w % 4, columns group * 32 ..
    const int quarter = warp & 3;
    const int group = (warp - 2) >> 2;
    const int c_in = 32 * quarter + lane;
    const float g2 = gamma * 1.4426950408889634f;   // K = 2^(-g2 |x - z|^2)
    const uint64_t m2 = dup2(-g2), p2 = dup2(2.0f * g2);
    float* stage = reinterpret_cast<float*>(smem + TL::STAGE_OFF) + (warp - 2) * 3 * PK_WP;
    // What a lane needs of a tile besides the product: its row's norm, and of
    // one of the warp's columns the norm, the output and label (SCORE) or the
    // coefficient (DECIDE); zero outside.  Read a tile ahead.
    struct Pre {
      float rn, cn, oi, yi;
      double b;
      int cb;
      int64_t pt;
    };
    auto fetch = [&](int64_t t) {
      Pre f{0.f, 0.f, 0.f, 0.f, 0.0, -1, 0};
      if (t >= T) return f;
      tile_coords<MODE>(t, nCB, nPT, f.cb, f.pt);
      const int64_t c = (TL::CTAS * (int64_t)f.cb + rank) * PK_M + c_in;
      const int64_t i = f.pt * N + group * PK_WP + lane;
      if (c < nrows) f.rn = rownorm[SCORE ? idx[c] : c];
      if (i < ncols) {
        f.cn = colnorm[STORE ? idx[i] : i];
        if (SCORE) {
          f.oi = o[i];
          f.yi = y[i];
        }
        if (DECIDE) f.b = beta[i];
      }
      return f;
    };
    Pre next = fetch(unit);
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);   // SCORE: compensated pairs of this thread's sums
    int flushes = 0;
    if (SCORE && group == 0 && !per_tile)
      for (int64_t c = rank * PK_M + c_in; c < nrows; c += TL::M) part[unit * nrows + c] = sum;
    int64_t j = 0;
    for (int64_t t = unit; t < T; t += units, ++j) {
      const int cb = next.cb;
      const int64_t pt = next.pt;
      const int64_t cblock = TL::CTAS * (int64_t)cb + rank;   // this CTA's 128 rows
      const int64_t c = cblock * PK_M + c_in;
      const bool crow = c < nrows;
      const int64_t ib = pt * N + group * PK_WP;
      const bool any = ib < ncols;   // uniform per warp
      const float zz = -g2 * next.rn;
      __syncwarp();   // the stage has been read
      stage[lane] = next.cn;
      if (SCORE) {
        const bool active = next.yi * next.oi < 1.0f && ib + lane < ncols;
        stage[PK_WP + lane] = active ? next.oi - next.yi : 0.f;
        stage[2 * PK_WP + lane] = active ? 1.f : 0.f;
      }
      if (DECIDE) stage[PK_WP + lane] = (float)next.b;
      __syncwarp();
      const int acc = (int)(j & 1);
      if (!__all_sync(~0u, wait(&tfull[acc], (uint32_t)((j >> 1) & 1), 25))) break;
      fence_after_sync();
      const uint32_t tb = tmem + acc * 2 * N + group * PK_WP + ((uint32_t)(32 * quarter) << 16);
      uint64_t v[16];   // x.z = large terms + small terms, two columns each
      {
        float a[32], b[32];
        tmem_ld32(tb, a);
        tmem_ld32(tb + N, b);
#pragma unroll
        for (int jj = 0; jj < 16; ++jj)
          v[jj] = pack2(a[2 * jj] + b[2 * jj], a[2 * jj + 1] + b[2 * jj + 1]);
      }
      // the accumulators are in registers: the next tile's MMAs may start
      fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR) mbar_arrive_cluster(map_rank(&tempty[acc], 0));
        else mbar_arrive(&tempty[acc]);
      }
      next = fetch(t + units);
      float gs = 0.f, hs = 0.f;
      if (any) {
        // arg = -g2 * max(|x|^2 + |z|^2 - 2 x.z, 0); columns past the last
        // carry zero norms here and are not stored or weighted by zero
        const uint64_t z2 = dup2(zz);
#pragma unroll
        for (int jj = 0; jj < 16; jj += 2) {
          const ulonglong2 x4 = *reinterpret_cast<const ulonglong2*>(stage + 2 * jj);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint64_t a = z2;
            fma2(a, p2, v[jj + h]);
            fma2(a, m2, h ? x4.y : x4.x);
            const float2 f = unpack2(a);
            v[jj + h] = pack2(ex2_approx(fminf(f.x, 0.0f)), ex2_approx(fminf(f.y, 0.0f)));
          }
        }
        if (STORE) {
          float* dst = out + ib * ld + c;
          const int64_t left = ncols - ib;
          if (crow) {
#pragma unroll
            for (int jj = 0; jj < 16; ++jj) {
              const float2 f = unpack2(v[jj]);
              if (2 * jj < left) dst[2 * jj * ld] = f.x;
              if (2 * jj + 1 < left) dst[(2 * jj + 1) * ld] = f.y;
            }
          }
        } else {
          // SCORE: the sums of (o - y) K and K^2 over the active columns;
          // DECIDE: of beta K over the columns; in chains of 8 and 4 terms
          uint64_t g2s[4] = {0, 0, 0, 0}, h2s[2] = {0, 0};
          constexpr int CH = SCORE ? 2 : 4;
#pragma unroll
          for (int jj = 0; jj < 16; jj += 2) {
            const ulonglong2 r4 = *reinterpret_cast<const ulonglong2*>(stage + PK_WP + 2 * jj);
            fma2(g2s[jj % CH], r4.x, v[jj]);
            fma2(g2s[jj % CH + 1], r4.y, v[jj + 1]);
            if (SCORE) {
              const ulonglong2 a4 = *reinterpret_cast<const ulonglong2*>(stage + 2 * PK_WP + 2 * jj);
              fma2(h2s[0], mul2(a4.x, v[jj]), v[jj]);
              fma2(h2s[1], mul2(a4.y, v[jj + 1]), v[jj + 1]);
            }
          }
          const float2 ga = unpack2(g2s[0]), gb = unpack2(g2s[1]), gc = unpack2(g2s[2]), gd = unpack2(g2s[3]);
          gs = (ga.x + ga.y) + (gb.x + gb.y);
          if (CH == 4) gs += (gc.x + gc.y) + (gd.x + gd.y);
          const float2 ha = unpack2(h2s[0]), hb = unpack2(h2s[1]);
          hs = (ha.x + ha.y) + (hb.x + hb.y);
        }
      }
      // one partial per 32 basis rows and query, summed in a fixed order by
      // the finish
      if (DECIDE && crow && any) dpart[ib / PK_WP * ldp + c] = gs;
      if (SCORE) {
        pair_add(sum.x, sum.y, gs);
        pair_add(sum.z, sum.w, hs);
        if (next.cb == cb && !per_tile) continue;   // the next tile's rows are the same: keep the sums
        // the warps of a lane quarter combine their groups of columns, in order
        const uint32_t par = (uint32_t)(flushes & 1);
        ++flushes;
        if (group > 0) {
          if (!__all_sync(~0u, note(mbar_wait(&rede[quarter], par ^ 1u, wc.st, 26, wc.lim)))) break;
          red[(group - 1) * 128 + c_in] = sum;
          mbar_arrive(&redf[quarter]);
        } else {
          if (!__all_sync(~0u, note(mbar_wait(&redf[quarter], par, wc.st, 27, wc.lim)))) break;
          float4* dst = part + (per_tile ? pt : unit) * nrows + c;
          float4 all = sum;
          if (crow && !per_tile) {
            const float4 r = *dst;
            pair_add(all.x, all.y, make_float2(r.x, r.y));
            pair_add(all.z, all.w, make_float2(r.z, r.w));
          }
#pragma unroll
          for (int g = 0; g < GROUPS - 1; ++g) {
            const float4 r = red[g * 128 + c_in];
            pair_add(all.x, all.y, make_float2(r.x, r.y));
            pair_add(all.z, all.w, make_float2(r.z, r.w));
          }
          mbar_arrive(&rede[quarter]);
          if (crow) *dst = all;
        }
        sum = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
  fence_before_sync();
  if constexpr (PAIR) {
    __syncwarp();
    cluster_sync();   // no copy, MMA or arrival of the pair is outstanding, or
    if (*(volatile uint32_t*)&leave->gave) {
      settle<PAIR, SLOTS>(full, drain, leave, slot_bytes, rank, wc.st);
      cluster_sync();
    }
    if (warp == 0) {
      fence_after_sync();
      tmem_dealloc_pair(tmem, 4 * N);
    }
  } else {
    __syncthreads();
    if (*(volatile uint32_t*)&leave->gave) {
      settle<PAIR, SLOTS>(full, drain, leave, slot_bytes, 0, wc.st);
      __syncthreads();
    }
    if (warp == 0) {
      __syncwarp();
      fence_after_sync();
      tmem_dealloc(tmem, 4 * N);
    }
  }
}

// Rows idx[0..m) of the three split planes, contiguous.
__global__ void gather_rows_bf16(const uint16_t* __restrict__ Xhi, const uint16_t* __restrict__ Xmid,
                                 const uint16_t* __restrict__ Xlo, int64_t ldh,
                                 const int64_t* __restrict__ idx, int32_t m,
                                 uint16_t* __restrict__ Zhi, uint16_t* __restrict__ Zmid,
                                 uint16_t* __restrict__ Zlo) {
  const int64_t chunks = ldh / 8;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= m * chunks) return;
  const int64_t r = e / chunks, ch = e % chunks;
  const int64_t src = idx[r] * ldh + ch * 8, dst = r * ldh + ch * 8;
  *reinterpret_cast<uint4*>(Zhi + dst) = *reinterpret_cast<const uint4*>(Xhi + src);
  *reinterpret_cast<uint4*>(Zmid + dst) = *reinterpret_cast<const uint4*>(Xmid + src);
  *reinterpret_cast<uint4*>(Zlo + dst) = *reinterpret_cast<const uint4*>(Xlo + src);
}

// ---------------------------------------------------------------------------
// Masked Gram matrix: P[a][b] (+)= sum_p Kc[a][p] Kc[b][p] over 256 x 256
// upper-triangular tiles, Kc = hi + lo with all four plane products, so P
// is the Gram matrix of the stored values up to FP32 accumulation rounding
// (positive semidefinite to that level).  A tile belongs to a pair of CTAs
// (cta_group::2): each stages 128 rows of A and 128 of B, the even CTA issues
// the 256 x 256 MMAs for both, and each drains its own 128 rows.  Per 64
// points a CTA then loads 64 KB for 1,024 MMA cycles; a 128 x 128 tile per
// CTA loads as much for 512, which the path from L2 to the SM cannot carry.
// ns = 86,000, m = 2,048: 0.764 ms, 1.89 PFLOP/s, tensor pipe 96% of active
// cycles (128 x 128 tiles: 1.9 ms, 35%).  Warp 0: TMEM owner and TMA producer;
// warp 1: MMA issuer; warps 2-9: epilogue (warps w and w + 4 share a lane
// quarter and split the columns).
// ---------------------------------------------------------------------------
// 32 FP32 sums into a row of the partial pairs (the first time, as they are);
// cols: columns left in the matrix; vec: whole vectors fit the row's pitch
// (columns past the matrix are padding).
__device__ __forceinline__ void gram_put(float2* __restrict__ row, const float (&v)[32], int64_t cols,
                                         bool vec, bool first) {
  if (vec) {
    float4* r4 = reinterpret_cast<float4*>(row);
    if (first) {
#pragma unroll
      for (int j = 0; j < 16; ++j) r4[j] = make_float4(v[2 * j], 0.f, v[2 * j + 1], 0.f);
      return;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float4 o[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = r4[8 * h + j];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        pair_add(o[j].x, o[j].y, v[16 * h + 2 * j]);
        pair_add(o[j].z, o[j].w, v[16 * h + 2 * j + 1]);
        r4[8 * h + j] = o[j];
      }
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    if (j < cols) {
      float2 s = first ? make_float2(0.f, 0.f) : row[j];
      pair_add(s.x, s.y, v[j]);
      row[j] = s;
    }
  }
}

constexpr int GR_THREADS = 320;
constexpr int GR_STAGES = 3;
constexpr int GR_TILE = 256;
constexpr int GR_HALF = GR_TILE / 2;           // rows per CTA
constexpr int GR_PLANE_BYTES = GR_HALF * 128;
constexpr int GR_STAGE = 4 * GR_PLANE_BYTES;   // A hi, A lo, B hi, B lo
constexpr int GR_BAR_OFF = GR_STAGES * GR_STAGE;
constexpr int GR_SMEM = GR_BAR_OFF + 256 + 1024;
constexpr int64_t GR_CHUNKS_PER_SLICE = GRAM_SLICE / 64;

__global__ void __launch_bounds__(GR_THREADS, 1) gram_tc_pair_kernel(
    const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
    int64_t m, const int64_t* __restrict__ ns_dev, GramPlan plan, float2* __restrict__ part,
    int64_t ldp, int vec, WaitCtx wc) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + GR_BAR_OFF);
  uint64_t* empty = full + GR_STAGES;
  uint64_t* accf = empty + GR_STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  uint32_t* bad = tmem_slot + 1;   // [2]: a wait had given up before, as each CTA saw it
  Leave* leave = reinterpret_cast<Leave*>(bad + 2);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank();
  const int64_t pair = blockIdx.x >> 1;
  // upper-triangular tile (ta <= tb)
  const int64_t T = ceil_div(m, (int64_t)GR_TILE);
  int64_t rem = pair, ta = 0;
  while (rem >= T - ta) {
    rem -= T - ta;
    ++ta;
  }
  const int64_t tb = ta + rem;
  const bool diag = ta == tb;   // the B rows are the A rows
  const int64_t a0 = ta * GR_TILE + rank * GR_HALF, b0 = tb * GR_TILE + rank * GR_HALF;
  const int64_t ns = *ns_dev;
  if (plan.single(ns)) return;   // both CTAs; single CTAs take these points
  const int64_t per = gram_split_points(ns, plan.s_pair, kGramQuantumTc);
  const int64_t c_begin = min64(ceil_div(ns, (int64_t)64), (int64_t)blockIdx.y * (per / 64));
  const int64_t c_end = min64(ceil_div(ns, (int64_t)64), c_begin + per / 64);
  const int64_t nch = c_end - c_begin;
  if (blockIdx.y > 0 && nch == 0) return;   // both CTAs; the finish skips the empty splits
  const int64_t nslices = ceil_div(nch, GR_CHUNKS_PER_SLICE);
  constexpr uint32_t IDESC = idesc_bf16_f32(GR_TILE, GR_TILE);
  float2* P = part + (int64_t)blockIdx.y * ldp * ldp;

  if (tid == 0) {
    for (int s = 0; s < GR_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 2 * 8);   // one arrival per epilogue warp of the pair
    }
    mbar_init(drain, 32);
    *leave = Leave{0u, {0u, 0u}};
    fence_barrier_init();
    prefetch_tmap(&map_hi);
    prefetch_tmap(&map_lo);
  }
  __syncwarp();
  cluster_sync();   // both CTAs run, and their barriers are initialised
  if (tid == 0) {
    const uint32_t st = *(volatile int*)wc.st != 0 ? 1u : 0u;
    st_cluster(map_rank(&bad[rank], 0), st);
    st_cluster(map_rank(&bad[rank], 1), st);
  }
  __syncwarp();
  if (warp == 0) tmem_alloc_pair(tmem_slot, 2 * GR_TILE);
  fence_before_sync();
  cluster_sync();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  const bool live = bad[0] == 0 && bad[1] == 0;   // the same in both CTAs
  auto note = [&](bool ok) {   // every wait's outcome goes through this
    if (!ok) leave_word<true>(&leave->gave, 1u);
    return ok;
  };
  const uint32_t bytes = (diag ? 2u : 4u) * GR_PLANE_BYTES;   // a CTA's per stage

  if (live && warp == 0 && lane == 0) {
    // ---- TMA producer: both CTAs' loads complete on the even CTA's barrier
    int64_t issued = 0;
    bool ok = true;
    for (int64_t q = 0; q < nch; ++q) {
      const int s = (int)(q % GR_STAGES);
      const uint32_t ph = (uint32_t)((q / GR_STAGES) & 1);
      if (!(ok = note(mbar_wait_cluster<true>(&empty[s], ph ^ 1u, wc.st, 11, wc.lim)))) break;
      uint8_t* st = smem + s * GR_STAGE;
      const int x = (int)((c_begin + q) * 64);
      if (rank == 0) mbar_expect_tx(&full[s], 2 * bytes);
      const uint32_t bar = map_rank(&full[s], 0);
      tma_load_2d_pair(st, &map_hi, x, (int)a0, bar);
      tma_load_2d_pair(st + GR_PLANE_BYTES, &map_lo, x, (int)a0, bar);
      if (!diag) {
        tma_load_2d_pair(st + 2 * GR_PLANE_BYTES, &map_hi, x, (int)b0, bar);
        tma_load_2d_pair(st + 3 * GR_PLANE_BYTES, &map_lo, x, (int)b0, bar);
      }
      issued = q + 1;
    }
    // the last stages consumed: their copies and the MMAs' arrivals here are done
    for (int64_t q = (issued > GR_STAGES ? issued - GR_STAGES : 0); q < issued && ok; ++q)
      ok = note(mbar_wait_cluster<true>(&empty[q % GR_STAGES], (uint32_t)((q / GR_STAGES) & 1), wc.st, 12, wc.lim));
    leave_word<true>(&leave->left[rank], (uint32_t)issued);
  } else if (live && warp == 1 && lane == 0 && rank == 0) {
    // ---- MMA issuer
    bool ok = true;
    for (int64_t t = 0; t < nslices && ok; ++t) {
      const int acc = (int)(t & 1);
      const uint32_t use = (uint32_t)((t >> 1) & 1);
      if (!note(mbar_wait_cluster<false>(&acce[acc], use ^ 1u, wc.st, 13, wc.lim))) break;
      fence_after_sync();
      const uint32_t d = tmem + acc * GR_TILE;
      const int64_t q0 = t * GR_CHUNKS_PER_SLICE;
      const int64_t q1 = min64(nch, q0 + GR_CHUNKS_PER_SLICE);
      for (int64_t q = q0; q < q1; ++q) {
        const int s = (int)(q % GR_STAGES);
        const uint32_t ph = (uint32_t)((q / GR_STAGES) & 1);
        if (!note(mbar_wait(&full[s], ph, wc.st, 14, wc.lim))) {
          ok = false;
          break;
        }
        fence_after_sync();
        const uint32_t base = smem_u32(smem + s * GR_STAGE);
        const uint32_t a_hi = base, a_lo = base + GR_PLANE_BYTES;
        const uint32_t b_hi = diag ? a_hi : base + 2 * GR_PLANE_BYTES;
        const uint32_t b_lo = diag ? a_lo : base + 3 * GR_PLANE_BYTES;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t koff = k * 32;
          mma_bf16_pair<A_FILL>(d, desc_sw128(a_hi + koff), desc_sw128(b_hi + koff), IDESC,
                        (q != q0 || k != 0) ? 1u : 0u);
          mma_bf16_pair<A_LASTUSE>(d, desc_sw128(a_hi + koff), desc_sw128(b_lo + koff), IDESC, 1u);
          mma_bf16_pair<A_FILL>(d, desc_sw128(a_lo + koff), desc_sw128(b_hi + koff), IDESC, 1u);
          // lo x lo too: without it the sum is (hi + lo)^T (hi + lo) - lo^T lo,
          // indefinite in the null space of a short K_SJ
          mma_bf16_pair<A_LASTUSE>(d, desc_sw128(a_lo + koff), desc_sw128(b_lo + koff), IDESC, 1u);
        }
        mma_commit_pair(&empty[s]);
      }
      mma_commit_pair(&accf[acc]);
    }
  } else if (live && warp >= 2) {
    // ---- epilogue: TMEM lanes 32 * (warp % 4) .. + 31, half the columns
    const int quarter = warp & 3;
    const int64_t a = a0 + 32 * quarter + lane;
    const int64_t bc = tb * GR_TILE + (warp >= 6 ? GR_HALF : 0);
    if (nslices == 0) {
      if (a < m)
        for (int64_t b = bc; b < min64(m, bc + GR_HALF); ++b) P[a * ldp + b] = make_float2(0.f, 0.f);
    }
    for (int64_t t = 0; t < nslices; ++t) {
      const int acc = (int)(t & 1);
      const uint32_t use = (uint32_t)((t >> 1) & 1);
      // (all lanes or none: the reads of TMEM are the warp's)
      if (!__all_sync(~0u, note(mbar_wait_cluster<false>(&accf[acc], use, wc.st, 15, wc.lim)))) break;
      fence_after_sync();
      const uint32_t tbase = tmem + acc * GR_TILE + (warp >= 6 ? GR_HALF : 0) + ((uint32_t)(32 * quarter) << 16);
      for (int cc = 0; cc < GR_HALF / 32; ++cc) {
        const int64_t c0 = bc + cc * 32;
        if (c0 >= m) break;   // uniform
        float v[32];
        __syncwarp();
        tmem_ld32(tbase + cc * 32, v);
        if (a < m) gram_put(P + a * ldp + c0, v, m - c0, vec && c0 + 32 <= ldp, t == 0);
      }
      __syncwarp();
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_rank(&acce[acc], 0));
    }
  }
  fence_before_sync();
  __syncwarp();
  cluster_sync();   // no copy, MMA or arrival of the pair is outstanding, or
  if (*(volatile uint32_t*)&leave->gave) {
    settle<true, GR_STAGES>(full, drain, leave, bytes, rank, wc.st);
    cluster_sync();
  }
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc_pair(tmem, 2 * GR_TILE);
  }
}

// The same over 128 x 128 tiles of single CTAs, for as many points as one wave
// of such tiles takes in separate slices (GramPlan): a slice then takes 1,160
// cycles per 64 points, where a pair's 256 x 256 tile takes 2,048 on SMs that
// would otherwise idle (m = 256, ns = 8,000: 90 us against 148).
constexpr int GS_THREADS = 192;
constexpr int GS_STAGES = 3;
constexpr int GS_TILE = 128;
constexpr int GS_PLANE_BYTES = GS_TILE * 128;
constexpr int GS_STAGE = 4 * GS_PLANE_BYTES;   // A hi, A lo, B hi, B lo
constexpr int GS_BAR_OFF = GS_STAGES * GS_STAGE;
constexpr int GS_SMEM = GS_BAR_OFF + 256 + 1024;

__global__ void __launch_bounds__(GS_THREADS, 1) gram_tc_single_kernel(
    const __grid_constant__ CUtensorMap map_hi, const __grid_constant__ CUtensorMap map_lo,
    int64_t m, const int64_t* __restrict__ ns_dev, GramPlan plan, float2* __restrict__ part,
    int64_t ldp, int vec, WaitCtx wc) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + GS_BAR_OFF);
  uint64_t* empty = full + GS_STAGES;
  uint64_t* accf = empty + GS_STAGES;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  Leave* leave = reinterpret_cast<Leave*>(tmem_slot + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (__syncthreads_or(tid == 0 && *(volatile int*)wc.st != 0)) return;
  // upper-triangular tile (ta <= tb)
  const int64_t T = ceil_div(m, (int64_t)GS_TILE);
  int64_t rem = blockIdx.x, ta = 0;
  while (rem >= T - ta) {
    rem -= T - ta;
    ++ta;
  }
  const int64_t tb = ta + rem;
  const int64_t a0 = ta * GS_TILE, b0 = tb * GS_TILE;
  const int64_t ns = *ns_dev;
  if (!plan.single(ns)) return;   // the pairs take these points
  const int64_t per = gram_split_points(ns, plan.s_single, kGramQuantumTc);
  const int64_t chunks = ceil_div(ns, (int64_t)64);
  const int64_t c_begin = min64(chunks, (int64_t)blockIdx.y * (per / 64));
  const int64_t c_end = min64(chunks, c_begin + per / 64);
  const int64_t nch = c_end - c_begin;
  if (blockIdx.y > 0 && nch == 0) return;   // the finish skips the empty splits
  const int64_t nslices = ceil_div(nch, GR_CHUNKS_PER_SLICE);
  constexpr uint32_t IDESC = idesc_bf16_f32(GS_TILE, GS_TILE);
  float2* P = part + (int64_t)blockIdx.y * ldp * ldp;

  if (tid == 0) {
    for (int s = 0; s < GS_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 128);
    }
    mbar_init(drain, 32);
    *leave = Leave{0u, {0u, 0u}};
    fence_barrier_init();
    prefetch_tmap(&map_hi);
    prefetch_tmap(&map_lo);
  }
  if (warp == 0) tmem_alloc(tmem_slot, 256);
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  auto note = [&](bool ok) {   // every wait's outcome goes through this
    if (!ok) leave_word<false>(&leave->gave, 1u);
    return ok;
  };

  if (warp == 0 && lane == 0) {
    // ---- TMA producer
    int64_t issued = 0;
    bool ok = true;
    for (int64_t q = 0; q < nch; ++q) {
      const int s = (int)(q % GS_STAGES);
      const uint32_t ph = (uint32_t)((q / GS_STAGES) & 1);
      if (!(ok = note(mbar_wait(&empty[s], ph ^ 1u, wc.st, 11, wc.lim)))) break;
      uint8_t* st = smem + s * GS_STAGE;
      const int x = (int)((c_begin + q) * 64);
      mbar_expect_tx(&full[s], GS_STAGE);
      tma_load_2d(st, &map_hi, x, (int)a0, &full[s]);
      tma_load_2d(st + GS_PLANE_BYTES, &map_lo, x, (int)a0, &full[s]);
      tma_load_2d(st + 2 * GS_PLANE_BYTES, &map_hi, x, (int)b0, &full[s]);
      tma_load_2d(st + 3 * GS_PLANE_BYTES, &map_lo, x, (int)b0, &full[s]);
      issued = q + 1;
    }
    // the last stages consumed: their copies and the MMAs' arrivals here are done
    for (int64_t q = (issued > GS_STAGES ? issued - GS_STAGES : 0); q < issued && ok; ++q)
      ok = note(mbar_wait(&empty[q % GS_STAGES], (uint32_t)((q / GS_STAGES) & 1), wc.st, 12, wc.lim));
    leave_word<false>(&leave->left[0], (uint32_t)issued);
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer
    bool ok = true;
    for (int64_t t = 0; t < nslices && ok; ++t) {
      const int acc = (int)(t & 1);
      const uint32_t use = (uint32_t)((t >> 1) & 1);
      if (!note(mbar_wait(&acce[acc], use ^ 1u, wc.st, 13, wc.lim))) break;
      fence_after_sync();
      const uint32_t d = tmem + acc * GS_TILE;
      const int64_t q0 = t * GR_CHUNKS_PER_SLICE;
      const int64_t q1 = min64(nch, q0 + GR_CHUNKS_PER_SLICE);
      for (int64_t q = q0; q < q1; ++q) {
        const int s = (int)(q % GS_STAGES);
        const uint32_t ph = (uint32_t)((q / GS_STAGES) & 1);
        if (!note(mbar_wait(&full[s], ph, wc.st, 14, wc.lim))) {
          ok = false;
          break;
        }
        fence_after_sync();
        const uint32_t base = smem_u32(smem + s * GS_STAGE);
        const uint32_t a_hi = base, a_lo = base + GS_PLANE_BYTES;
        const uint32_t b_hi = base + 2 * GS_PLANE_BYTES, b_lo = base + 3 * GS_PLANE_BYTES;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t koff = k * 32;
          mma_bf16<A_FILL>(d, desc_sw128(a_hi + koff), desc_sw128(b_hi + koff), IDESC,
                   (q != q0 || k != 0) ? 1u : 0u);
          mma_bf16<A_LASTUSE>(d, desc_sw128(a_hi + koff), desc_sw128(b_lo + koff), IDESC, 1u);
          mma_bf16<A_FILL>(d, desc_sw128(a_lo + koff), desc_sw128(b_hi + koff), IDESC, 1u);
          // lo x lo too: without it the sum is (hi + lo)^T (hi + lo) - lo^T lo,
          // indefinite in the null space of a short K_SJ
          mma_bf16<A_LASTUSE>(d, desc_sw128(a_lo + koff), desc_sw128(b_lo + koff), IDESC, 1u);
        }
        mma_commit(&empty[s]);
      }
      mma_commit(&accf[acc]);
    }
  } else if (warp >= 2) {
    // ---- epilogue: TMEM lanes 32 * (warp % 4) .. + 31
    const int quarter = warp & 3;
    const int64_t a = a0 + 32 * quarter + lane;
    if (nslices == 0) {
      if (a < m)
        for (int64_t b = b0; b < min64(m, b0 + GS_TILE); ++b) P[a * ldp + b] = make_float2(0.f, 0.f);
    }
    for (int64_t t = 0; t < nslices; ++t) {
      const int acc = (int)(t & 1);
      const uint32_t use = (uint32_t)((t >> 1) & 1);
      // (all lanes or none: the reads of TMEM are the warp's)
      if (!__all_sync(~0u, note(mbar_wait(&accf[acc], use, wc.st, 15, wc.lim)))) break;
      fence_after_sync();
      const uint32_t tbase = tmem + acc * GS_TILE + ((uint32_t)(32 * quarter) << 16);
      for (int cc = 0; cc < GS_TILE / 32; ++cc) {
        const int64_t c0 = b0 + cc * 32;
        if (c0 >= m) break;   // uniform
        float v[32];
        __syncwarp();
        tmem_ld32(tbase + cc * 32, v);
        if (a < m) gram_put(P + a * ldp + c0, v, m - c0, vec && c0 + 32 <= ldp, t == 0);
      }
      __syncwarp();
      fence_before_sync();
      mbar_arrive(&acce[acc]);
    }
  }
  fence_before_sync();
  __syncthreads();
  if (*(volatile uint32_t*)&leave->gave) {
    settle<false, GS_STAGES>(full, drain, leave, GS_STAGE, 0, wc.st);
    __syncthreads();
  }
  if (warp == 0) {
    __syncwarp();
    fence_after_sync();
    tmem_dealloc(tmem, 256);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  // thread-safe one-time lookup of the driver's tensor-map encoder
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
    return (PFN_cuTensorMapEncodeTiled_v12000) nullptr;
  }();
  return fn;
}

// 2-D map over rows x inner (row pitch `pitch_elems`) of BF16, boxes of
// 64 elements (128 bytes, 128-byte swizzle) x box_rows, zero fill outside the
// tensor.
int make_map(CUtensorMap* map, const void* base, int64_t inner, int64_t rows, int64_t pitch_elems,
             uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn) return set_error(SPSVM_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (pitch_elems * 2) % 16)
    return set_error(SPSVM_ERR_ARG, "tensor map: base or pitch not 16-byte aligned");
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)(rows > 0 ? rows : 1)};
  cuuint64_t strides[1] = {(cuuint64_t)(pitch_elems * 2)};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(SPSVM_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return SPSVM_OK;
}

// What the modes read and write besides the products of rows A by columns B.
struct KbArgs {
  const uint16_t *a_hi, *a_mid, *a_lo, *b_hi, *b_mid, *b_lo;
  int64_t ldh, nrows, ncols;
  const float *colnorm, *rownorm;
  const int64_t* idx;                 // of the columns' (STORE) or rows' (SCORE) norms
  float gamma;
  float* out;                         // STORE: the first column's row
  int64_t ld;
  const float *y, *o;                 // SCORE
  float4* part;
  int64_t* parts;                     // receives the number of partial sums
  const double* beta;                 // DECIDE
  float* dpart;
  int64_t ldp;
};

template <int MODE, bool PAIR, int N, int RA = PK_M>
int launch_kb_as(const KbArgs& a, cudaStream_t s) {
  using TL = Kb<PAIR, N, RA>;
  CUtensorMap mah, mam, mal, mbh, mbm, mbl;
  // few rows: only theirs are loaded
  const int box_a = PAIR || a.nrows >= RA ? RA : (int)round_up(a.nrows, (int64_t)8);
  SPSVM_TRY(make_map(&mah, a.a_hi, a.ldh, a.nrows, a.ldh, box_a));
  SPSVM_TRY(make_map(&mam, a.a_mid, a.ldh, a.nrows, a.ldh, box_a));
  SPSVM_TRY(make_map(&mal, a.a_lo, a.ldh, a.nrows, a.ldh, box_a));
  SPSVM_TRY(make_map(&mbh, a.b_hi, a.ldh, a.ncols, a.ldh, TL::ROWS_B));
  SPSVM_TRY(make_map(&mbm, a.b_mid, a.ldh, a.ncols, a.ldh, TL::ROWS_B));
  SPSVM_TRY(make_map(&mbl, a.b_lo, a.ldh, a.ncols, a.ldh, TL::ROWS_B));
  auto kern = kblock_tc_kernel<MODE, PAIR, N, RA>;
  SPSVM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TL::SMEM));
  constexpr int W = TL::CTAS;
  const int64_t tiles = ceil_div(a.nrows, (int64_t)TL::M) * ceil_div(a.ncols, (int64_t)N);
  WaitCtx wc;
  SPSVM_TRY(wait_ctx(s, &wc));
  cudaLaunchConfig_t cfg{};
  const int64_t units = max64(1, min64(tiles, (int64_t)sm_count() / W));
  // sums per CTA or pair, unless those outnumber the tiles of points
  const int64_t col_tiles = ceil_div(a.ncols, (int64_t)N);
  const int per_tile = MODE == KB_SCORE && units > col_tiles;
  if (MODE == KB_SCORE) *a.parts = per_tile ? col_tiles : units;
  cfg.gridDim = dim3((unsigned)(W * units));
  cfg.blockDim = dim3(TL::THREADS);
  cfg.dynamicSmemBytes = TL::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = W;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  SPSVM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, mah, mam, mal, mbh, mbm, mbl, a.ldh, a.ncols, a.nrows, box_a,
                                    a.colnorm, a.rownorm, a.idx, a.gamma, a.out, a.ld, a.y, a.o, a.part, per_tile,
                                    a.beta, a.dpart, a.ldp, wc));
  SPSVM_LAUNCH_CHECK();
  return SPSVM_OK;
}

// Single CTAs where their tiles cost less than a pair's, which take 256 rows and
// a microsecond more to start:
//   * up to 128 rows, or one wave of tiles (3,000 points by 200 basis rows, d =
//     128: 8.8 us against 10.3);
//   * three or five blocks of 128 rows, of which pairs would compute four or six
//     (300 candidates, d = 20: n = 500,000 154 us against 176, n = 20,000 17.5
//     against 19.3; 600: 205 against 270; seven blocks, d = 128 115 against 104);
//   * a few waves at small d, where the MMAs are not the bound (200 candidates, n =
//     20,000, d = 20: 15.3 us against 15.8; kernel block of 12,000 points by 512
//     rows, d = 30: 12.0 against 13.4), and every kernel block that its stores
//     bound (500,000 by 512, d = 54: 210 us against 214).
// Else pairs (256 candidates, n = 500,000, d = 128: 130 us against 143; 100,000
// queries by 4,096 rows: 418 against 454).  Scores of up to 64 candidates stage 64
// rows, which leaves more of the ring to the points.
template <int MODE>
int launch_kb(const KbArgs& a, cudaStream_t s) {
  constexpr int NARROW = MODE == KB_SCORE ? 128 : 64;   // (score columns are the points)
  const bool narrow = a.ncols <= NARROW;
  const int64_t blocks = ceil_div(a.nrows, (int64_t)PK_M);
  const int64_t tiles = blocks * ceil_div(a.ncols, (int64_t)(narrow ? NARROW : 128));
  constexpr bool STORE = MODE == KB_STORE_F32;
  const int waves = a.ldh == 64 || (STORE && a.ldh == 128) ? 4 : 1;
  if (MODE == KB_SCORE && a.nrows <= 64) return launch_kb_as<MODE, false, 128, MODE == KB_SCORE ? 64 : PK_M>(a, s);
  if (blocks == 1 || blocks == 3 || blocks == 5 || tiles <= waves * (int64_t)sm_count() || (STORE && a.ldh == 64))
    return narrow ? launch_kb_as<MODE, false, NARROW>(a, s) : launch_kb_as<MODE, false, 128>(a, s);
  return narrow ? launch_kb_as<MODE, true, NARROW>(a, s) : launch_kb_as<MODE, true, 128>(a, s);
}

}  // namespace

size_t kernel_block_tc_scratch(int64_t m, int64_t ldh) {
  return (size_t)(round_up(m, (int64_t)PK_M) * ldh * 6);   // three BF16 planes of the rows
}

namespace {

// The planes of the m points idx, gathered into zbuf.
int gather_rows(const spsvm_points* p, const int64_t* idx, int32_t m, void* zbuf, size_t zbytes,
                cudaStream_t s, const uint16_t* (&z)[3]) {
  if (!zbuf || zbytes < kernel_block_tc_scratch(m, p->ldh))
    return set_error(SPSVM_ERR_OOM, "BF16SPLIT kernel block: scratch too small for the basis planes");
  uint16_t* zhi = static_cast<uint16_t*>(zbuf);
  uint16_t* zmid = zhi + m * p->ldh;
  uint16_t* zlo = zmid + m * p->ldh;
  gather_rows_bf16<<<(unsigned)ceil_div(m * (p->ldh / 8), (int64_t)256), 256, 0, s>>>(
      p->hi, p->mid, p->lo, p->ldh, idx, m, zhi, zmid, zlo);
  SPSVM_LAUNCH_CHECK();
  z[0] = zhi;
  z[1] = zmid;
  z[2] = zlo;
  return SPSVM_OK;
}

}  // namespace

bool tc_available() { return encode_fn() != nullptr; }

int launch_kernel_block_tc(const spsvm_points* p, const int64_t* idx, int32_t m, float gamma,
                           spsvm_kmat* out, int64_t row0, void* scratch, size_t scratch_bytes,
                           cudaStream_t s) {
  if (m == 0 || p->n == 0) return SPSVM_OK;
  if (out->format != SPSVM_FP32 || (out->ld % 8) != 0)
    return set_error(SPSVM_ERR_ARG, "BF16SPLIT kernel block: stores FP32 (ld %% 8 == 0)");
  const uint16_t* z[3];
  SPSVM_TRY(gather_rows(p, idx, m, scratch, scratch_bytes, s, z));
  KbArgs a{p->hi, p->mid, p->lo, z[0], z[1], z[2], p->ldh, p->n, m, p->norms, p->norms, idx, gamma};
  a.out = static_cast<float*>(out->data) + row0 * out->ld;
  a.ld = out->ld;
  return launch_kb<KB_STORE_F32>(a, s);
}

// Partial sums per candidate at most.
int64_t score_tc_parts(int64_t n) { return ceil_div(n, (int64_t)128); }

int launch_score_tc(const spsvm_points* p, const float* y, const float* o, const int64_t* idx,
                    int32_t kappa, float gamma, float4* part, int64_t* parts, void* zbuf,
                    size_t zbytes, cudaStream_t s) {
  const uint16_t* z[3];
  SPSVM_TRY(gather_rows(p, idx, kappa, zbuf, zbytes, s, z));
  KbArgs a{z[0], z[1], z[2], p->hi, p->mid, p->lo, p->ldh, kappa, p->n, p->norms, p->norms, idx, gamma};
  a.y = y;
  a.o = o;
  a.part = part;
  a.parts = parts;
  return launch_kb<KB_SCORE>(a, s);
}

int64_t decision_tc_parts(int64_t m) { return ceil_div(m, (int64_t)PK_WP); }

int launch_decision_tc(const spsvm_points* q, const void* zplanes, size_t zbytes, int64_t m,
                       const float* znorm, const double* beta, float gamma, float* dpart,
                       int64_t ldp, cudaStream_t s) {
  if (m == 0 || q->n == 0) return SPSVM_OK;
  if (!zplanes || zbytes < (size_t)(m * q->ldh * 6))
    return set_error(SPSVM_ERR_OOM, "BF16SPLIT decision: scratch too small for the basis planes");
  const uint16_t* z = static_cast<const uint16_t*>(zplanes);
  KbArgs a{q->hi, q->mid, q->lo, z, z + m * q->ldh, z + 2 * m * q->ldh, q->ldh, q->n, m, znorm, q->norms, nullptr, gamma};
  a.beta = beta;
  a.dpart = dpart;
  a.ldp = ldp;
  return launch_kb<KB_DECIDE>(a, s);
}

GramPlan gram_tc_plan(int64_t m, int64_t ns_max) {
  const int64_t sms = sm_count();
  const int64_t T1 = ceil_div(m, (int64_t)GS_TILE), T2 = ceil_div(m, (int64_t)GR_TILE);
  GramPlan p;
  p.s_single = min64(sms / max64(1, T1 * (T1 + 1) / 2), ceil_div(ns_max, kGramQuantumTc));
  p.s_pair = gram_splits(max64(1, T2 * (T2 + 1) / 2), max64(1, sms / 2), 1, 0.9, ns_max, kGramQuantumTc);
  return p;
}

// ns_hint: the number of active points when the caller knows it (only the
// kernel it selects is launched), else -1 (both are, unless ns_max decides;
// the one not selected returns at once).
int launch_gram_tc(const spsvm_kmat* Kc, const int64_t* ns_dev, int64_t ns_max, int64_t ns_hint,
                   int64_t m, float2* part, int64_t ldp, const GramPlan& plan, cudaStream_t s) {
  const uint16_t* hi = static_cast<const uint16_t*>(Kc->data);
  const uint16_t* lo = hi + Kc->plane;
  const int vec = (reinterpret_cast<uintptr_t>(part) & 15) == 0;
  CUtensorMap mh, ml;   // boxes of 128 rows in both kernels
  static_assert(GS_TILE == GR_HALF, "one tensor map for both kernels");
  SPSVM_TRY(make_map(&mh, hi, Kc->ld, m, Kc->ld, GR_HALF));
  SPSVM_TRY(make_map(&ml, lo, Kc->ld, m, Kc->ld, GR_HALF));
  WaitCtx wc;
  SPSVM_TRY(wait_ctx(s, &wc));
  const bool known = ns_hint >= 0;
  if (known ? plan.single(ns_hint) : plan.s_single > 0) {
    SPSVM_CUDA_TRY(cudaFuncSetAttribute(gram_tc_single_kernel,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, GS_SMEM));
    const int64_t T = ceil_div(m, (int64_t)GS_TILE);
    const dim3 grid((unsigned)(T * (T + 1) / 2), (unsigned)plan.s_single);
    gram_tc_single_kernel<<<grid, GS_THREADS, GS_SMEM, s>>>(mh, ml, m, ns_dev, plan, part, ldp, vec, wc);
    SPSVM_LAUNCH_CHECK();
  }
  if (known ? !plan.single(ns_hint) : !plan.single(ns_max)) {
    SPSVM_CUDA_TRY(cudaFuncSetAttribute(gram_tc_pair_kernel,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, GR_SMEM));
    const int64_t T = ceil_div(m, (int64_t)GR_TILE);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(T * (T + 1)), (unsigned)plan.s_pair);   // two CTAs per tile
    cfg.blockDim = dim3(GR_THREADS);
    cfg.dynamicSmemBytes = GR_SMEM;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    SPSVM_CUDA_TRY(cudaLaunchKernelEx(&cfg, gram_tc_pair_kernel, mh, ml, m, ns_dev, plan, part, ldp, vec, wc));
    SPSVM_LAUNCH_CHECK();
  }
  return SPSVM_OK;
}

}  // namespace spsvm
