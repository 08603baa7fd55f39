// Step a2 (mixed precision): the Cholesky's dense contractions on the fifth-
// generation tensor cores (tcgen05.mma, TMEM accumulators, TMA-staged tiles).
//
// The MP variant of Section II-A (Fig. 1(d)) keeps the tiles next to the
// diagonal in double precision and lowers the precision of the rest.  Here
// every operand is stored in FP64 and each product C -= A B^T runs as one of:
//
//  * T3 (off-band tiles): A = A_hi + A_lo with A_hi = tf32(A), A_lo = tf32(A - A_hi)
//    (both rounded to nearest), C -= A_hi B_hi^T + A_hi B_lo^T + A_lo B_hi^T,
//    accumulated in FP32 in TMEM (~22 significant bits per product).
//  * OZ (band tiles, where the Schur complement cancels most): each row is scaled
//    by a power of two 2^e_r so that |a| <= 1 and cut into S = 5 signed 7-bit
//    integer digits held exactly in BF16, a = 2^e_r sum_s d_s 2^{-7(s+1)}
//    (|d_0| <= 128, |d_s| <= 64 after it).  A group g = s + t sums at most two
//    products with a leading digit (<= 2^13, or 2^14 for g = 0) and g - 1 others
//    (<= 2^12), at most 7 * 2^12 per k; with K <= 512 every partial sum stays
//    below 2^24, so FP32 accumulation in TMEM is exact.  The 15 products with g <= 4 go to five accumulators that
//    the epilogue combines in FP64 (error ~2^-35 of the row maxima).
//
// Both kernels are persistent and warp-specialised: warp 0 issues TMA loads,
// warp 1 owns TMEM and issues tcgen05.mma from one thread, warps 2-5 drain the
// accumulators into the FP64 matrix.  Every wait is bounded; on time-out the
// CTA records EXA_ERR_TIMEOUT, drains its in-flight copies, frees TMEM and exits.
#include <type_traits>
#include <cuda.h>
#include <math.h>

#include <climits>

#include "ctx.cuh"
#include "gemm_tc.cuh"
#include "tc_common.cuh"

namespace exa {

using namespace tc;

__device__ __forceinline__ void tile_tri_decode(long long b, int& ti, int& tj) {
  long long t = (long long)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
  while (t * (t + 1) / 2 > b) --t;
  while ((t + 1) * (t + 2) / 2 <= b) ++t;
  ti = (int)t;
  tj = (int)(b - t * (t + 1) / 2);
}

// Output-tile enumeration shared by all roles of a CTA.  Returns false if the
// tile is to be skipped.  (bi, bj) are tile indices in units of (TM, TN).
template <int TM, int TN>
__device__ __forceinline__ bool decode_tile(const GemmArgs& g, long long t, int& bi, int& bj) {
  if (g.enum_mode == kEnumFull) {
    bi = (int)(t / g.nt);
    bj = (int)(t % g.nt);
    return true;
  }
  if (g.enum_mode == kEnumLowerOffBand) {
    // TM == TN == 128, g.nt tile rows, band measured in panel-wide tiles.  Tiles are
    // taken in supertiles of kSuper x kSuper (lower-triangle order of supertiles,
    // row-major inside), so the CTAs of one wave share a few operand row blocks
    // in L2 instead of streaming a different B row block each from DRAM.
    constexpr int kSuper = kRasterSuper;
    const long long sidx = t / (kSuper * kSuper);
    const int loc = (int)(t % (kSuper * kSuper));
    int SI, SJ;
    tile_tri_decode(sidx, SI, SJ);
    bi = SI * kSuper + loc / kSuper;
    bj = SJ * kSuper + loc % kSuper;
    if (bi >= g.nt || bj > bi) return false;
    const int per = g.panel / 128;
    return (bi / per - bj / per) > g.band;
  }
  // kEnumBand: pairs (I, J) of panel-wide tiles with 0 <= I - J <= band, each split in
  // (panel/TM) x (panel/TN) sub-tiles
  const int SI = g.panel / TM, SJ = g.panel / TN;
  const long long pair = t / (SI * SJ);
  const int sub = (int)(t % (SI * SJ));
  const int b = g.band;
  const long long head = (long long)b * (b + 1) / 2;
  int I, J;
  if (pair < head) {
    tile_tri_decode(pair, I, J);
  } else {
    I = b + (int)((pair - head) / (b + 1));
    J = I - b + (int)((pair - head) % (b + 1));
  }
  bi = I * SI + sub / SJ;
  bj = J * SJ + sub % SJ;
  // skip sub-tiles strictly above the diagonal
  return (long long)bj * TN <= (long long)bi * TM + TM - 1;
}

// T3 (128 x 128 tiles): operand rows and output origin of tile t, from the enumeration or the
// launch's task list.  Returns false if the tile is to be skipped.
struct T3Tile {
  int ya, yb;
  double* C;
  int64_t ldc;
  bool diag;
  int chunks;  // 32-column steps of the reduction
  int shift;   // second operand: rows below ya, yb
};
__device__ __forceinline__ bool t3_tile(const GemmArgs& g, long long t, T3Tile& o) {
  o.chunks = (g.K + g.K2) / 32;
  o.shift = 0;
  if (g.enum_mode == kEnumTasks) {
    const TcTask tk = g.tasks[t];
    o.ya = tk.a_row;
    o.yb = tk.b_row;
    o.C = tk.C;
    o.ldc = tk.ldc;
    o.diag = tk.lower != 0;
    o.shift = tk.shift;
    return true;
  }
  int bi, bj;
  if (!decode_tile<128, 128>(g, t, bi, bj)) return false;
  o.ya = g.a_row0 + bi * 128;
  o.yb = g.b_row0 + bj * 128;
  o.C = g.C + (g.c_row0 + (int64_t)bi * 128) + (g.c_col0 + (int64_t)bj * 128) * g.ldc;
  o.ldc = g.ldc;
  o.diag = g.lower_mask && (bi == bj);
  if (g.tri) o.chunks = min(o.chunks, (bj + 1) * 4);
  return true;
}

// Far 128 x 128 tiles of the single-CTA kernel: the same test as the pair kernel's far tiles,
// on the 256-row block exponents of the two operand row blocks (never in task mode).
__device__ __forceinline__ bool far_t3(const GemmArgs& g, const T3Tile& tl) {
  if (g.enum_mode == kEnumTasks || g.far_thr == INT_MIN || !g.ea_blk || !g.eb_blk) return false;
  return (long long)g.ea_blk[tl.ya / 256] + (long long)g.eb_blk[tl.yb / 256] <= (long long)g.far_thr;
}

__device__ __forceinline__ void record_timeout(DevStatus* st, int site) {
  if (atomicExch(&st->timeout, 1) == 0) st->timeout_where = site;
}

// ===========================================================================
// T3 kernel: tile 128 x 128, K chunks of 32 FP32 (TF32) values, 3 stages.
// ===========================================================================
constexpr int kEpiThreads = 256;                 // 8 epilogue warps
constexpr int kGemmThreads = 64 + kEpiThreads;   // + TMA producer warp + MMA warp

namespace t3 {
constexpr int TM = 128, TN = 128, KC = 32, STAGES = 3;
constexpr int OP_BYTES = TM * KC * 4;           // 16 KB per operand tile
constexpr int STAGE_BYTES = 4 * OP_BYTES;       // A_hi, A_lo, B_hi, B_lo
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr uint32_t IDESC = idesc(kFmtTF32, TM, TN);
constexpr int TMEM_COLS = 512;                  // 2 accumulator buffers x 128 columns, for each operand pair
constexpr int kThreads = 64 + 2 * kEpiThreads;  // eight epilogue warps for each accumulator
}  // namespace t3

__global__ void __launch_bounds__(t3::kThreads)
    gemm_t3_kernel(const __grid_constant__ CUtensorMap tA_hi, const __grid_constant__ CUtensorMap tA_lo,
                   const __grid_constant__ CUtensorMap tB_hi, const __grid_constant__ CUtensorMap tB_lo,
                   const __grid_constant__ CUtensorMap tS_hi, const __grid_constant__ CUtensorMap tS_lo,
                   const __grid_constant__ GemmArgs g) {
  using namespace t3;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accfull = empty + STAGES;
  uint64_t* accempty = accfull + 2;
  uint32_t* tmem_slot = (uint32_t*)(accempty + 2);
  volatile int* abort = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], kEpiThreads);
    }
    *abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, TMEM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const int kc1 = g.K / KC;  // chunks of the first operand pair

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    const uint64_t pol = l2_evict_last_policy();
    prefetch_tmap(&tA_hi);
    prefetch_tmap(&tA_lo);
    prefetch_tmap(&tB_hi);
    prefetch_tmap(&tB_lo);
    int stage = 0;
    uint32_t phase = 0;
    int last_par[STAGES];
    for (int s = 0; s < STAGES; ++s) last_par[s] = -1;
    for (long long t = blockIdx.x; t < g.ntiles && !*abort; t += gridDim.x) {
      T3Tile tl;
      if (!t3_tile(g, t, tl)) continue;
      const int ya = tl.ya, yb = tl.yb;
      const bool one = far_t3(g, tl);  // far tile: the hi halves only
      for (int kc = 0; kc < tl.chunks; ++kc) {
        if (!mbar_wait(&empty[stage], phase ^ 1, abort)) {
          *abort = 1;
          record_timeout(g.st, 11);
          break;
        }
        uint8_t* sb = smem + stage * STAGE_BYTES;
        mbar_expect_tx(&full[stage], one ? 2 * OP_BYTES : STAGE_BYTES);
        if (kc < kc1) {
          tma_load_2d_hint(sb, &tA_hi, &full[stage], kc * KC, ya, pol);
          tma_load_2d_hint(sb + 2 * OP_BYTES, &tB_hi, &full[stage], kc * KC, yb, pol);
          if (!one) {
            tma_load_2d_hint(sb + OP_BYTES, &tA_lo, &full[stage], kc * KC, ya, pol);
            tma_load_2d_hint(sb + 3 * OP_BYTES, &tB_lo, &full[stage], kc * KC, yb, pol);
          }
        } else {
          const int kx = (kc - kc1) * KC;
          tma_load_2d_hint(sb, &tS_hi, &full[stage], kx, ya - tl.shift, pol);
          tma_load_2d_hint(sb + 2 * OP_BYTES, &tS_hi, &full[stage], kx, yb - tl.shift, pol);
          if (!one) {
            tma_load_2d_hint(sb + OP_BYTES, &tS_lo, &full[stage], kx, ya - tl.shift, pol);
            tma_load_2d_hint(sb + 3 * OP_BYTES, &tS_lo, &full[stage], kx, yb - tl.shift, pol);
          }
        }
        last_par[stage] = (int)phase;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    if (*abort) {  // let every copy this thread issued land before the CTA exits
      for (int s = 0; s < STAGES; ++s)
        if (last_par[s] >= 0) {
          volatile int never = 0;
          mbar_wait(&full[s], (uint32_t)last_par[s], &never);
        }
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    int stage = 0;
    uint32_t phase = 0;
    int it = 0;
    for (long long t = blockIdx.x; t < g.ntiles && !*abort; t += gridDim.x) {
      T3Tile tl;
      if (!t3_tile(g, t, tl)) continue;
      const int b = it & 1;
      const uint32_t ap = (it >> 1) & 1;
      if (!mbar_wait(&accempty[b], ap ^ 1, abort)) {
        *abort = 1;
        record_timeout(g.st, 12);
        break;
      }
      fence_after();
      const bool one = far_t3(g, tl);
      bool ok = true;
      for (int kc = 0; kc < tl.chunks; ++kc) {
        if (!mbar_wait(&full[stage], phase, abort)) {
          *abort = 1;
          record_timeout(g.st, 13);
          ok = false;
          break;
        }
        fence_after();
        const uint32_t sb = smem_u32(smem + stage * STAGE_BYTES);
        const uint64_t ahi = sdesc_sw128(sb), alo = sdesc_sw128(sb + OP_BYTES);
        const uint64_t bhi = sdesc_sw128(sb + 2 * OP_BYTES), blo = sdesc_sw128(sb + 3 * OP_BYTES);
        const uint32_t d = tmem + (kc < kc1 ? 0 : 2 * TN) + b * TN;
        const bool start = kc == 0 || kc == kc1;
#pragma unroll
        for (int kk = 0; kk < KC / 8; ++kk) {  // K = 8 per instruction: advance 32 bytes
          const uint64_t o = (uint64_t)(kk * 2);
          mma_tf32(d, ahi + o, bhi + o, IDESC, start && kk == 0 ? 0u : 1u);
          if (!one) {
            mma_tf32(d, ahi + o, blo + o, IDESC, 1u);
            mma_tf32(d, alo + o, bhi + o, IDESC, 1u);
          }
        }
        mma_commit(&empty[stage]);
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (!ok) break;
      mma_commit(&accfull[b]);
      ++it;
    }
  } else if (warp >= 2) {
    // ---------------- epilogue: TMEM -> FP64 C ----------------
    // Two groups of 8 warps take the tiles in turn, one accumulator each: while one waits for C or stores it, the other
    // subtracts (the three phases of one group, 64 KB read and written and 16,384 FP64 additions an SM, took 22,000
    // cycles a tile one after another, the memory alone 11,000).  Warp w drains TMEM lanes 32*(w%4).. (its row quarter)
    // and one column half.
    const int quad = warp & 3;
    const int b = (warp - 2) >> 3, half = ((warp - 2) >> 2) & 1;
    const int r = quad * 32 + lane;
    int it = 0;
    for (long long t = blockIdx.x; t < g.ntiles && !*abort; t += gridDim.x) {
      T3Tile tl;
      if (!t3_tile(g, t, tl)) continue;
      if ((it++ & 1) != b) continue;
      const uint32_t ap = ((it - 1) >> 1) & 1;
      const bool diag = tl.diag;
      const int64_t ldc = tl.ldc;
      double* cp = tl.C + r;
      if (!g.store) {  // this warp's lines into L2 while the products run
#pragma unroll
        for (int l = 0; l < 4; ++l)
          prefetch_l2(tl.C + quad * 32 + 16 * (lane & 1) + (int64_t)(half * 64 + l * 16 + (lane >> 1)) * ldc);
      }
      if (!mbar_wait(&accfull[b], ap, abort)) {
        *abort = 1;
        record_timeout(g.st, 14);
        break;
      }
      fence_after();
#pragma unroll 1
      for (int h4 = 0; h4 < 4; ++h4) {
        const int cb = half * 64 + h4 * 16;
        double cv[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) cv[j] = g.store ? 0.0 : __ldcs(cp + (int64_t)(cb + j) * ldc);
        uint32_t acc[16];
        const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + b * TN + cb;
        tmem_ld16(ta, acc);
        tmem_ld_wait();
        if (g.K2 > 0) {
#pragma unroll
          for (int j = 0; j < 16; ++j) cv[j] -= f32_bits_to_f64(acc[j]);
          tmem_ld16(ta + 2 * TN, acc);
          tmem_ld_wait();
        }
        if (h4 == 3) {
          fence_before();
          mbar_arrive(&accempty[b]);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int cc = cb + j;
          if (diag && cc > r) continue;
          const double v = f32_bits_to_f64(acc[j]);
          __stcs(cp + (int64_t)cc * ldc, g.store ? v : cv[j] - v);
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ===========================================================================
// T3 on CTA pairs: a 256 x 256 output tile per cluster of two CTAs.  Each CTA
// stages its 128 rows of A and its 128 rows of B (TF32 halves); the leader's
// tcgen05.mma.cta_group::2 (M = N = 256) reads both CTAs' stages, so every
// staged byte feeds twice the products of the single-CTA kernel.  Each CTA's
// TMEM receives its own 128 rows x 256 columns; both epilogues drain their own.
// Barriers: full[] lives in the leader (both CTAs' TMA loads complete on it,
// the leader expects both byte counts); empty[] and accfull[] in both (the
// leader's commits multicast to the pair); accempty[] in the leader (every
// epilogue warp of both CTAs arrives on it).
// ===========================================================================
namespace t3p {
constexpr int KC = 32, STAGES = 3;
constexpr int HALF_ROWS = 128;                  // rows of A (and of B) staged by one CTA
constexpr int OP_BYTES = HALF_ROWS * KC * 4;    // 16 KB
constexpr int STAGE_BYTES = 4 * OP_BYTES;       // A_hi, A_lo, B_hi, B_lo halves
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
constexpr int TILE = 256;
constexpr uint32_t IDESC = idesc(kFmtTF32, TILE, TILE);
constexpr int TMEM_COLS = 512;                  // 2 accumulator buffers x 256 columns
constexpr int kSuper = kPairSuper;              // supertile edge in 256-tiles
}  // namespace t3p

// Pair tiles (units of 256): kEnumFull (bi = t / nt) or kEnumLowerOffBand (supertiles of the
// lower triangle, g.nt tile rows, band in panel-wide tiles).
__device__ __forceinline__ bool decode_pair_tile(const GemmArgs& g, long long t, int& bi, int& bj) {
  if (g.enum_mode == kEnumFull) {
    bi = (int)(t / g.nt);
    bj = (int)(t % g.nt);
    return true;
  }
  constexpr int S = t3p::kSuper;
  const long long sidx = t / (S * S);
  const int loc = (int)(t % (S * S));
  int SI, SJ;
  tile_tri_decode(sidx, SI, SJ);
  bi = SI * S + loc / S;
  bj = SJ * S + loc % S;
  if (bi >= g.nt || bj > bi) return false;
  const int per = g.panel / t3p::TILE;
  return (bi / per - bj / per) > g.band;
}

// Far tiles: when the largest |entries| of the two operand blocks are at most 2^eA and 2^eB
// with eA + eB <= far_thr, the single product hi * hi (relative error ~2^-10 per term) has
// an absolute error no larger than the three-product form makes on blocks of size 1; the
// caller sets far_thr from the scale of Sigma.  Producer and MMA issuer decide alike.
// src 1 asks about the second operand pair (g.K2 > 0), whose rows start at a2_row0 / b2_row0.
__device__ __forceinline__ bool far_tile(const GemmArgs& g, int bi, int bj, int src) {
  const int* eab = src ? g.ea2_blk : g.ea_blk;
  const int* ebb = src ? g.eb2_blk : g.eb_blk;
  if (g.far_thr == INT_MIN || !eab || !ebb) return false;
  const int ea = eab[(src ? g.a2_row0 : g.a_row0) / t3p::TILE + bi];
  const int eb = ebb[(src ? g.b2_row0 : g.b_row0) / t3p::TILE + bj];
  return (long long)ea + (long long)eb <= (long long)g.far_thr;
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
    gemm_t3_pair_kernel(const __grid_constant__ CUtensorMap tA_hi, const __grid_constant__ CUtensorMap tA_lo,
                        const __grid_constant__ CUtensorMap tB_hi, const __grid_constant__ CUtensorMap tB_lo,
                        const __grid_constant__ CUtensorMap tA2_hi, const __grid_constant__ CUtensorMap tA2_lo,
                        const __grid_constant__ CUtensorMap tB2_hi, const __grid_constant__ CUtensorMap tB2_lo,
                        const __grid_constant__ GemmArgs g) {
  using namespace t3p;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accfull = empty + STAGES;
  uint64_t* accempty = accfull + 2;
  uint64_t* drain = accempty + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort = (volatile int*)(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = (rank == 0);
  const long long pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 2 * (kEpiThreads / 32));
    }
    mbar_init(drain, 1);
    *abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, TMEM_COLS);
  fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers are initialised before any remote arrival or copy
  fence_after();
  const uint32_t tmem = *tmem_slot;
  // chunks [0, kc1) reduce over the first operand pair, [kc1, kchunks) over the second
  const int kc1 = g.K / KC;
  const int kchunks = kc1 + g.K2 / KC;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    const uint64_t pol = l2_evict_last_policy();
    prefetch_tmap(&tA_hi);
    prefetch_tmap(&tA_lo);
    prefetch_tmap(&tB_hi);
    prefetch_tmap(&tB_lo);
    if (g.K2 > 0) {
      prefetch_tmap(&tA2_hi);
      prefetch_tmap(&tA2_lo);
      prefetch_tmap(&tB2_hi);
      prefetch_tmap(&tB2_lo);
    }
    int stage = 0;
    uint32_t phase = 0;
    int last_par[STAGES];
    for (int s = 0; s < STAGES; ++s) last_par[s] = -1;
    for (long long t = pair; t < g.ntiles && !*abort; t += npairs) {
      int bi, bj;
      if (!decode_pair_tile(g, t, bi, bj)) continue;
      const int ya1 = g.a_row0 + bi * TILE + (int)rank * HALF_ROWS;
      const int yb1 = g.b_row0 + bj * TILE + (int)rank * HALF_ROWS;
      const int ya2 = g.a2_row0 + bi * TILE + (int)rank * HALF_ROWS;
      const int yb2 = g.b2_row0 + bj * TILE + (int)rank * HALF_ROWS;
      const bool one1 = far_tile(g, bi, bj, 0);
      const bool one2 = g.K2 > 0 && far_tile(g, bi, bj, 1);
      for (int kc = 0; kc < kchunks; ++kc) {
        if (!mbar_wait(&empty[stage], phase ^ 1, abort)) {
          *abort = 1;
          record_timeout(g.st, 51);
          break;
        }
        const bool second = kc >= kc1;
        const bool one = second ? one2 : one1;
        const int kx = (second ? kc - kc1 : kc) * KC;
        const int ya = second ? ya2 : ya1, yb = second ? yb2 : yb1;
        uint8_t* sb = smem + stage * STAGE_BYTES;
        if (leader) mbar_expect_tx(&full[stage], (one ? 1 : 2) * STAGE_BYTES);
        const uint32_t fl = map_to_rank(smem_u32(&full[stage]), 0);
        tma_load_2d_pair_hint(sb, second ? &tA2_hi : &tA_hi, fl, kx, ya, pol);
        if (!one) tma_load_2d_pair_hint(sb + OP_BYTES, second ? &tA2_lo : &tA_lo, fl, kx, ya, pol);
        tma_load_2d_pair_hint(sb + 2 * OP_BYTES, second ? &tB2_hi : &tB_hi, fl, kx, yb, pol);
        if (!one) tma_load_2d_pair_hint(sb + 3 * OP_BYTES, second ? &tB2_lo : &tB_lo, fl, kx, yb, pol);
        last_par[stage] = (int)phase;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    if (*abort && leader) {  // the leader's full barriers also count the peer's bytes
      for (int s = 0; s < STAGES; ++s)
        if (last_par[s] >= 0) {
          volatile int never = 0;
          mbar_wait(&full[s], (uint32_t)last_par[s], &never);
        }
    }
  } else if (warp == 1 && lane == 0 && leader) {
    // ---------------- MMA issuer (leader only) ----------------
    int stage = 0;
    uint32_t phase = 0;
    int it = 0;
    for (long long t = pair; t < g.ntiles && !*abort; t += npairs) {
      int bi, bj;
      if (!decode_pair_tile(g, t, bi, bj)) continue;
      const int b = it & 1;
      const uint32_t ap = (it >> 1) & 1;
      if (!mbar_wait(&accempty[b], ap ^ 1, abort)) {
        *abort = 1;
        record_timeout(g.st, 52);
        break;
      }
      fence_after();
      const uint32_t d = tmem + b * TILE;
      const bool one1 = far_tile(g, bi, bj, 0);
      const bool one2 = g.K2 > 0 && far_tile(g, bi, bj, 1);
      bool ok = true;
      for (int kc = 0; kc < kchunks; ++kc) {
        if (!mbar_wait(&full[stage], phase, abort)) {
          *abort = 1;
          record_timeout(g.st, 53);
          ok = false;
          break;
        }
        fence_after();
        const bool one = kc >= kc1 ? one2 : one1;
        const uint32_t sb = smem_u32(smem + stage * STAGE_BYTES);
        const uint64_t ahi = sdesc_sw128(sb), alo = sdesc_sw128(sb + OP_BYTES);
        const uint64_t bhi = sdesc_sw128(sb + 2 * OP_BYTES), blo = sdesc_sw128(sb + 3 * OP_BYTES);
#pragma unroll
        for (int kk = 0; kk < KC / 8; ++kk) {  // K = 8 per instruction: advance 32 bytes
          const uint64_t o = (uint64_t)(kk * 2);
          mma_tf32_pair(d, ahi + o, bhi + o, IDESC, (kc | kk) ? 1u : 0u);
          if (!one) {
            mma_tf32_pair(d, ahi + o, blo + o, IDESC, 1u);
            mma_tf32_pair(d, alo + o, bhi + o, IDESC, 1u);
          }
        }
        mma_commit_pair(&empty[stage], (uint16_t)0x3);
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (!ok) break;
      mma_commit_pair(&accfull[b], (uint16_t)0x3);
      ++it;
    }
    // every MMA issued has finished before the pair leaves (matters after a time-out)
    mma_commit_pair(drain, (uint16_t)0x1);
    volatile int never = 0;
    mbar_wait(drain, 0, &never);
  } else if (warp >= 2) {
    // ---------------- epilogue (both CTAs): own TMEM -> FP64 C ----------------
    // warp w drains TMEM lanes 32*(w%4).. and the 128-column half (w-2)/4 of the 256 columns
    const int quad = warp & 3;
    const int half = (warp - 2) >> 2;
    const int r = quad * 32 + lane;
    const uint32_t accempty_l[2] = {map_to_rank(smem_u32(&accempty[0]), 0), map_to_rank(smem_u32(&accempty[1]), 0)};
    int it = 0;
    for (long long t = pair; t < g.ntiles && !*abort; t += npairs) {
      int bi, bj;
      if (!decode_pair_tile(g, t, bi, bj)) continue;
      const int b = it & 1;
      const uint32_t ap = (it >> 1) & 1;
      if (!mbar_wait(&accfull[b], ap, abort)) {
        *abort = 1;
        record_timeout(g.st, 54);
        break;
      }
      fence_after();
      const int64_t row = g.c_row0 + (int64_t)bi * TILE + (int64_t)rank * HALF_ROWS + r;
      const int64_t col0 = g.c_col0 + (int64_t)bj * TILE + half * 128;
      double* cp = g.C + row + col0 * g.ldc;
      // L2 prefetch two chunks ahead (lane l: column l / 2 of the chunk, rows 16 (l % 2) .. of
      // this warp's 32), and in the last two chunks the first two of this pair's next tile: the
      // loads below then wait on L2 rather than DRAM, and each SM keeps more C lines in flight
      // than its registers hold
      const double* pf = g.C + (row - lane + 16 * (lane & 1)) + (col0 + (lane >> 1)) * g.ldc;
      const double* pf_next = nullptr;
      if (!g.store) {
        for (long long t2 = t + npairs; t2 < g.ntiles; t2 += npairs) {
          int bi2, bj2;
          if (!decode_pair_tile(g, t2, bi2, bj2)) continue;
          pf_next = g.C + (g.c_row0 + (int64_t)bi2 * TILE + (int64_t)rank * HALF_ROWS + quad * 32 + 16 * (lane & 1)) +
                    (g.c_col0 + (int64_t)bj2 * TILE + half * 128 + (lane >> 1)) * g.ldc;
          break;
        }
      }
      // eight 16-column chunks of this warp's 128 columns, the C loads of chunk q + 1 issued
      // before chunk q is drained from TMEM, so their latency hides behind its conversion and stores
      double cbuf[2][16];
#pragma unroll
      for (int j = 0; j < 16; ++j) cbuf[0][j] = g.store ? 0.0 : __ldcs(cp + (int64_t)j * g.ldc);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (!g.store) {
          if (q + 2 < 8)
            prefetch_l2(pf + (int64_t)((q + 2) * 16) * g.ldc);
          else if (pf_next)
            prefetch_l2(pf_next + (int64_t)((q - 6) * 16) * g.ldc);
        }
        if (q + 1 < 8) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            cbuf[(q + 1) & 1][j] = g.store ? 0.0 : __ldcs(cp + (int64_t)((q + 1) * 16 + j) * g.ldc);
        }
        uint32_t acc[16];
        tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + b * TILE + half * 128 + q * 16, acc);
        tmem_ld_wait();
        if (q == 7) {
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(accempty_l[b]);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const double v = f32_bits_to_f64(acc[j]);
          __stcs(cp + (int64_t)(q * 16 + j) * g.ldc, g.store ? v : cbuf[q & 1][j] - v);
        }
      }
      ++it;
    }
  }
  fence_before();
  __syncthreads();
  cluster_sync();  // the leader's MMAs read this CTA's shared memory: both stay until both are done
  if (warp == 1) {
    fence_after();
    tmem_dealloc_pair(tmem, TMEM_COLS);
  }
}

// ===========================================================================
// OZ kernel: exact products of 5-digit operands, tiles 128 x tn with tn = 96, 64 or 32.
// ===========================================================================
namespace oz {
constexpr int TM = 128, TN = 96, S = kOzSlices;
constexpr int A_BYTES = TM * 32;                       // one digit plane of a 16-column step
constexpr int STAGE_BYTES = S * (A_BYTES + TN * 32), STAGES = 6;
constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 256;
constexpr int kEpiWarps = 16, kThreads = 64 + 32 * kEpiWarps;
constexpr int TMEM_COLS = 512;
static_assert(SMEM_BYTES <= 232448 && S * TN <= TMEM_COLS && 2 * S * 32 <= TMEM_COLS, "stages and accumulators fit");

struct Args {
  double* C;
  int64_t ldc, c_row0, c_col0;
  const uint8_t *A, *B;      // first plane, at the operand's row origin
  int64_t a_plane, b_plane;  // bytes between planes
  const int *ea, *eb;
  int mode, band, panel;     // kEnumFull or kEnumBand
  int mt, n;                 // row blocks; columns (kEnumFull)
  int tn, nbuf, k16;
  int store, lower, tri;
  long long ntiles;
  DevStatus* st;
};

// Tile t: row block bi, column offset cofs and width (a multiple of 32).  Band tiles run along each row block from its
// first panel of the band to the diagonal; `at` and `base` (row block, tiles before it) follow the growing t of a CTA.
// False: skip the tile (above the diagonal).
struct Cursor {
  int at = 0;
  long long base = 0;
};
__device__ __forceinline__ bool tile_of(const Args& g, long long t, Cursor& c, int& bi, int& cofs, int& width) {
  if (g.mode == kEnumFull) {
    const int per = (g.n + g.tn - 1) / g.tn;
    bi = (int)(t / per);
    cofs = (int)(t % per) * g.tn;
    width = min(g.tn, g.n - cofs);
    return !(g.lower && g.c_col0 + cofs > g.c_row0 + (int64_t)bi * TM + TM - 1);
  }
  const int SI = g.panel / TM;
  while (true) {
    const int start = max(0, c.at / SI - g.band) * g.panel, end = (c.at + 1) * TM;
    const int count = (end - start + g.tn - 1) / g.tn;
    if (t < c.base + count) {
      bi = c.at;
      cofs = start + (int)(t - c.base) * g.tn;
      width = min(g.tn, end - cofs);
      return true;
    }
    c.base += count;
    ++c.at;
  }
}

// One warp's part of a tile: 32 rows x CH columns out of TMEM, `release` once the accumulators are read.
template <int CH, class Release>
__device__ __forceinline__ void drain(const Args& g, int bi, int cofs, int quad, int part, uint32_t acc, Release release) {
  const int lane = threadIdx.x & 31, r = quad * 32 + lane;
  const int lc0 = CH * part;
  const int64_t row = g.c_row0 + (int64_t)bi * TM + r, col0 = g.c_col0 + cofs + lc0;
  double* cp = g.C + row + col0 * g.ldc;
  const int last = g.lower ? (int)min((int64_t)CH, row - col0) : CH;  // columns up to this one are written
  // group q holds an exact integer a_q (|a_q| < 2^24) of weight 2^(-7(q+2)): V = sum_q a_q 2^(7(4-q)) is an integer
  // below 2^53, combined from two 32-bit words (|a_0|, |a_2| < 2^23.4) and a_4.  Half of the conversions go by
  // additions: F2I converts 16 lanes a cycle on an SM.
  long long V[CH];
  const uint32_t ta = acc + ((uint32_t)(quad * 32) << 16) + lc0;
  const int width = 4 * CH;
#pragma unroll
  for (int h = 0; h < CH; h += 4) {
    uint32_t x[S][4];
#pragma unroll
    for (int q = 0; q < S; ++q) tmem_ld4(ta + q * width + h, x[q]);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int w01 = f32_to_int(__uint_as_float(x[0][j])) * 128 + __float2int_rn(__uint_as_float(x[1][j]));
      const int w23 = f32_to_int(__uint_as_float(x[2][j])) * 128 + __float2int_rn(__uint_as_float(x[3][j]));
      V[h + j] = ((long long)w01 * 16384 + w23) * 128 + __float2int_rn(__uint_as_float(x[4][j]));
    }
  }
  fence_before();
  release();
  const int base = g.ea[bi * TM + r] - 7 * (S + 1);
  const int* eb = g.eb + cofs + lc0;
#pragma unroll
  for (int j0 = 0; j0 < CH; j0 += 4) {
    asm volatile("" ::: "memory");  // four outputs at a time: more would not fit the registers
    double cv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) cv[j] = !g.store && j0 + j <= last ? __ldcs(cp + (int64_t)(j0 + j) * g.ldc) : 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double x = i53_to_f64_scaled(V[j0 + j], base + eb[j0 + j]);
      if (j0 + j <= last) __stcs(cp + (int64_t)(j0 + j) * g.ldc, g.store ? x : cv[j] - x);
    }
  }
}
}  // namespace oz

// One CTA per SM, persistent: warp 0 copies digit planes into a ring of 16-column stages, one thread of warp 1 issues
// the MMAs, warps 2-17 drain TMEM into C.  The S B planes of a stage lie one after another and group q = s + t follows
// group q - 1 in TMEM, so A digit s against B digits 0 .. S-1-s is one run of columns (two MMAs where N > 256).  The
// first (s = 0) of a tile writes all groups; sums stay exact integers, so neither order nor tile shape changes a bit.
//
// Bound: the tensor pipe (15 BF16 products: 125 TFLOP/s at 1,872) if the operands come in fast enough, which the tile
// width decides: a 16-column step takes 7.9 tn cycles of MMA for 20 KB + 160 tn bytes, 46 bytes a cycle at tn = 96,
// 60 at 64, 100 at 32, against the ~46 an SM was seen to take in.  96 columns leave room for one accumulator set, whose
// drain is then not hidden; 32-wide tiles, for launches with few tiles, have two.  With tiles of 48 columns (and 32
// outside the band) in two sets, 73 bytes a cycle, the band products of an n = 90,000 factorisation took 324 ms, now 286.
__global__ void __launch_bounds__(oz::kThreads, 1) gemm_oz_kernel(const __grid_constant__ oz::Args g) {
  using namespace oz;
  extern __shared__ __align__(256) uint8_t smem_oz[];
  uint8_t* smem = smem_oz;
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accfull = empty + STAGES;
  uint64_t* accempty = accfull + 2;
  uint32_t* tmem_slot = (uint32_t*)(accempty + 2);
  volatile int* abort = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 32 * kEpiWarps);
    }
    *abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, TMEM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  Cursor cur;
  int bi, cofs, width;

  if (warp == 0) {
    // ---------------- copies: lane s < S brings A plane s, lane S + s B plane s ----------------
    int stage = 0;
    uint32_t phase = 0;
    int last_par[STAGES];
    for (int s = 0; s < STAGES; ++s) last_par[s] = -1;
    bool ok = true;  // the same for every lane
    for (long long t = blockIdx.x; t < g.ntiles && ok; t += gridDim.x) {
      if (!tile_of(g, t, cur, bi, cofs, width)) continue;
      const int steps = g.tri ? min(g.k16, (cofs + width) / 16) : g.k16;
      const bool isA = lane < S;
      const uint8_t* src = isA ? g.A + lane * g.a_plane + (int64_t)bi * A_BYTES
                               : g.B + (lane - S) * g.b_plane + (int64_t)cofs * 32;
      const int64_t step_bytes = S * (isA ? g.a_plane : g.b_plane);
      const uint32_t bytes = isA ? A_BYTES : width * 32;
      const uint32_t off = isA ? lane * A_BYTES : S * A_BYTES + (lane - S) * bytes;
      for (int kc = 0; kc < steps; ++kc) {
        if (lane == 0) {
          ok = mbar_wait(&empty[stage], phase ^ 1, abort);
          if (ok) {
            mbar_expect_tx(&full[stage], S * (A_BYTES + width * 32));
          } else {
            *abort = 1;
            record_timeout(g.st, 21);
          }
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        if (lane < 2 * S) bulk_load(smem_u32(smem + stage * STAGE_BYTES) + off, src, bytes, smem_u32(&full[stage]));
        src += step_bytes;
        last_par[stage] = (int)phase;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
    }
    if (!ok || *abort) {  // let every copy of this warp land before the CTA exits
      for (int s = 0; s < STAGES; ++s)
        if (last_par[s] >= 0) {
          volatile int never = 0;
          mbar_wait(&full[s], (uint32_t)last_par[s], &never);
        }
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issue ----------------
    int stage = 0, it = 0;
    uint32_t phase = 0;
    for (long long t = blockIdx.x; t < g.ntiles && !*abort; t += gridDim.x) {
      if (!tile_of(g, t, cur, bi, cofs, width)) continue;
      const int steps = g.tri ? min(g.k16, (cofs + width) / 16) : g.k16;
      const int b = g.nbuf > 1 ? it & 1 : 0;
      const uint32_t ap = (g.nbuf > 1 ? it >> 1 : it) & 1;
      if (!mbar_wait(&accempty[b], ap ^ 1, abort)) {
        *abort = 1;
        record_timeout(g.st, 22);
        break;
      }
      fence_after();
      const uint32_t d0 = tmem + b * (TMEM_COLS / 2);
      bool ok = true;
      // the width as a constant: with run-time shapes the one issuing thread would not keep up with the tensor pipe
      auto products = [&](auto w) {
        constexpr int W = decltype(w)::value;
        for (int kc = 0; kc < steps; ++kc) {
          if (!mbar_wait(&full[stage], phase, abort)) {
            *abort = 1;
            record_timeout(g.st, 23);
            ok = false;
            return;
          }
          fence_after();
          const uint32_t sb = smem_u32(smem + stage * STAGE_BYTES);
          const uint64_t b0 = sdesc_flat(sb + S * A_BYTES);
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const uint64_t a = sdesc_flat(sb + s * A_BYTES);
            const int n = W * (S - s);
            const uint32_t acc = (kc | s) ? 1u : 0u;
            if (n > 256) {
              const int h = n / 2;  // a multiple of 16
              mma_bf16(d0 + s * W, a, b0, idesc(kFmtBF16, TM, h), acc);
              mma_bf16(d0 + s * W + h, a, b0 + (uint64_t)(h * 32 >> 4), idesc(kFmtBF16, TM, h), acc);
            } else {
              mma_bf16(d0 + s * W, a, b0, idesc(kFmtBF16, TM, n), acc);
            }
          }
          mma_commit(&empty[stage]);
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
      };
      if (width == 96)
        products(std::integral_constant<int, 96>{});
      else if (width == 64)
        products(std::integral_constant<int, 64>{});
      else
        products(std::integral_constant<int, 32>{});
      if (!ok) break;
      mma_commit(&accfull[b]);
      ++it;
    }
  } else if (warp >= 2) {
    // ---------------- drain: warp w takes TMEM lanes 32 (w % 4).. and a quarter of the columns ----------------
    const int quad = warp & 3, part = (warp - 2) >> 2;
    int it = 0;
    for (long long t = blockIdx.x; t < g.ntiles; t += gridDim.x) {
      if (!tile_of(g, t, cur, bi, cofs, width)) continue;
      const int b = g.nbuf > 1 ? it & 1 : 0;
      const uint32_t ap = (g.nbuf > 1 ? it >> 1 : it) & 1;
      const int ch = width / 4;
      if (!g.store) {  // this warp's lines of C into L2 while the products run
        const int64_t col0 = g.c_col0 + cofs + ch * part;
        for (int l = lane; l < 2 * ch; l += 32)
          prefetch_l2(g.C + g.c_row0 + (int64_t)bi * TM + quad * 32 + 16 * (l & 1) + (col0 + (l >> 1)) * g.ldc);
      }
      if (!__all_sync(0xffffffffu, mbar_wait(&accfull[b], ap, abort))) {
        if (lane == 0) {
          *abort = 1;
          record_timeout(g.st, 24);
        }
        break;
      }
      fence_after();
      const uint32_t acc = tmem + b * (TMEM_COLS / 2);
      auto release = [&] { mbar_arrive(&accempty[b]); };
      if (width == 96)
        drain<24>(g, bi, cofs, quad, part, acc, release);
      else if (width == 64)
        drain<16>(g, bi, cofs, quad, part, acc, release);
      else
        drain<8>(g, bi, cofs, quad, part, acc, release);
      ++it;
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ===========================================================================
// Split kernel: FP64 rows -> T3 (TF32 hi/lo, row-major) and OZ digit planes.  16 rows per CTA, every value in a
// register: thread (row, group) of 16 x 16 holds K / 16 consecutive columns of its row, at most 32, and eight columns
// give 16-byte stores.  On a panel's look-ahead stream its grid is held to that stream's SMs: larger grids get between the
// main stream's kernels (the trailing update of n = 90,000 then takes 680 ms instead of 635).  Bound: the integer pipe (~25 instructions a value for T3, ~45 for the digits), on the few SMs of
// the look-ahead stream, and HBM (8 bytes read, 18 written).  All splits of n = 90,000: 289 ms through shared memory with
// 64-bit integers, now 220.
// ===========================================================================
// TF32 rounding (11 significant bits, half away from zero in magnitude) of the double with upper word w, as FP32 bits;
// below the FP32 normal range 0.  *up: the upper word of the rounded value (its lower word is 0).  Bit 41 of the
// pattern, where the rounding adds, is bit 9 of the upper word.
__device__ __forceinline__ uint32_t tf32_of(uint32_t w, uint32_t* up) {
  const uint32_t sign = w & 0x80000000u, m = ((w & 0x7FFFFFFFu) + 0x200u) & ~0x3FFu;
  const int fe = (int)(m >> 20) - 896;  // FP64 bias 1023 -> FP32 bias 127
  *up = fe <= 0 ? sign : sign | m;
  return fe <= 0 ? sign : sign | ((uint32_t)fe << 23) | ((m & 0xFFFFFu) << 3);
}
// a's two TF32 parts.  The one FP64 instruction (exact: a's bits below the rounding point) runs beside the integer ones.
__device__ __forceinline__ void tf32_parts(double a, uint32_t& h, uint32_t& l) {
  uint32_t up;
  h = tf32_of((uint32_t)__double2hiint(a), &up);
  l = tf32_of((uint32_t)__double2hiint(a - __hiloint2double((int)up, 0)), &up);
}

// The five OZ digits of a 2^(35-e) rounded to an integer N (|a| < 2^e: |N| <= 2^35), as FP32 values: balanced base-128
// digits from the least significant end, the leading one keeping the rest (|d_0| <= 128, |d_s| <= 64 otherwise; all exact
// in BF16).  With 64 (1 + 128 + 128^2 + 128^3) added, the lower four are plain digits plus 64.
__device__ __forceinline__ void oz_digits(uint32_t dh, uint32_t dl, int e, float (&d)[kOzSlices]) {
  const int E = (int)((dh >> 20) & 0x7FFu);
  // a = M 2^(E-1075) with its 53-bit significand M: N = M 2^-sh, sh = 1040 + e - E >= 18; one bit more for the rounding
  const int sh = 1040 + e - E;
  const unsigned long long M = E ? ((unsigned long long)((dh & 0xFFFFFu) | 0x100000u) << 32) | dl : 0ull;
  const unsigned long long N = ((M >> min(sh - 1, 63)) + 1) >> 1;
  constexpr unsigned long long B = 64ull * (1 + 128 + 128 * 128 + 128 * 128 * 128);
  const unsigned long long x = (int)dh < 0 ? B - N : B + N;
  constexpr float kMagic = 12582912.0f;
  const uint32_t lo = (uint32_t)x;
#pragma unroll
  for (int s = 1; s < kOzSlices; ++s)
    d[s] = __uint_as_float(((lo >> (7 * (kOzSlices - 1 - s))) & 127u) | 0x4B400000u) - (kMagic + 64.0f);
  d[0] = __int_as_float((int)((long long)x >> 28) + 0x4B400000) - kMagic;
}

// Rows [r0, r0 + kSplitRows) of the split (one CTA); the digit planes hold dig_rows rows.
constexpr int kSplitThreads = 256, kSplitGroups = kSplitThreads / kSplitRows;
__device__ __forceinline__ void split_rows_body(const double* __restrict__ src, int64_t rs, int64_t cs, int rows, int K,
                                                float* __restrict__ hi, float* __restrict__ lo,
                                                uint8_t* __restrict__ dig, int64_t dig_rows, int* __restrict__ ex,
                                                int out_row0, int r0) {
  extern __shared__ __align__(16) float stage[];  // 2 kSplitRows x ld: the TF32 parts on their way out
  __shared__ unsigned int s_max[kSplitRows][kSplitGroups + 1], s_low[kSplitRows][kSplitGroups + 1];
  const int ld = K + 4;
  const int tid = threadIdx.x, r = tid % kSplitRows, g = tid / kSplitRows;
  const int row = r0 + r;
  constexpr int U = kSplitMaxK / 8 / kSplitGroups;
  const int octets = K / 8;  // dealt to the groups in runs: group g takes octets [o0, o1), at most U
  const int o0 = octets * g / kSplitGroups, o1 = octets * (g + 1) / kSplitGroups;
  const double* p = src + (int64_t)row * rs + (int64_t)(8 * o0) * cs;
  double v[U][8];
#pragma unroll
  for (int u = 0; u < U; ++u)
#pragma unroll
    for (int j = 0; j < 8; ++j) v[u][j] = o0 + u < o1 && row < rows ? p[(int64_t)(8 * u + j) * cs] : 0.0;
  const int64_t orow = (int64_t)(out_row0 + row);
  int e = 0;
  if (dig) {
    // row maximum of |a| on the bit patterns: f 2^e with f in [0.5, 1), e = biased exponent - 1022 (0: all zero)
    unsigned int mx = 0, low = 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        mx = max(mx, (unsigned int)__double2hiint(v[u][j]) & 0x7FFFFFFFu);
        low |= (unsigned int)__double2loint(v[u][j]);
      }
    s_max[r][g] = mx;
    s_low[r][g] = low;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSplitGroups; ++q) {
      mx = max(mx, s_max[r][q]);
      low |= s_low[r][q];
    }
    e = mx | low ? (int)(mx >> 20) - 1022 : 0;
    if (g == 0 && row < rows && ex) ex[orow] = e;
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int o = o0 + u;
    if (o >= o1 || row >= rows) continue;
    if (hi) {
      uint32_t h[8], l[8];
#pragma unroll
      for (int j = 0; j < 8; ++j)
        tf32_parts(v[u][j], h[j], l[j]);
      uint4* ph = reinterpret_cast<uint4*>(stage + r * ld + 8 * o);
      uint4* pl = reinterpret_cast<uint4*>(stage + (kSplitRows + r) * ld + 8 * o);
      ph[0] = make_uint4(h[0], h[1], h[2], h[3]);
      ph[1] = make_uint4(h[4], h[5], h[6], h[7]);
      pl[0] = make_uint4(l[0], l[1], l[2], l[3]);
      pl[1] = make_uint4(l[4], l[5], l[6], l[7]);
    }
    if (dig) {
      uint32_t w[kOzSlices][4];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float d[kOzSlices];
        oz_digits((uint32_t)__double2hiint(v[u][j]), (uint32_t)__double2loint(v[u][j]), e, d);
#pragma unroll
        for (int s = 0; s < kOzSlices; ++s) {  // exact in BF16: the upper half of the word
          const uint32_t b = __float_as_uint(d[s]);
          w[s][j >> 1] = (j & 1) ? __byte_perm(w[s][j >> 1], b, 0x7632) : b;
        }
      }
      uint8_t* po = dig + (int64_t)(o >> 1) * kOzSlices * dig_rows * 32 + (orow >> 3) * 256 + (o & 1) * 128 +
                    (orow & 7) * 16;
#pragma unroll
      for (int s = 0; s < kOzSlices; ++s)
        *reinterpret_cast<uint4*>(po + (int64_t)s * dig_rows * 32) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
  }
  if (hi) {  // whole lines
    __syncthreads();
    const int quads = K / 4;
    for (int idx = tid; idx < kSplitRows * quads; idx += kSplitThreads) {
      const int rr = idx / quads, q = idx - rr * quads;
      if (r0 + rr >= rows) break;
      const int64_t at = (int64_t)(out_row0 + r0 + rr) * K + 4 * q;
      *reinterpret_cast<uint4*>(hi + at) = *reinterpret_cast<const uint4*>(stage + rr * ld + 4 * q);
      *reinterpret_cast<uint4*>(lo + at) = *reinterpret_cast<const uint4*>(stage + (kSplitRows + rr) * ld + 4 * q);
    }
  }
}

__global__ void __launch_bounds__(kSplitThreads) split_rows_kernel(const double* __restrict__ src, int64_t rs,
                                                                      int64_t cs, int rows, int K,
                                                                      float* __restrict__ hi, float* __restrict__ lo,
                                                                      uint8_t* __restrict__ dig, int64_t dig_rows,
                                                                      int* __restrict__ ex, int out_row0) {
  for (int r0 = blockIdx.x * kSplitRows; r0 < rows; r0 += gridDim.x * kSplitRows) {
    split_rows_body(src, rs, cs, rows, K, hi, lo, dig, dig_rows, ex, out_row0, r0);
    __syncthreads();
  }
}

// Many pieces in one launch: blockIdx.y = piece, blockIdx.x = 16-row chunk of it.
__global__ void __launch_bounds__(kSplitThreads) split_rows_tasks_kernel(const SplitTask* __restrict__ tasks, int K,
                                                                            float* __restrict__ hi,
                                                                            float* __restrict__ lo,
                                                                            uint8_t* __restrict__ dig, int64_t dig_rows,
                                                                            int* __restrict__ ex) {
  const SplitTask t = tasks[blockIdx.y];
  const int r0 = blockIdx.x * kSplitRows;
  if (r0 >= t.rows) return;  // uniform over the CTA, before any barrier
  split_rows_body(t.src, t.rs, t.cs, t.rows, K, hi, lo, dig, dig_rows, ex, t.out_row0, r0);
}

// Per 256-row block maximum of the row exponents (rows past the end count as -infinity).
__global__ void __launch_bounds__(256) row_exp_blockmax_kernel(const int* __restrict__ ex, int64_t rows,
                                                               int* __restrict__ exb) {
  const int64_t r = (int64_t)blockIdx.x * 256 + threadIdx.x;
  int v = r < rows ? ex[r] : INT_MIN;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  __shared__ int w[8];
  if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    int m = w[0];
    for (int i = 1; i < 8; ++i) m = max(m, w[i]);
    exb[blockIdx.x] = m;
  }
}

// ===========================================================================
// host side
// ===========================================================================
static PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  }
  return fn;
}

// 2-D row-major tensor [rows][K] of 4-byte (fp32) or 2-byte (bf16) elements,
// box = (box_k, box_rows), 128-byte swizzle.
cudaError_t make_tmap(CUtensorMap* m, const void* base, int64_t rows, int K, int elem_bytes, int box_k, int box_rows) {
  auto enc = get_encode();
  if (!enc) return cudaErrorNotSupported;
  if (((uintptr_t)base & 15) != 0 || ((int64_t)K * elem_bytes) % 16 != 0 || box_k * elem_bytes != 128)
    return cudaErrorInvalidValue;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)K * elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_k, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, elem_bytes == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                   const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t make_split_maps(SplitOperand& op) {
  cudaError_t e = cudaSuccess;
  if (op.hi) {
    if ((e = make_tmap(&op.t_hi, op.hi, op.rows, op.K, 4, 32, 128)) != cudaSuccess) return e;
    if ((e = make_tmap(&op.t_lo, op.lo, op.rows, op.K, 4, 32, 128)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// (Always the size for K = 512: with less, the CTAs of the look-ahead stream's splits would find room beside those of the
// main stream's products.)
constexpr int kSplitSmem = 2 * kSplitRows * (kSplitMaxK + 4) * (int)sizeof(float);

static cudaError_t split_attr() {
  static PerDeviceOnce once;
  return once([] {
    cudaError_t r = cudaFuncSetAttribute(split_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(split_rows_tasks_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem);
    return r;
  });
}

cudaError_t launch_split_rows(cudaStream_t s, const double* src, int64_t rs, int64_t cs, int rows, int K,
                              SplitOperand& op, int out_row0, int max_ctas) {
  if (rows <= 0) return cudaSuccess;
  if (K > kSplitMaxK || K % 16) return cudaErrorInvalidValue;
  const cudaError_t e = split_attr();
  if (e != cudaSuccess) return e;
  int grid = (rows + kSplitRows - 1) / kSplitRows;
  if (max_ctas > 0 && grid > 2 * max_ctas) grid = 2 * max_ctas;
  split_rows_kernel<<<grid, kSplitThreads, kSplitSmem, s>>>(src, rs, cs, rows, K, op.hi, op.lo, (uint8_t*)op.dig, op.rows,
                                                            op.ex, out_row0);
  return cudaGetLastError();
}

cudaError_t launch_split_rows_tasks(cudaStream_t s, const SplitTask* d_tasks, int ntasks, int max_rows, int K,
                                    SplitOperand& op) {
  if (ntasks <= 0 || max_rows <= 0) return cudaSuccess;
  if (K > kSplitMaxK || K % 16) return cudaErrorInvalidValue;
  const cudaError_t e = split_attr();
  if (e != cudaSuccess) return e;
  split_rows_tasks_kernel<<<dim3((unsigned)((max_rows + kSplitRows - 1) / kSplitRows), (unsigned)ntasks), kSplitThreads,
                            kSplitSmem, s>>>(d_tasks, K, op.hi, op.lo, (uint8_t*)op.dig, op.rows, op.ex);
  return cudaGetLastError();
}

static int num_sms() {
  static std::atomic<int> cache[64];
  const int n = per_device_int(cache, [] {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
  });
  return n > 0 ? n : 148;
}

int tc_num_sms() { return num_sms(); }

cudaError_t launch_gemm_t3(cudaStream_t s, const SplitOperand& A, const SplitOperand& B, const GemmArgs& g,
                           int max_ctas, const SplitOperand* second) {
  if (g.ntiles <= 0) return cudaSuccess;
  if (g.K2 > 0 && (!second || g.enum_mode != kEnumTasks || g.store)) return cudaErrorInvalidValue;
  if (!second) second = &A;
  static PerDeviceOnce attr_once;
  {
    const cudaError_t e =
        attr_once([] { return cudaFuncSetAttribute(gemm_t3_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, t3::SMEM_BYTES); });
    if (e != cudaSuccess) return e;
  }
  int cap = num_sms();
  if (max_ctas > 0 && max_ctas < cap) cap = max_ctas;
  const int grid = (int)(g.ntiles < cap ? g.ntiles : cap);
  gemm_t3_kernel<<<grid, t3::kThreads, t3::SMEM_BYTES, s>>>(A.t_hi, A.t_lo, B.t_hi, B.t_lo, second->t_hi,
                                                                 second->t_lo, g);
  return cudaGetLastError();
}

cudaError_t launch_row_exp_blockmax(cudaStream_t s, SplitOperand& op, int64_t rows) {
  if (!op.ex || !op.exb || rows <= 0) return cudaSuccess;
  row_exp_blockmax_kernel<<<(unsigned)((rows + 255) / 256), 256, 0, s>>>(op.ex, rows, op.exb);
  return cudaGetLastError();
}

cudaError_t launch_gemm_t3_pair(cudaStream_t s, const SplitOperand& A, const SplitOperand& B, const GemmArgs& g,
                                int max_ctas, const SplitOperand* A2, const SplitOperand* B2) {
  if (g.K2 > 0 && (!A2 || !B2)) return cudaErrorInvalidValue;
  if (g.K2 <= 0) A2 = &A, B2 = &B;
  if (g.ntiles <= 0) return cudaSuccess;
  static PerDeviceOnce attr_once;
  {
    const cudaError_t e =
        attr_once([] { return cudaFuncSetAttribute(gemm_t3_pair_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, t3p::SMEM_BYTES); });
    if (e != cudaSuccess) return e;
  }
  int cap = num_sms();
  if (max_ctas > 0 && max_ctas < cap) cap = max_ctas;
  const long long pairs = g.ntiles < cap / 2 ? g.ntiles : cap / 2;
  if (pairs < 1) return cudaErrorInvalidValue;
  gemm_t3_pair_kernel<<<(unsigned)(2 * pairs), kGemmThreads, t3p::SMEM_BYTES, s>>>(
      A.t_hi, A.t_lo, B.t_hi, B.t_lo, A2->t_hi, A2->t_lo, B2->t_hi, B2->t_lo, g);
  return cudaGetLastError();
}

// Tiles of width tn of a launch.
static long long oz_tiles(const GemmArgs& g, int tn) {
  if (g.enum_mode == kEnumFull) return (long long)g.mt * (((long long)g.nt * 32 + tn - 1) / tn);
  long long t = 0;
  const int SI = g.panel / oz::TM;
  for (int bi = 0; bi < g.mt; ++bi) {
    const int I = bi / SI, start = (I > g.band ? I - g.band : 0) * g.panel;
    t += ((bi + 1) * oz::TM - start + tn - 1) / tn;
  }
  return t;
}

cudaError_t launch_gemm_oz(cudaStream_t s, const SplitOperand& A, const SplitOperand& B, const GemmArgs& g,
                           int max_ctas) {
  if (g.mt <= 0 || (g.enum_mode == kEnumFull && g.nt <= 0)) return cudaSuccess;
  if (g.K % 16 || g.K > kSplitMaxK || (g.enum_mode != kEnumFull && g.enum_mode != kEnumBand) ||
      A.rows % 8 || B.rows % 8 || g.a_row0 % 8 || g.b_row0 % 8)
    return cudaErrorInvalidValue;
  static PerDeviceOnce attr_once;
  const cudaError_t e = attr_once([] {
    return cudaFuncSetAttribute(gemm_oz_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM_BYTES);
  });
  if (e != cudaSuccess) return e;
  int cap = num_sms();
  if (max_ctas > 0 && max_ctas < cap) cap = max_ctas;
  oz::Args a{};
  a.C = g.C;
  a.ldc = g.ldc;
  a.c_row0 = g.c_row0;
  a.c_col0 = g.c_col0;
  a.A = (const uint8_t*)A.dig + (int64_t)g.a_row0 * 32;
  a.B = (const uint8_t*)B.dig + (int64_t)g.b_row0 * 32;
  a.a_plane = A.rows * 32;
  a.b_plane = B.rows * 32;
  a.ea = A.ex + g.a_row0;
  a.eb = B.ex + g.b_row0;
  a.mode = g.enum_mode;
  a.band = g.band;
  a.panel = g.panel;
  a.mt = g.mt;
  a.n = g.nt * 32;
  a.k16 = g.K / 16;
  a.tri = g.tri;
  a.store = g.store;
  a.lower = g.lower_mask || g.enum_mode == kEnumBand;
  a.st = g.st;
  // the width whose waves end first: a tile takes about 30, 24 and 17 thousand cycles for K = 512
  constexpr struct { int tn, cost; } kWidths[] = {{96, 30}, {64, 24}, {32, 17}};
  long long best = 0;
  for (const auto& w : kWidths) {
    const long long t = oz_tiles(g, w.tn), cost = (t + cap - 1) / cap * w.cost;
    if (best == 0 || cost < best) {
      best = cost;
      a.tn = w.tn;
      a.ntiles = t;
    }
  }
  a.nbuf = a.tn == 32 ? 2 : 1;
  const int grid = (int)(a.ntiles < cap ? a.ntiles : cap);
  gemm_oz_kernel<<<grid, oz::kThreads, oz::SMEM_BYTES, s>>>(a);
  return cudaGetLastError();
}

}  // namespace exa
