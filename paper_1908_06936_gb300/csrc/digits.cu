// FP64 contractions on the fifth-generation tensor cores (steps a2, a7 and the prediction variance).
//
// FP64 units issue 1.26 TFLOP/s on this part, BF16 tensor cores 1,870: one 1,490th.  A product of two FP64
// matrices is therefore formed from BF16 ones.  Each row is scaled by a power of two so that |a| < 1 and cut
// into S = 8 signed 7-bit digits, a = sum_s d_s 2^(-6-7s), |d_s| <= 64, exact in BF16 (the error-free splitting
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).  Digit products are integers up to 2^12; group
// g = s + t sums at most 8 of them for each of K <= 512 columns, so every partial sum stays within 2^24 and FP32
// accumulation in TMEM is exact whatever its order.  The 36 products with g <= 7 are formed.  What is left out is
// a rounding-like error of about 2^-52 of the product of the two row maxima per pass, without a sign of its own
// except on the diagonal of A A^T, where the squares of the left-out digits add up to a bias: there the split's
// row sums sq put the left-out group g = 8 back.
#include "digits.cuh"

#include <cuda_bf16.h>

#include "ctx.cuh"
#include "tc_common.cuh"

namespace exa {

using namespace tc;

namespace dig {
constexpr int TM = 128, TN = kDigTN;
constexpr int kEpiWarps = 16, kThreads = 64 + 32 * kEpiWarps;

template <int S>
struct Cfg {
  static_assert(S == 4 || S == 8, "the drain's words");
  static constexpr int A_BYTES = TM * 32, B_BYTES = TN * 32;  // one digit plane of a 16-column step
  static constexpr int STAGE_BYTES = S * (A_BYTES + B_BYTES);
  static constexpr int STAGES = S == kDigSlices ? 4 : 9;
  static constexpr int SMEM = STAGES * STAGE_BYTES + 512;
  static constexpr int TMEM_COLS = S * TN;  // group g in columns [TN g, TN g + TN)
};
static_assert(Cfg<kDigSlices>::SMEM <= 232448 && Cfg<kDigLow>::SMEM <= 232448, "stages fit in shared memory");

// Lower-triangle enumeration of 128 x TN tiles: bands of kBand row blocks, each a rectangle left of the band's
// diagonal square (column tiles outer, rows inner: the tiles of one wave share operand rows in L2) and then the
// square's own lower tiles.  Row block b holds 2 (b + 1) column tiles.
constexpr int kBand = 16;
__device__ __forceinline__ void lower_tile(long long t, int mt, int& bi, int& bj) {
  int q = (int)(sqrtf((float)t) / kBand);  // t >= R (R + 1) with R = kBand q
  while (q > 0 && (long long)kBand * q * (kBand * q + 1) > t) --q;
  while ((long long)kBand * (q + 1) * (kBand * (q + 1) + 1) <= t) ++q;
  const int R = kBand * q, h = mt - R < kBand ? mt - R : kBand;
  t -= (long long)R * (R + 1);
  const long long rect = (long long)h * 2 * R;
  if (t < rect) {
    bj = (int)(t / h);
    bi = R + (int)(t % h);
    return;
  }
  const int u = (int)(t - rect);  // the square: row block R + b holds column tiles 2 R .. 2 (R + b) + 1
  int b = (int)sqrtf((float)u);
  while (b > 0 && b * (b + 1) > u) --b;
  while ((b + 1) * (b + 2) <= u) ++b;
  bi = R + b;
  bj = 2 * R + u - b * (b + 1);
}

struct Args {
  double* C;
  const double* Cin;
  int64_t ldc, ldcin;
  const uint8_t *A, *B;           // first plane, at the operand's row origin
  int64_t a_plane, b_plane;       // bytes between planes
  const int *ea, *eb, *sq;
  const DigitTask* tasks;         // kDigTasks
  int mt, nt;                     // row blocks, column tiles
  int shape, tri;
  int k16;
  uint32_t sign;                  // sign bit of the product's factor
  long long t0, ntiles;           // tiles [t0, ntiles)
  DevStatus* st;
};

// Operand rows and output of tile t.  diag: column minus row index of the tile's corner in a symmetric output, whose
// entries with diag + column > row are left out (kNoDiag: none).
constexpr int kNoDiag = -(1 << 30);
struct Tile {
  int64_t ar, br;
  double* C;
  const double* Cin;
  int64_t ldc, ldcin;
  int diag, bj;
};
__device__ __forceinline__ void tile_of(const Args& g, long long t, Tile& o) {
  if (g.shape == kDigTasks) {
    const DigitTask k = g.tasks[t];
    o.ar = k.a_row;
    o.br = k.b_row;
    o.C = k.C;
    o.Cin = k.diag == kDigStore ? nullptr : k.C;
    o.ldc = o.ldcin = k.ldc;
    o.diag = k.diag >= 0 ? k.diag : kNoDiag;
    o.bj = 0;
    return;
  }
  int bi, bj;
  if (g.shape == kDigRect) {
    bi = (int)(t % g.mt);
    bj = (int)(t / g.mt);
    if (g.tri) bj = g.nt - 1 - bj;  // the longest reductions first
    o.diag = kNoDiag;
  } else {
    lower_tile(t, g.mt, bi, bj);
    o.diag = bj * TN - bi * TM;
  }
  o.ar = (int64_t)bi * TM;
  o.br = (int64_t)bj * TN;
  o.C = g.C + o.ar + o.br * g.ldc;
  o.Cin = g.Cin ? g.Cin + o.ar + o.br * g.ldcin : nullptr;
  o.ldc = g.ldc;
  o.ldcin = g.ldcin;
  o.bj = bj;
}

__device__ __forceinline__ void timeout(DevStatus* st, volatile int* abort, int site) {
  *abort = 1;
  if (atomicExch(&st->timeout, 1) == 0) st->timeout_where = site;
}

// V 2^sh, rounded to nearest, for |V| < 2^63: the double is built from V's bits (FP64 instructions issue two lanes a
// cycle on an SM: one per output is what the epilogue can hide).  Below the normal range 0, above it infinity, and NaN
// where sh counts a row with kDigBad.
__device__ __forceinline__ double i63_to_f64_scaled(long long V, int sh) {
  const unsigned long long sign = (unsigned long long)V & 0x8000000000000000ull;
  const unsigned long long m = V < 0 ? (unsigned long long)(-V) : (unsigned long long)V;
  const int lz = __clzll((long long)m);
  const unsigned long long r = ((m << (lz - 1)) + 0x200) >> 10;  // leading one at bit 52 (53 after a carry)
  const int be = 1022 + 63 - lz + sh;                            // one below the biased exponent: the leading one adds it
  if (be >= 0x7FE) return __longlong_as_double((long long)(sign | (be > kDigBad / 2 ? 0x7FF8ull : 0x7FF0ull) << 48));
  if (m == 0 || be < 0) return __longlong_as_double((long long)sign);
  return __longlong_as_double((long long)(sign | (((unsigned long long)be << 52) + r)));
}

// FP32 integers as integers.  F2I converts 16 lanes a cycle on an SM, which for the 65,536 accumulators of a tile is a
// ninth of its MMA time, so half of the groups go by additions instead:
// |a| <= 2^22: the low bits of a + 1.5 2^23 (above, f32_to_int).
__device__ __forceinline__ uint32_t small_int_bits(float a) { return __float_as_uint(a + 12582912.0f); }  // + 0x4B400000
// One CTA per SM, persistent: warp 0 copies operand planes into a ring of 16-column stages, one thread of warp 1
// issues the MMAs, warps 2-17 drain TMEM into C.  The S B planes of a stage lie one after another and group g
// follows group g - 1 in TMEM, so A digit s against B digits 0 .. S-1-s is one run of columns (two MMAs where
// N > 256): 12 MMAs a step instead of 36.
//
// Bound: the tensor pipe (36 BF16 products per FP64 one: 52 TFLOP/s at the 1,872 of a burst).  Eight groups of a
// 128 x 64 tile fill TMEM (512 columns), and the tile has to be that large: each 16-column step moves 48 KB into
// shared memory for 1,152 cycles of MMA, 42 bytes a cycle, against the ~46 an SM was seen to take in.  So there is
// one accumulator set, and the drain's first part (TMEM to integers, four 32-bit words an output) is not hidden.
template <int S>
__global__ void __launch_bounds__(kThreads, 1) gemm_digits_kernel(const __grid_constant__ Args g) {
  using C_ = Cfg<S>;
  constexpr int A_BYTES = C_::A_BYTES, B_BYTES = C_::B_BYTES, STAGES = C_::STAGES, STAGE_BYTES = C_::STAGE_BYTES;
  extern __shared__ __align__(256) uint8_t smem[];
  uint64_t* full = (uint64_t*)(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accfull = empty + STAGES;
  uint64_t* accempty = accfull + 1;
  uint32_t* tmem_slot = (uint32_t*)(accempty + 1);
  volatile int* abort = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accfull, 1);
    mbar_init(accempty, 32 * kEpiWarps);
    *abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, C_::TMEM_COLS);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    // ---------------- copies: lane s < S brings A plane s, lane S + s B plane s ----------------
    int stage = 0;
    uint32_t phase = 0;
    int last_par[STAGES];
    for (int s = 0; s < STAGES; ++s) last_par[s] = -1;
    bool ok = true;  // the same for every lane
    for (long long t = g.t0 + blockIdx.x; t < g.ntiles && ok; t += gridDim.x) {
      Tile o;
      tile_of(g, t, o);
      const int steps = g.tri ? min(g.k16, (o.bj + 1) * (TN / 16)) : g.k16;
      const bool isA = lane < S;
      const uint8_t* src = isA ? g.A + (int64_t)lane * g.a_plane + o.ar * 32
                               : g.B + (int64_t)(lane - S) * g.b_plane + o.br * 32;
      const int64_t step_bytes = S * (isA ? g.a_plane : g.b_plane);
      const uint32_t off = isA ? lane * A_BYTES : S * A_BYTES + (lane - S) * B_BYTES;
      for (int kc = 0; kc < steps; ++kc) {
        if (lane == 0) {
          ok = mbar_wait(&empty[stage], phase ^ 1, abort);
          if (ok) mbar_expect_tx(&full[stage], STAGE_BYTES);
          else timeout(g.st, abort, 81);
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok) break;
        if (lane < 2 * S)
          bulk_load(smem_u32(smem + stage * STAGE_BYTES) + off, src, isA ? A_BYTES : B_BYTES, smem_u32(&full[stage]));
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
    int stage = 0;
    uint32_t phase = 0, it = 0;
    for (long long t = g.t0 + blockIdx.x; t < g.ntiles && !*abort; t += gridDim.x) {
      int steps = g.k16;
      if (g.tri) {
        Tile o;
        tile_of(g, t, o);
        steps = min(steps, (o.bj + 1) * (TN / 16));
      }
      if (!mbar_wait(accempty, (it & 1) ^ 1, abort)) {
        timeout(g.st, abort, 82);
        break;
      }
      fence_after();
      bool ok = true;
      for (int kc = 0; kc < steps; ++kc) {
        if (!mbar_wait(&full[stage], phase, abort)) {
          timeout(g.st, abort, 83);
          ok = false;
          break;
        }
        fence_after();
        const uint32_t sb = smem_u32(smem + stage * STAGE_BYTES);
        const uint64_t b0 = sdesc_flat(sb + S * A_BYTES);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const uint64_t a = sdesc_flat(sb + s * A_BYTES);
          const int n = TN * (S - s);
          // the first step's s = 0 writes every group, all others add
          const uint32_t acc = (kc | s) ? 1u : 0u;
          if (n > 256) {
            const int h = n / 2;  // a multiple of 32
            mma_bf16(tmem + s * TN, a, b0, idesc(kFmtBF16, TM, h), acc);
            mma_bf16(tmem + s * TN + h, a, b0 + (uint64_t)(h * 32 >> 4), idesc(kFmtBF16, TM, h), acc);
          } else {
            mma_bf16(tmem + s * TN, a, b0, idesc(kFmtBF16, TM, n), acc);
          }
        }
        mma_commit(&empty[stage]);
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
      if (!ok) break;
      mma_commit(accfull);
      ++it;
    }
  } else if (warp >= 2) {
    // ---------------- drain: warp w takes TMEM lanes 32 (w % 4).. and columns CH ((w - 2) / 4) .. ----------------
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const int r = quad * 32 + lane;
    constexpr int CH = TN * 4 / kEpiWarps;
    static_assert(CH == 16, "two lanes per column in the prefetch");
    uint32_t it = 0;
    for (long long t = g.t0 + blockIdx.x; t < g.ntiles; t += gridDim.x) {
      Tile o;
      tile_of(g, t, o);
      const int er = g.ea[o.ar + r];
      const int* ebp = g.eb + o.br + half * CH;
      double* cp = o.C + r + (int64_t)(half * CH) * o.ldc;
      const double* cip = o.Cin ? o.Cin + r + (int64_t)(half * CH) * o.ldcin : nullptr;
      const int last = r - o.diag - half * CH;  // columns up to this one of the half are on or below the diagonal
      if (o.Cin)  // this warp's lines of C into L2 while the products run: lane l column l / 2, rows 16 (l % 2) ..
        prefetch_l2(o.Cin + quad * 32 + 16 * (lane & 1) + (int64_t)(half * CH + (lane >> 1)) * o.ldcin);
      if (!__all_sync(0xffffffffu, mbar_wait(accfull, it & 1, abort))) {
        if (lane == 0) timeout(g.st, abort, 84);
        break;
      }
      fence_after();
      // groups 2p and 2p + 1 hold exact integers of weights 2^(-12-14p), 2^(-19-14p): a 32-bit word for both (at most
      // 7 2^28 + 2^24), a 64-bit one for groups 0-3 (S = 4: V, in units of the last) and one for 4-7, and V for all, in
      // units of 2^8 of the last
      long long V[CH];
      const uint32_t ta = tmem + ((uint32_t)(quad * 32) << 16) + half * CH;
#pragma unroll
      for (int h = 0; h < CH; h += 4) {
        uint32_t x[4][4];
#pragma unroll
        for (int p = 0; p < 4; ++p) tmem_ld4(ta + p * TN + h, x[p]);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int w01 = (int)(small_int_bits(__uint_as_float(x[0][j])) * 128u +  // modulo 2^32
                                small_int_bits(__uint_as_float(x[1][j])) - 129u * 0x4B400000u);
          V[h + j] = (long long)w01 * 16384 + (__float2int_rn(__uint_as_float(x[2][j])) * 128 +
                                               __float2int_rn(__uint_as_float(x[3][j])));
          if constexpr (S == 8) V[h + j] = V[h + j] << 20;
        }
        if constexpr (S == 8) {
#pragma unroll
          for (int p = 0; p < 4; ++p) tmem_ld4(ta + (4 + p) * TN + h, x[p]);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int w45 = __float2int_rn(__uint_as_float(x[0][j])) * 128 + __float2int_rn(__uint_as_float(x[1][j]));
            const int w67 = f32_to_int(__uint_as_float(x[2][j])) * 128 + f32_to_int(__uint_as_float(x[3][j]));
            V[h + j] += ((long long)w45 * 16384 + w67 + 128) >> 8;
          }
        }
      }
      fence_before();
      mbar_arrive(accempty);
      ++it;
      const int base = er - 12 - 7 * (S - 1) + (S == 8 ? 8 : 0);  // weight of V's unit, without the column's exponent
      if (S == 8 && o.diag > -TM) {  // the diagonal's left-out group
        const long long sq = (g.sq[o.ar + r] + (1 << 14)) >> 15;
#pragma unroll
        for (int j = 0; j < CH; ++j) V[j] += j == last ? sq : 0;
      }
#pragma unroll
      for (int j0 = 0; j0 < CH; j0 += 4) {
        asm volatile("" ::: "memory");  // four outputs at a time: more would not fit the registers
        double cv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) cv[j] = cip && j0 + j <= last ? cip[(int64_t)(j0 + j) * o.ldcin] : 0.0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int ec = ebp[j0 + j];
          double x = i63_to_f64_scaled(V[j0 + j], base + ec);
          x = __hiloint2double(__double2hiint(x) ^ (int)g.sign, __double2loint(x));
          if (j0 + j <= last) cp[(int64_t)(j0 + j) * o.ldc] = cip ? cv[j] + x : x;
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 1) {
    fence_after();
    tmem_dealloc(tmem, C_::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// Split: 16 rows per CTA, every value in a register.  Thread (row, group) of 16 x 16 holds K / 16 consecutive columns of
// its row, at most 32: all its loads are in flight at once, row maxima come from the bit patterns, and every eight
// columns give one 16-byte store per digit (eight lanes a 128-byte line).  Bound: the integer pipe (~55 instructions a
// value) and HBM (8 bytes read, 2 S written).  The splits of an n = 12,300 factorisation take 3.0 ms; through shared memory,
// with 64-bit digit arithmetic, they took 4.5 ms.
// ---------------------------------------------------------------------------
constexpr int kRows = 16, kSplitThreads = 256;

// v 2^c on the exponent field (0, infinities and NaNs as they are; below the normal range 0, above it infinity).
__device__ __forceinline__ double scale_exp(double v, int c) {
  const unsigned long long D = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((D >> 52) & 0x7FF);
  if (E == 0 || E == 0x7FF) return v;
  const int F = E + c;
  const unsigned long long rest = D & 0x800FFFFFFFFFFFFFull, sign = D & 0x8000000000000000ull;
  return __longlong_as_double((long long)(F <= 0      ? sign
                                          : F >= 0x7FF ? sign | 0x7FF0000000000000ull
                                                       : rest | ((unsigned long long)F << 52)));
}

// The S digits, as FP32 values, of a 2^(7S-1-e) rounded to an integer N (|a| < 2^e, so |N| <= 2^(7S-1); e = kDigBad: 0).
// With B = 64 (1 + 128 + .. + 128^(S-2)) added, the lower S - 1 base-128 digits of N + B are the balanced ones plus 64:
// no carry from digit to digit.  A digit f goes to FP32 as the low bits of 1.5 2^23 + f, by an addition (conversions run
// at a quarter of that rate).
template <int S>
__device__ __forceinline__ void digits_of(double a, int e, float (&d)[S]) {
  const int hi = __double2hiint(a);
  const int E = (hi >> 20) & 0x7FF;
  // a = M 2^(E-1075) with its 53-bit significand M: N = M 2^-sh, sh = 1075 - (7S - 1) + e - E >= 53 - (7S - 1); one
  // more bit is kept for the rounding
  const int sh = 1075 - (7 * S - 1) + e - E;
  const unsigned int mh = E ? ((unsigned int)hi & 0xFFFFFu) | 0x100000u : 0u, ml = E ? (unsigned int)__double2loint(a) : 0u;
  const unsigned long long M = (((unsigned long long)mh << 32) | ml) << 10;  // below 2^63
  const unsigned long long N = ((M >> min(sh + 9, 63)) + 1) >> 1;
  constexpr unsigned long long B = 64ull * ((1ull << (7 * (S - 1))) - 1) / 127;
  const unsigned long long x = hi < 0 ? B - N : B + N;
  constexpr float kMagic = 12582912.0f;
  // digits 1 .. S-1 from the 28 bits of each half
  const unsigned int lo = (unsigned int)x, up = S == 8 ? (unsigned int)(x >> 28) : 0u;
#pragma unroll
  for (int s = 1; s < S; ++s) {
    const int pos = 7 * (S - 1 - s);  // bit position in x
    const unsigned int w = S == 8 && s < 4 ? up >> (pos - 28) : lo >> pos;
    d[s] = __uint_as_float((w & 127u) | 0x4B400000u) - (kMagic + 64.0f);
  }
  d[0] = __int_as_float((int)((long long)x >> (7 * (S - 1))) + 0x4B400000) - kMagic;
}

template <int S>
__device__ __forceinline__ void split_body(const double* __restrict__ src, int64_t rs, int64_t cs, int64_t rows, int K,
                                           int lower, const int* __restrict__ colex, int colsign,
                                           const DigitOperand& op, int64_t out_row0) {
  __shared__ unsigned int s_max[kRows][17];
  __shared__ int s_sq[kRows][17];
  const int tid = threadIdx.x, r = tid & 15, g = tid >> 4;
  const int64_t row = (int64_t)blockIdx.x * kRows + r;
  const int octets = K / 8;  // dealt to the groups in runs: group g takes octets [o0, o1), at most four
  const int o0 = octets * g / 16, o1 = octets * (g + 1) / 16;
  const double* p = src + row * rs + (int64_t)(8 * o0) * cs;
  double v[4][8];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = 8 * (o0 + u) + j;
      v[u][j] = o0 + u < o1 && row < rows && !(lower && k > row) ? p[(int64_t)(8 * u + j) * cs] : 0.0;
    }
  if (colex) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (o0 + u < o1) {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[u][j] = scale_exp(v[u][j], colsign * colex[8 * (o0 + u) + j]);
      }
  }
  // The row's values are below 2^e in magnitude; only their exponents count, so the upper words do (a non-zero value's
  // is non-zero but for subnormals below 2^-1042, which count as 0).
  unsigned int mx = 0;
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int j = 0; j < 8; ++j) mx = max(mx, (unsigned int)__double2hiint(v[u][j]) & 0x7FFFFFFFu);
  s_max[r][g] = mx;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 16; ++q) mx = max(mx, s_max[r][q]);
  const int be = (int)(mx >> 20);
  const int e = be == 0x7FF ? kDigBad : mx == 0 ? 0 : be ? be - 1022 : -1021;
  const int64_t orow = out_row0 + row;
  uint8_t* out = op.dig + ((int64_t)(o0 >> 1) * S * op.rows) * 32 + (orow >> 3) * 256 + (orow & 7) * 16;
  float sq = 0.0f, sq4 = 0.0f;  // integers below 2^20
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    if (o0 + u >= o1 || row >= rows) continue;
    uint32_t w[S][4];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float d[S];
      digits_of<S>(v[u][j], e, d);
      if constexpr (S == 8) {
        sq = fmaf(d[1], d[7], fmaf(d[2], d[6], fmaf(d[3], d[5], sq)));
        sq4 = fmaf(d[4], d[4], sq4);
      }
#pragma unroll
      for (int s = 0; s < S; ++s) {  // exact in BF16: the upper half of the word
        const uint32_t b = __float_as_uint(d[s]);
        w[s][j >> 1] = (j & 1) ? __byte_perm(w[s][j >> 1], b, 0x7632) : b;
      }
    }
    const int o = o0 + u;
    uint8_t* po = out + (int64_t)((o >> 1) - (o0 >> 1)) * S * op.rows * 32 + (o & 1) * 128;
#pragma unroll
    for (int s = 0; s < S; ++s)
      *reinterpret_cast<uint4*>(po + (int64_t)s * op.rows * 32) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
  }
  s_sq[r][g] = (int)fmaf(2.0f, sq, sq4);
  __syncthreads();
  if (g == 0 && row < rows) {
    int sum = s_sq[r][0];
#pragma unroll
    for (int q = 1; q < 16; ++q) sum += s_sq[r][q];
    op.ex[orow] = e;
    op.sq[orow] = sum;
  }
}

template <int S>
__global__ void __launch_bounds__(kSplitThreads) digit_split_kernel(const double* __restrict__ src, int64_t rs,
                                                                    int64_t cs, int64_t rows, int K, int lower,
                                                                    const int* __restrict__ colex, int colsign,
                                                                    DigitOperand op, int64_t out_row0) {
  split_body<S>(src, rs, cs, rows, K, lower, colex, colsign, op, out_row0);
}

// Many pieces in one launch: blockIdx.y = piece, blockIdx.x = 16-row chunk of it.
template <int S>
__global__ void __launch_bounds__(kSplitThreads) digit_split_tasks_kernel(const DigitSplitTask* __restrict__ tasks,
                                                                          int K, DigitOperand op) {
  const DigitSplitTask t = tasks[blockIdx.y];
  if ((int64_t)blockIdx.x * kRows >= t.rows) return;  // uniform over the CTA, before any barrier
  split_body<S>(t.src, t.rs, t.cs, t.rows, K, t.lower, t.colex, t.colsign, op, t.out_row0);
}

}  // namespace dig

size_t digit_bytes(int64_t rows, int K, int S) {
  rows = round_up(rows, 8);
  return (size_t)(K / 16) * S * rows * 32 + 2 * (size_t)round_up(rows, 64) * sizeof(int);
}

void digit_layout(DigitOperand& op, void* base, int64_t rows, int K, int S) {
  rows = round_up(rows, 8);
  op.rows = rows;
  op.dig = (uint8_t*)base;
  op.ex = (int*)(op.dig + (size_t)(K / 16) * S * rows * 32);
  op.sq = op.ex + round_up(rows, 64);
}

template <int S>
static cudaError_t split_impl(cudaStream_t s, const double* src, int64_t rs, int64_t cs, int64_t rows, int K,
                              bool lower, const int* colex, int colsign, const DigitOperand& op, int64_t out_row0) {
  dig::digit_split_kernel<S><<<(unsigned)ceil_div(rows, dig::kRows), dig::kSplitThreads, 0, s>>>(
      src, rs, cs, rows, K, lower, colex, colsign, op, out_row0);
  return cudaGetLastError();
}

cudaError_t launch_digit_split(cudaStream_t s, const double* src, int64_t rs, int64_t cs, int64_t rows, int K, int S,
                               const DigitOperand& op, int64_t out_row0, bool lower, const int* colex, int colsign) {
  if (rows <= 0) return cudaSuccess;
  if (K <= 0 || K % 16 || K > kDigMaxK || out_row0 % 8 || out_row0 + rows > op.rows) return cudaErrorInvalidValue;
  if (S == kDigSlices) return split_impl<kDigSlices>(s, src, rs, cs, rows, K, lower, colex, colsign, op, out_row0);
  if (S == kDigLow) return split_impl<kDigLow>(s, src, rs, cs, rows, K, lower, colex, colsign, op, out_row0);
  return cudaErrorInvalidValue;
}

cudaError_t launch_digit_split_tasks(cudaStream_t s, const DigitSplitTask* d_tasks, int ntasks, int64_t max_rows,
                                     int K, int S, const DigitOperand& op) {
  if (ntasks <= 0 || max_rows <= 0) return cudaSuccess;
  if (K <= 0 || K % 16 || K > kDigMaxK || (S != kDigSlices && S != kDigLow)) return cudaErrorInvalidValue;
  constexpr int kMaxY = 65535;  // of a grid
  for (int t = 0; t < ntasks; t += kMaxY) {
    const dim3 grid((unsigned)ceil_div(max_rows, dig::kRows), (unsigned)(ntasks - t < kMaxY ? ntasks - t : kMaxY));
    if (S == kDigSlices)
      dig::digit_split_tasks_kernel<kDigSlices><<<grid, dig::kSplitThreads, 0, s>>>(d_tasks + t, K, op);
    else
      dig::digit_split_tasks_kernel<kDigLow><<<grid, dig::kSplitThreads, 0, s>>>(d_tasks + t, K, op);
  }
  return cudaGetLastError();
}

template <int S>
static cudaError_t gemm_impl(cudaStream_t s, const dig::Args& a, int max_ctas) {
  static PerDeviceOnce once;
  cudaError_t e = once([] {
    return cudaFuncSetAttribute(dig::gemm_digits_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                dig::Cfg<S>::SMEM);
  });
  if (e != cudaSuccess) return e;
  int cap = tc_num_sms();
  if (max_ctas > 0 && max_ctas < cap) cap = max_ctas;
  if (a.ntiles <= a.t0) return cudaSuccess;
  const int grid = (int)(a.ntiles - a.t0 < cap ? a.ntiles - a.t0 : cap);
  dig::gemm_digits_kernel<S><<<grid, dig::kThreads, dig::Cfg<S>::SMEM, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_gemm_digits(cudaStream_t s, const DigitGemm& g, int max_ctas) {
  if (g.m <= 0 || g.n <= 0) return cudaSuccess;
  if (g.m % dig::TM || g.n % dig::TN || g.K <= 0 || g.K % 16 || g.K > kDigMaxK || g.a_row0 % 8 || g.b_row0 % 8 ||
      g.a_row0 + g.m > g.A.rows || g.b_row0 + g.n > g.B.rows || (g.shape == kDigLower && g.m != g.n) || g.skip % dig::TM ||
      g.skip > (g.shape == kDigLower ? dig::kBand * dig::TM : 0))
    return cudaErrorInvalidValue;
  dig::Args a{};
  a.C = g.C;
  a.Cin = g.Cin;
  a.ldc = g.ldc;
  a.ldcin = g.ldcin;
  a.A = g.A.dig + g.a_row0 * 32;
  a.B = g.B.dig + g.b_row0 * 32;
  a.a_plane = g.A.rows * 32;
  a.b_plane = g.B.rows * 32;
  a.ea = g.A.ex + g.a_row0;
  a.eb = g.B.ex + g.b_row0;
  a.sq = g.A.sq + g.a_row0;
  a.mt = (int)(g.m / dig::TM);
  a.nt = (int)(g.n / dig::TN);
  a.shape = g.shape;
  a.tri = g.tri;
  a.k16 = g.K / 16;
  a.ntiles = g.shape == kDigLower ? (long long)a.mt * (a.mt + 1) : (long long)a.mt * a.nt;
  a.sign = g.neg ? 0x80000000u : 0u;
  const long long skip = g.skip / dig::TM;  // within the first band, where tiles go row block by row block
  a.t0 = skip * (skip + 1);
  a.st = g.st;
  if (g.S == kDigSlices) return gemm_impl<kDigSlices>(s, a, max_ctas);
  if (g.S == kDigLow) return gemm_impl<kDigLow>(s, a, max_ctas);
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm_digits_tasks(cudaStream_t s, const DigitTask* d_tasks, long long ntasks, int K, int S,
                                     const DigitOperand& A, const DigitOperand& B, bool neg, DevStatus* st) {
  if (ntasks <= 0) return cudaSuccess;
  if (K <= 0 || K % 16 || K > kDigMaxK) return cudaErrorInvalidValue;
  dig::Args a{};
  a.A = A.dig;
  a.B = B.dig;
  a.a_plane = A.rows * 32;
  a.b_plane = B.rows * 32;
  a.ea = A.ex;
  a.eb = B.ex;
  a.sq = A.sq;
  a.tasks = d_tasks;
  a.shape = kDigTasks;
  a.k16 = K / 16;
  a.ntiles = ntasks;
  a.sign = neg ? 0x80000000u : 0u;
  a.st = st;
  if (S == kDigSlices) return gemm_impl<kDigSlices>(s, a, 0);
  if (S == kDigLow) return gemm_impl<kDigLow>(s, a, 0);
  return cudaErrorInvalidValue;
}

}  // namespace exa
