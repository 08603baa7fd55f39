// FP64 factorisation and inversion of one diagonal block of up to 512 rows: the diagonal tiles that the MP variant of
// Section II-A, Fig. 1(d), keeps in double precision, and the serial part of the FP64 factorisation.  ONE cooperative
// launch on a few SMs.
//
// Every CTA of a cooperative grid works through the same steps, separated by grid-wide barriers (bounded waits; every
// CTA reaches every barrier; a failed pivot only turns values into NaN and is recorded in the status):
//
//   Cholesky, right-looking in 32-wide steps j (c0 = 32 j):
//     (a) CTA 0: D = chol(A_jj) (diag_leaf)
//     (b) L_rj = A_rj D^-T for the rows below by substitution, 8 rows a task, also into a scratch panel P
//     (c) A_rc -= L_rj L_cj^T: the next leaf first, on CTAs 0-3, which CTA 0 then factors while the others apply the
//         rest in 32 x 16 tasks (look-ahead) and the last CTA forms V_j = D^-1
//   Inverse W = L^-1 by doubling: a 2b block [[X_A, 0], [L_BA, X_B]] has inverse [[W_A, 0], [-W_B (L_BA W_A), W_B]],
//   formed for b = 32, 64, 128, 256 as two steps of 8 x 32 product tasks each.
//
// Bound: the chain of (a) and (b).  A dependent FP64 instruction costs 64 cycles here (an SM quarter issues half a lane
// a cycle) and FP64 work on one SM 2 multiply-adds a cycle, so a wide leaf is throughput bound (64 wide with its
// inverse: 88 us) and a narrow one pays for barriers (~1.5 us each).
//
// Outputs: L in the block's lower triangle (upper triangle untouched), log L_ii summed in a
// fixed order per 128 sub-tile, the 128 x 128 sub-tile inverses (row-major, zero above the
// diagonal) and, for a 512 block, its inverse (row-major, zero above the diagonal).
#include <math.h>

#include <type_traits>

#include "exa_internal.cuh"
#include "tc_common.cuh"

namespace exa {

constexpr int kDB = 512;        // largest block, leading dimension of its inverse
constexpr int kDW = 32;         // Cholesky step / inverse leaf
constexpr int kDThreads = 256;
constexpr int kDLd = kDW + 1;   // row stride of 32-wide tiles in shared memory (odd in doubles)
// scratch (doubles): the 32-inverses, the 256 x 256 product of the widest inverse step, then the current step's panel
constexpr int64_t kDiagT = (int64_t)(kDB / kDW) * kDW * kDW;
constexpr int64_t kDiagP = kDiagT + 256 * 256;
constexpr int64_t kDiagR = kDiagP + (int64_t)(kDB - kDW) * kDW;  // 1 / L_cc
constexpr int64_t kDiagBar = kDiagR + kDB;  // barrier counter, abort flag, lead counter
constexpr int64_t kDiagScratch = kDiagBar + 2;
constexpr long long kDiagSpin = 2000000000LL;  // bound of one barrier wait, SM clock cycles (~1 s)

struct DiagArgs {
  double* a;            // column-major matrix, element (i, j) at a[i + j * ld]
  int64_t ld, k0;       // block origin (k0, k0)
  double* w_sub;        // 128 x 128 row-major sub-tile inverses (w_all + (k0 / 128) 128^2)
  double* logdet;       // sub-tile log sums (logdet_part + k0 / 128)
  double* w2;           // 512 x 512 row-major inverse
  double* scr;          // kDiagScratch doubles
  DevStatus* st;
  int size;             // rows of the block, a multiple of 128 up to 512
};

// Waits, bounded, until *count >= target (every later wait is released by *abort).
__device__ __forceinline__ void wait_at_least(const unsigned int* count, unsigned int target, volatile int* abort,
                                              DevStatus* st, int site) {
  const long long t0 = clock64();
  while (*(const volatile unsigned int*)count < target && !*abort) {
    if (clock64() - t0 > kDiagSpin) {
      if (atomicExch((int*)abort, 1) == 0 && atomicExch(&st->timeout, 1) == 0) st->timeout_where = site;
      break;
    }
  }
  __threadfence();
}

// Grid-wide barrier of the cooperative launch (all CTAs co-resident) on a monotone counter.  On
// time-out the status records it, the abort flag releases every later wait, and the
// (then meaningless) results are discarded by the caller through the status.
__device__ __forceinline__ void grid_barrier(unsigned int* count, volatile int* abort, unsigned int target,
                                             DevStatus* st) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    wait_at_least(count, target, abort, st, 71);
  }
  __syncthreads();
}

// d positive, finite and not subnormal, on its bits (an FP64 comparison costs 64 cycles).
__device__ __forceinline__ bool normal_positive(double d) {
  return (unsigned int)(__double2hiint(d) >> 20) - 1u < 0x7FEu;
}

// 1 / sqrt(d) to rounding (0.51 ulp) for d with normal_positive(d), in ~35 integer instructions: the FP64 routine is a
// chain of seven FP64 instructions (~430 cycles on this part), once per column of the block.  d = m 2^2k with
// 1 <= m < 4; y0 = Y 2^-24 from the FP32 approximation; the residual E = 1 - m y0^2 (|E| < 2^-20) is exact but for a
// truncation at 2^-60, and y = y0 (1 + E / 2 + 3/8 E^2) (the Taylor series of (1 - E)^(-1/2); the next term is below
// 2^-61).
__device__ __forceinline__ double rsqrt_int(double d) {
  const unsigned int hi = (unsigned int)__double2hiint(d), lo = (unsigned int)__double2loint(d);
  const int e = (int)(hi >> 20);
  const int odd = (e & 1) ^ 1;         // the bias is odd: e - 1023 odd <=> e even
  const int k = (e - 1023 - odd) >> 1;
  // m 2^52 = Mh 2^32 + Ml
  const unsigned int mh = (hi & 0xFFFFFu) | 0x100000u;
  const unsigned int Mh = odd ? __funnelshift_l(lo, mh, 1) : mh, Ml = lo << odd;
  // in [1/2, 1], or an ulp above
  const float y0 = fmaxf(rsqrtf(__uint_as_float(((127u + odd) << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29))), 0.5f);
  const unsigned int yb = __float_as_uint(y0);
  const unsigned int Y = ((yb & 0x7FFFFFu) | 0x800000u) << ((yb >> 23) - 126u);
  const unsigned long long Q = (unsigned long long)Y * Y;  // below 2^49
  const unsigned int Ql = (unsigned int)Q, Qh = (unsigned int)(Q >> 32);
  // E 2^60 = (2^100 - M Q) 2^-40
  unsigned long long t = ((unsigned long long)Ml * Ql) >> 32;
  t = (unsigned long long)Mh * Ql + t;
  t = (unsigned long long)Ml * Qh + t;
  const long long E = (long long)((1ull << 60) - (((unsigned long long)(Mh * (unsigned long long)Qh) << 24) + (t >> 8)));
  const int E1 = (int)(E >> 20);
  const int sq = (int)(((long long)E1 * E1) >> 20);
  const long long h = (E + ((3 * sq) >> 2)) >> 1;
  // y 2^62 = Y 2^38 + Y h 2^-22
  const long long Yh = (long long)((unsigned long long)Y * (unsigned int)h) +
                       ((long long)((int)Y * (int)(h >> 32)) << 32);
  const unsigned long long Z = ((unsigned long long)Y << 38) + (unsigned long long)(Yh >> 22);
  return __longlong_as_double((long long)(((Z + 256) >> 9) + ((unsigned long long)(unsigned int)((1021 - k) << 20) << 32)));
}

// acc[u] += sum_k A(r + 8 u, k) B(c, k), k < K (a multiple of 32), for r = warp, c = lane: an 8 H x 32 tile with
// A(i, k) = pa[i ars + k acs], B(c, k) = pb[c brs + k bcs].  sA: 8 H x 33, sB: 32 x 33.
template <int H>
__device__ __forceinline__ void tile_gemm(double (&acc)[H], const double* pa, int64_t ars, int64_t acs,
                                          const double* pb, int64_t brs, int64_t bcs, int K, double* sA, double* sB) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int k0 = 0; k0 < K; k0 += kDW) {
    __syncthreads();  // the previous chunk (or the caller's use of sA / sB) is finished
    // consecutive threads walk the dimension with the smaller stride; L2 loads (ld.global.cg): the operands were
    // written by other CTAs since the last barrier
    double va[H], vb[4];
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const int idx = tid + u * kDThreads, i = acs == 1 ? idx >> 5 : idx % (8 * H), k = acs == 1 ? idx & 31 : idx / (8 * H);
      va[u] = __ldcg(pa + i * ars + (k0 + k) * acs);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = tid + u * kDThreads, c = bcs == 1 ? idx >> 5 : idx & 31, k = bcs == 1 ? idx & 31 : idx >> 5;
      vb[u] = __ldcg(pb + c * brs + (k0 + k) * bcs);
    }
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const int idx = tid + u * kDThreads, i = acs == 1 ? idx >> 5 : idx % (8 * H), k = acs == 1 ? idx & 31 : idx / (8 * H);
      sA[i * kDLd + k] = va[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int idx = tid + u * kDThreads, c = bcs == 1 ? idx >> 5 : idx & 31, k = bcs == 1 ? idx & 31 : idx >> 5;
      sB[c * kDLd + k] = vb[u];
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < kDW; ++k) {
      const double b = sB[lane * kDLd + k];
#pragma unroll
      for (int u = 0; u < H; ++u) acc[u] = fma(sA[(warp + 8 * u) * kDLd + k], b, acc[u]);
    }
  }
}

// A flag in shared memory between warps of one CTA: what was written before post is seen after await, which polls (a
// few tens of cycles; an mbarrier wait takes longer to wake) and gives up after ~2^24 polls.
__device__ __forceinline__ void post(int* flag, int v) {
  asm volatile("st.release.cta.shared.b32 [%0], %1;" ::"r"(tc::smem_u32(flag)), "r"(v) : "memory");
}
__device__ __forceinline__ void await(const int* flag, int v) {
  int got;
  for (int n = 0; n < 1 << 24; ++n) {
    asm volatile("ld.acquire.cta.shared.b32 %0, [%1];" : "=r"(got) : "r"(tc::smem_u32(flag)) : "memory");
    if (got == v) return;
  }
}

// (a) of step j on one CTA: chol of the 32 x 32 block at c0, with a lane per row and the columns spread over four warps,
// one per SM quarter (column c in register c / 4 of warp c mod 4).  The owner of column c scales it by
// r_c = 1 / sqrt(d_c) and publishes it in shared memory (done[c] = j + 1); every warp then
// subtracts it from its own columns, the owner of column c + 1 that one first, which it publishes before the others:
// the chain per column is one multiply-add, one shuffle, one reciprocal square root and one product.
__device__ void diag_leaf(const DiagArgs& g, int j, double* S, int* done) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t c0 = g.k0 + (int64_t)j * kDW;
  double* A = g.a + c0 + c0 * g.ld;
  const int epoch = j + 1;
  // S[c kDLd + i] = A(i, c), later L(i, c)
  for (int idx = tid; idx < kDW * kDW; idx += kDThreads) {
    const int i = idx & (kDW - 1), c = idx / kDW;
    S[c * kDLd + i] = i >= c ? __ldcg(A + i + (int64_t)c * g.ld) : 0.0;
  }
  __syncthreads();
  if (warp < 4) {
    double a[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) a[u] = S[(warp + 4 * u) * kDLd + lane];
    // column c, in a0 of this warp: pivot, scale, publish
    auto publish = [&](int c, double a0) {
      const double d = __shfl_sync(0xffffffffu, a0, c);
      double r;
      if (normal_positive(d)) {  // uniform across the warp
        r = rsqrt_int(d);
      } else if (d > 0.0 && isfinite(d)) {
        r = rsqrt(d);
      } else {
        if (lane == 0) {
          atomicMin(&g.st->pivot, (long long)(c0 + c));
          atomicExch(&g.st->info, 1);
        }
        r = NAN;  // the rest becomes NaN; every barrier is still reached
      }
      S[c * kDLd + lane] = lane >= c ? a0 * r : 0.0;
      __syncwarp();
      if (lane == 0) {
        post(done + c, epoch);
        g.scr[kDiagR + j * kDW + c] = r;
      }
    };
    if (warp == 0) publish(0, a[0]);
    // columns 4 q4 .. 4 q4 + 3, of which this warp's is a[0]; N: registers that may hold later columns (a predicated-off
    // multiply-add takes its 64 cycles too, so the count is a constant of the code, in four versions)
    auto quad = [&](auto width, int q4) {
      constexpr int N = decltype(width)::value;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int c = 4 * q4 + q;
        if (warp != q) await(done + c, epoch);
        const double* col = S + c * kDLd;
        const double lic = col[lane];
        // the next column's owner: warp q + 1 (its a[0]), or warp 0 (its a[1]) at the end of the four
        const int nextw = (q + 1) & 3;
        constexpr int kLast = N > 1 ? 1 : 0;
        const int nu = q == 3 ? kLast : 0;
        if (warp == nextw && c + 1 < kDW) {
          a[nu] = fma(-lic, col[c + 1], a[nu]);
          publish(c + 1, a[nu]);
        }
        if (warp > nextw && q < 3) a[0] = fma(-lic, col[warp + 4 * q4], a[0]);  // still to come in these four
#pragma unroll
        for (int u = 1; u < N; ++u)
          if (!(q == 3 && u == 1 && warp == 0)) a[u] = fma(-lic, col[min(warp + 4 * (q4 + u), kDW - 1)], a[u]);
      }
#pragma unroll
      for (int u = 0; u + 1 < N; ++u) a[u] = a[u + 1];
    };
    for (int q4 = 0; q4 < 2; ++q4) quad(std::integral_constant<int, 8>{}, q4);
    for (int q4 = 2; q4 < 4; ++q4) quad(std::integral_constant<int, 6>{}, q4);
    for (int q4 = 4; q4 < 6; ++q4) quad(std::integral_constant<int, 4>{}, q4);
    for (int q4 = 6; q4 < 8; ++q4) quad(std::integral_constant<int, 2>{}, q4);
  }
  __syncthreads();
  for (int idx = tid; idx < kDW * kDW; idx += kDThreads) {
    const int i = idx & (kDW - 1), c = idx / kDW;
    if (i >= c) A[i + (int64_t)c * g.ld] = S[c * kDLd + i];
  }
}

// V_j = D^-1 of the factored block j (row-major, zero above the diagonal), on one CTA: the eliminations applied to the
// identity, a lane per row and four columns a warp, B_i -= (L_ic r_c) B_c; rows of V are r_i B_i.  S: 32 x 33.
__device__ void diag_leaf_inverse(const DiagArgs& g, int j, double* S) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t c0 = g.k0 + (int64_t)j * kDW;
  const double* A = g.a + c0 + c0 * g.ld;
  const double* R = g.scr + kDiagR + j * kDW;
  __syncthreads();
  for (int idx = tid; idx < kDW * kDW; idx += kDThreads) {
    const int i = idx & (kDW - 1), c = idx / kDW;
    S[c * kDLd + i] = i > c ? __ldcg(A + i + (int64_t)c * g.ld) * __ldcg(R + c) : 0.0;
  }
  const double ri = __ldcg(R + lane);
  __syncthreads();
  double b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) b[u] = lane == warp + 8 * u ? 1.0 : 0.0;
  for (int c = 0; c < kDW; ++c) {
    const double t = S[c * kDLd + lane];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (warp + 8 * u <= c) b[u] = fma(-t, __shfl_sync(0xffffffffu, b[u], c), b[u]);
  }
  double* Vg = g.scr + (int64_t)j * kDW * kDW;
#pragma unroll
  for (int u = 0; u < 4; ++u) Vg[lane * kDW + warp + 8 * u] = warp + 8 * u <= lane ? b[u] * ri : 0.0;
  __syncthreads();
}

__global__ void __launch_bounds__(kDThreads) diag_block_kernel(const __grid_constant__ DiagArgs g) {
  __shared__ double S[kDW * kDLd];         // the leaf, or its inverse
  __shared__ double sA[16 * kDLd], sB[kDW * kDLd];
  __shared__ int done[kDW];
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned int* bar = (unsigned int*)(g.scr + kDiagBar);
  volatile int* abort = (volatile int*)(bar + 1);
  unsigned int* leadcnt = bar + 2;  // lead tasks finished by CTAs other than 0 (monotone)
  unsigned int nbar = 0, lead_target = 0;
  auto sync_all = [&]() { grid_barrier(bar, abort, (++nbar) * (unsigned int)G, g.st); };
  const int64_t ld = g.ld, k0 = g.k0;
  double* a = g.a;
  double* P = g.scr + kDiagP;  // the current step's panel below the leaf, row-major, 32 wide
  if (tid < kDW) done[tid] = 0;
  __syncthreads();

  // ---------------- Cholesky in 32-wide steps ----------------
  if (b == 0) diag_leaf(g, 0, S, done);
  sync_all();
  const int size = g.size, nsteps = size / kDW;
  for (int j = 0; j + 1 < nsteps; ++j) {
    const int64_t c0 = k0 + (int64_t)j * kDW, r0 = c0 + kDW;
    const int below = size - (j + 1) * kDW;  // rows of the block below step j
    // (b) x D^T = A(r, c0 ..) row by row, eight rows a task: warps 0-3 (an SM quarter each) take two rows, 16 lanes a
    //     row with columns q and q + 16; step c: x_c = a_c r_c, then a_l -= x_c L_lc for l > c
    for (int t = b; t < below / 8; t += G) {
      double* rows = a + r0 + 8 * t + c0 * ld;
      __syncthreads();
      {
        const double v = __ldcg(rows + (tid & 7) + (int64_t)(tid >> 3) * ld);
        double vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = __ldcg(a + c0 + lane + (c0 + warp + 8 * u) * ld);  // D(lane, warp + 8 u)
        sA[(tid & 7) * kDLd + (tid >> 3)] = v;
#pragma unroll
        for (int u = 0; u < 4; ++u) sB[(warp + 8 * u) * kDLd + lane] = vv[u];
        if (warp == 7) sA[8 * kDLd + lane] = __ldcg(g.scr + kDiagR + j * kDW + lane);
      }
      __syncthreads();
      if (warp < 4) {
        const int r = 2 * warp + (lane >> 4), q = lane & 15;
        double x0 = sA[r * kDLd + q], x1 = sA[r * kDLd + q + 16];
#pragma unroll
        for (int c = 0; c < kDW; ++c) {
          const double rc = sA[8 * kDLd + c];
          const double* col = sB + c * kDLd;
          if (c < 16) {
            const double l0 = q > c ? col[q] : 0.0, l1 = col[q + 16];
            if (q == c) x0 *= rc;
            const double xc = __shfl_sync(0xffffffffu, x0, c, 16);
            x0 = fma(-xc, l0, x0);
            x1 = fma(-xc, l1, x1);
          } else {
            const double l1 = q + 16 > c ? col[q + 16] : 0.0;
            if (q + 16 == c) x1 *= rc;
            x1 = fma(-__shfl_sync(0xffffffffu, x1, c - 16, 16), l1, x1);
          }
        }
        sA[r * kDLd + q] = x0;
        sA[r * kDLd + q + 16] = x1;
      }
      __syncthreads();
      P[(8 * t + warp) * kDW + lane] = sA[warp * kDLd + lane];
      rows[(tid & 7) + (int64_t)(tid >> 3) * ld] = sA[(tid & 7) * kDLd + (tid >> 3)];
    }
    sync_all();
    // (c) the next leaf: rows 8 q .. of it on CTA q (CTA 0 where the grid is smaller); the others count their part on
    //     a monotone counter that CTA 0 waits for before the leaf
    int foreign = 0;
    for (int q = 0; q < 4; ++q) {
      const int owner = q < G ? q : 0;
      foreign += owner != 0;
      if (owner != b) continue;
      __syncthreads();
      for (int idx = tid; idx < kDW * kDW; idx += kDThreads) sB[(idx >> 5) * kDLd + lane] = __ldcg(P + idx);
      __syncthreads();
      const int i = 8 * q + warp;
      double* pc = a + (r0 + i) + (r0 + lane) * ld;
      double s0 = lane <= i ? __ldcg(pc) : 0.0;
#pragma unroll 8
      for (int k = 0; k < kDW; ++k) s0 = fma(-sB[i * kDLd + k], sB[lane * kDLd + k], s0);
      if (lane <= i) *pc = s0;
    }
    if (b != 0 && b < 4) {
      __syncthreads();
      if (tid == 0) {
        __threadfence();
        atomicAdd(leadcnt, 1u);
      }
    }
    lead_target += (unsigned int)foreign;
    if (b == 0) {
      if (tid == 0) wait_at_least(leadcnt, lead_target, abort, g.st, 72);
      __syncthreads();
      diag_leaf(g, j + 1, S, done);
    } else {
      if (b == G - 1) diag_leaf_inverse(g, j, S);
      // A_rc -= L_r L_c^T over 32-row blocks R and 16-wide column strips s <= 2 R + 1, but for the leaf's (R = 0):
      // block R has 2 R + 2 tasks, numbered from R (R + 1) - 2 on; lanes along the rows of the column-major matrix.
      // The CTA that forms V_j takes its share of the last ones.
      const int nr = below / kDW, nt = nr * (nr + 1) - 2;
      for (int t = b - 1; t < nt; t += G - 1) {
        int R = (int)sqrtf((float)(t + 2));
        while (R * (R + 1) > t + 2) --R;
        while ((R + 1) * (R + 2) <= t + 2) ++R;
        const int s = t + 2 - R * (R + 1);
        double acc[2] = {0.0, 0.0};
        tile_gemm<2>(acc, P + s * 16 * kDW, kDW, 1, P + R * kDW * kDW, kDW, 1, kDW, sA, sB);
        const int i = R * kDW + lane;
        double* pc = a + (r0 + i) + (r0 + s * 16 + warp) * ld;
        const bool lo = s * 16 + warp <= i, hi = s * 16 + warp + 8 <= i;
        const double v0 = lo ? __ldcg(pc) : 0.0, v1 = hi ? __ldcg(pc + 8 * ld) : 0.0;
        if (lo) *pc = v0 - acc[0];
        if (hi) pc[8 * ld] = v1 - acc[1];
      }
    }
    sync_all();
  }

  // ---------------- log-determinant parts, leaves of the inverse ----------------
  for (int s4 = b; s4 < size / 128; s4 += G) {  // uniform over the CTA
    __syncthreads();
    if (tid < 128) {
      const int64_t r = k0 + 128 * s4 + tid;
      sB[tid] = log(__ldcg(a + r + r * ld));
    }
    __syncthreads();
    if (warp == 0) {  // in a fixed order
      double s = (sB[lane] + sB[lane + 32]) + (sB[lane + 64] + sB[lane + 96]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) g.logdet[s4] = s;
    }
  }
  if (b == G - 1) diag_leaf_inverse(g, nsteps - 1, S);
  sync_all();  // the last leaf's inverse
  double* w2 = g.w2;
  // W2 <- zero above the diagonal, the 32-inverses on the diagonal (other lower entries later)
  for (int64_t idx = (int64_t)b * kDThreads + tid; idx < (int64_t)size * kDB; idx += (int64_t)G * kDThreads) {
    const int r = (int)(idx / kDB), c = (int)(idx % kDB);
    if (c >= size) continue;
    if (c > r) {
      w2[idx] = 0.0;
    } else if (r / kDW == c / kDW) {
      const double* V = g.scr + (int64_t)(r / kDW) * kDW * kDW;
      w2[idx] = __ldcg(V + (r % kDW) * kDW + (c % kDW));
    }
  }
  sync_all();

  // ---------------- inverse by doubling: widths h = 32, 64, 128, 256 ----------------
  // Tasks run from the longest reductions to the shortest in the first half of the list and back in the second, so
  // that a CTA with two has a long and a short one.
  double* T = g.scr + kDiagT;  // h x h products, row-major
  auto fold = [](int q, int n) { return q < n / 2 ? q : n - 1 - (q - n / 2); };
  // (a smaller block is the last of its matrix: only its 128 sub-tile inverses are wanted)
  for (int h = kDW; h < (size == kDB ? kDB : 128); h *= 2) {
    const int pairs = size / (2 * h), nr = h / 8, nc = h / kDW;  // blocks of width 2h; tiles of one h x h product
    // first product: T_p = L_BA W_A  (L_BA: rows p 2h + h .., columns p 2h ..; W_A lower, row-major in w2)
    for (int t = b; t < pairs * nr * nc; t += G) {
      const int p = t % pairs, q = t / pairs, ti = q % nr, tj = fold(q / nr, nc);
      const int64_t o = (int64_t)p * 2 * h;  // block origin within the block
      double acc[1] = {0.0};
      // T(r, c) = sum_k L(o + h + r, o + k) W(o + k, o + c): W_A(k, c) = 0 for k < c
      const int kstart = tj * kDW;
      tile_gemm<1>(acc, a + (k0 + o + h + ti * 8) + (k0 + o + kstart) * ld, 1, ld,
                w2 + (o + kstart) * kDB + (o + tj * kDW), 1, kDB, h - kstart, sA, sB);
      double* Tp = T + (int64_t)p * h * h;
      Tp[(ti * 8 + warp) * h + tj * kDW + lane] = acc[0];
    }
    sync_all();
    // second product: W_BA = -W_B T_p  (W_B lower, row-major in w2 at (o + h, o + h), zero above its diagonal)
    for (int t = b; t < pairs * nr * nc; t += G) {
      const int p = t % pairs, q = t / pairs, tj = q % nc, ti = nr - 1 - fold(q / nc, nr);
      const int64_t o = (int64_t)p * 2 * h;
      const double* Tp = T + (int64_t)p * h * h;
      double acc[1] = {0.0};
      // W_BA(r, c) = -sum_k W_B(r, k) T(k, c): W_B(r, k) = 0 for k > r
      const int kend = (ti * 8 + 8 + kDW - 1) / kDW * kDW;
      tile_gemm<1>(acc, w2 + (o + h + ti * 8) * kDB + (o + h), kDB, 1, Tp + tj * kDW, 1, h, kend, sA, sB);
      w2[(o + h + ti * 8 + warp) * kDB + o + tj * kDW + lane] = -acc[0];
    }
    sync_all();
  }

  // ---------------- the 128 sub-tile inverses (diagonal blocks of W2) ----------------
  for (int64_t idx = (int64_t)b * kDThreads + tid; idx < (int64_t)size * 128; idx += (int64_t)G * kDThreads) {
    const int s = (int)(idx / (128 * 128)), rc = (int)(idx % (128 * 128)), r = rc / 128, c = rc % 128;
    g.w_sub[idx] = __ldcg(w2 + (int64_t)(128 * s + r) * kDB + 128 * s + c);
  }
}

size_t diag_block_scratch_doubles() { return (size_t)kDiagScratch; }

cudaError_t launch_diag_block(cudaStream_t s, double* a, int64_t ld, int64_t k0, double* w_sub, double* logdet_part,
                              double* w2, double* scratch, DevStatus* st, int grid, int size) {
  // at least 116 KB of shared memory, so that no SM holds two CTAs (the FP64 pipe of an SM is
  // the resource: two CTAs on one SM would leave another idle)
  const size_t smem = (size_t)116 * 1024;
  static PerDeviceOnce attr_once;
  cudaError_t e = attr_once([&] {
    return cudaFuncSetAttribute(diag_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
  if (e != cudaSuccess) return e;
  if (grid < 2) grid = 2;  // CTA 0 runs the leaves; the updates need at least one more CTA
  e = cudaMemsetAsync(scratch + kDiagBar, 0, 2 * sizeof(double), s);
  if (e != cudaSuccess) return e;
  DiagArgs g{a, ld, k0, w_sub, logdet_part, w2, scratch, st, size};
  void* args[] = {&g};
  // cooperative launch: every CTA is resident at once, so the grid barriers cannot wait on an
  // unscheduled CTA
  return cudaLaunchCooperativeKernel((const void*)diag_block_kernel, grid, kDThreads, args, smem, s);
}

}  // namespace exa
