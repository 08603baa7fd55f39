// FP64 factorisation and inversion of diagonal blocks: of up to 512 rows on a cooperative grid (the tiles that the MP
// variant of Section II-A, Fig. 1(d), keeps in double precision, and the serial part of the FP64 factorisation), and of
// many 128 x 128 tiles at once, a thread-block cluster each (the batched paths).
//
// The CTAs of a group (the grid, or a cluster) work through the same steps, separated by group-wide barriers (a failed
// pivot only turns values into NaN and is recorded in the status, so every CTA reaches every barrier).  In 32-wide
// steps j (c0 = 32 j):
//     (b) L_rj = A_rj D_j^-T for the rows below by substitution, 8 or 16 rows a task; W_j-1 = V_j-1 T_j-1 (see below)
//     (c) A_rc -= L_rj L_cj^T: the next leaf first, on a few CTAs, which CTA 0 then factors, D_j+1 =
//         chol(A_j+1,j+1) (diag_leaf), while the others apply the rest in 32 x 16 tiles and the last ones form V_j = D_j^-1
//   The inverse W = L^-1 keeps pace, one step behind: row block i of W starts as zero and (c) adds
//   T_i -= L_i,j-1 W_j-1 in tiles of the same shape; then W_i = V_i T_i.  After the last leaf only the last row blocks
//   are left.
//
// Bound: the chain of (b) and (c), 26 us a step: leaf 14, rows 4.3, two barriers 2.8, the next leaf's update and its
// hand-over 4.1.  An FP64 instruction keeps its SM quarter busy for 64 cycles here, so FP64 work on one SM does 2
// multiply-adds a cycle: a wide leaf is throughput bound (64 wide with its inverse: 88 us) and a narrow one pays for
// barriers.  A 512 block takes 427 us on 104 CTAs, 464 on 64, 698 on 32, 1,180 on 16; with the columns of a leaf dealt
// out one by one and the inverse by doubling after the last leaf, 610 on 64.  A 128 tile on a cluster of 4 takes 128 us;
// on one CTA, as a blocked factorisation and then the inverse, 570.
//
// Outputs: L in the block's lower triangle (upper triangle untouched), log L_ii summed in a fixed order per 128
// sub-tile, the 128 x 128 sub-tile inverses (row-major, zero above the diagonal) and, for a 512 block, its inverse
// (row-major, zero above the diagonal).
#include <math.h>

#include "exa_internal.cuh"
#include "gemm_tc.cuh"
#include "shares.cuh"
#include "tc_common.cuh"

namespace exa {

constexpr int kDB = 512;        // largest block, leading dimension of its inverse
constexpr int kDSub = 128;      // sub-tile
constexpr int kDW = 32;         // step
constexpr int kDThreads = 256;
constexpr int kDLd = kDW + 1;   // row stride of 32-wide tiles in shared memory (odd in doubles)
constexpr int kDLead = 8;       // CTAs of a leaf's last update, at most (then 4 rows each)
constexpr int64_t kDiagScratch = 2;  // doubles: barrier counter, abort flag, lead counter
constexpr long long kDiagSpin = 2000000000LL;  // bound of one barrier wait, SM clock cycles (~1 s)

struct DiagArgs {
  double* a;        // column-major matrix, element (i, j) at a[i + j * ld]
  int64_t ld, k0;   // block origin (k0, k0)
  double* w;        // inverse, row-major, size x size, leading dimension ldw
  int ldw;
  int inv;          // the inverse is formed within diagonal blocks of this width: size, or kDSub
  double* w_sub;    // also the 128 x 128 sub-tile inverses (row-major), or null
  double* logdet;   // sub-tile log sums
  DevStatus* st;
  int size;         // rows of the block, a multiple of 128 up to 512
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

// The CTAs of a cooperative grid (all co-resident), with barriers on a monotone counter.  On time-out the status
// records it, the abort flag releases every later wait, and the (then meaningless) results are discarded by the caller
// through the status.
struct GridGroup {
  unsigned int *bar, *leadcnt;  // leadcnt: lead tasks finished by CTAs other than 0 (monotone)
  volatile int* abort;
  DevStatus* st;
  unsigned int nbar = 0, nlead = 0;
  __device__ GridGroup(double* scr, DevStatus* s)
      : bar((unsigned int*)scr), leadcnt((unsigned int*)scr + 2), abort((volatile int*)scr + 1), st(s) {}
  __device__ int size() const { return (int)gridDim.x; }
  __device__ int rank() const { return (int)blockIdx.x; }
  __device__ void sync() {
    ++nbar;
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(bar, 1u);
      wait_at_least(bar, nbar * gridDim.x, abort, st, 71);
    }
    __syncthreads();
  }
  // CTA 0 goes on once the others have finished their part of the next leaf; no other waits
  __device__ void lead_sync() {
    const unsigned int foreign = min(gridDim.x, (unsigned int)kDLead) - 1;
    nlead += foreign;
    __syncthreads();
    if (threadIdx.x == 0) {
      if (blockIdx.x == 0) {
        wait_at_least(leadcnt, nlead, abort, st, 72);
      } else if (blockIdx.x <= foreign) {
        __threadfence();
        atomicAdd(leadcnt, 1u);
      }
    }
    __syncthreads();
  }
};

// A thread-block cluster.
struct ClusterGroup {
  __device__ int size() const {
    unsigned int n;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    return (int)n;
  }
  __device__ int rank() const {
    unsigned int r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
  }
  __device__ void sync() {
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  __device__ void lead_sync() { sync(); }
};

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

// D_j = chol of the 32 x 32 block at step j, on one CTA: a lane per row, the columns on four warps, one per SM quarter:
// warp w holds columns 4 w .. 4 w + 3 and 16 + 4 w .. 16 + 4 w + 3.  Finished columns go to shared memory, where the
// other warps wait for them (done[c] = j + 1) and subtract them from their own.  The chain per column is a product, a
// multiply-add, a shuffle and a reciprocal square root (~500 cycles), within one warp but for every fourth column; with
// the columns dealt out one by one the hand-over cost ~300 cycles at each.  1 / L_cc goes to the diagonal of w.
__device__ void diag_leaf(const DiagArgs& g, int j, double* S, int* done) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t c0 = g.k0 + (int64_t)j * kDW;
  double* A = g.a + c0 + c0 * g.ld;
  const int epoch = j + 1;
  // S[c kDLd + i] = A(i, c), later L(i, c)
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = warp + 8 * u;
    S[c * kDLd + lane] = lane >= c ? __ldcg(A + lane + (int64_t)c * g.ld) : 0.0;
  }
  __syncthreads();
  if (warp < 4) {
    double x0[4], x1[4];
    int polls = tc::kFlagPolls;  // of all the waits below
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x0[u] = S[(4 * warp + u) * kDLd + lane];
      x1[u] = S[(16 + 4 * warp + u) * kDLd + lane];
    }
    __syncwarp();
    // x(columns cb ..) minus the contributions of columns 4 q .. 4 q + 3
    auto subtract = [&](double (&x)[4], int cb, int q) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int c = 4 * q + v;
        tc::await(done + c, epoch, polls);
        const double* col = S + c * kDLd;
        const double lic = col[lane];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = fma(-lic, col[cb + u], x[u]);
      }
    };
    double rr = 0.0;  // 1 / L_cc of column c = lane, if it is one of this warp's
    auto factor = [&](double (&x)[4], int cb) {
      // (the next column's pivot and its reciprocal root come before everything else that follows from a column)
      double d = __shfl_sync(0xffffffffu, x[0], cb), r = rsqrt_int(d);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = cb + u;
        if (!normal_positive(d)) {  // uniform across the warp
          r = rsqrt(d);
          if (!(d > 0.0) || !isfinite(d)) {
            if (lane == 0) {
              atomicMin(&g.st->pivot, (long long)(c0 + c));
              atomicExch(&g.st->info, 1);
            }
            r = NAN;  // the rest becomes NaN; every barrier is still reached
          }
        }
        const double t = x[u] * r;
        const double l = lane >= c ? t : 0.0;
        if (lane == c) rr = r;
        S[c * kDLd + lane] = l;
        if (u < 3) {
          d = __shfl_sync(0xffffffffu, fma(-l, l, x[u + 1]), c + 1);
          r = rsqrt_int(d);
        }
#pragma unroll
        for (int v = u + 1; v < 4; ++v) x[v] = fma(-l, __shfl_sync(0xffffffffu, l, cb + v), x[v]);
        __syncwarp();
        if (lane == 0) tc::post(done + c, epoch);
      }
    };
    // the columns that this warp factors next come first; the later ones fill the time while other warps factor
    for (int q = 0; q < warp; ++q) {
      subtract(x0, 4 * warp, q);
      if (q + 1 < warp) subtract(x1, 16 + 4 * warp, q);
    }
    factor(x0, 4 * warp);
    for (int q = max(warp - 1, 0); q < 4 + warp; ++q) subtract(x1, 16 + 4 * warp, q);
    factor(x1, 16 + 4 * warp);
    tc::report_waits(polls, g.st, 73);
    if ((lane & 15) >> 2 == warp) g.w[(int64_t)(j * kDW + lane) * (g.ldw + 1)] = rr;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = warp + 8 * u;
    if (lane >= c) A[lane + (int64_t)c * g.ld] = S[c * kDLd + lane];
  }
}

// Element (r, c) of the inverse, both counted within the block.
__device__ __forceinline__ void put_inverse(const DiagArgs& g, int r, int c, double v) {
  g.w[(int64_t)r * g.ldw + c] = v;
  if (g.w_sub && r / kDSub == c / kDSub) g.w_sub[(int64_t)r * kDSub + c % kDSub] = v;
}

// Columns 8 q .. 8 q + 7 of V_j = D_j^-1 into the diagonal block of w: the eliminations applied to the identity, a lane
// per row and a column a warp, B_i -= (L_ic r_c) B_c; rows of V are r_i B_i.  S: 32 x 33.
__device__ void diag_leaf_inverse(const DiagArgs& g, int j, int q, double* S) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t c0 = g.k0 + (int64_t)j * kDW;
  const double* A = g.a + c0 + c0 * g.ld;
  const double* R = g.w + (int64_t)(j * kDW) * (g.ldw + 1);  // the diagonal: 1 / L_cc
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = warp + 8 * u;
    S[c * kDLd + lane] = lane > c ? __ldcg(A + lane + (int64_t)c * g.ld) * __ldcg(R + (int64_t)c * (g.ldw + 1)) : 0.0;
  }
  const double ri = __ldcg(R + (int64_t)lane * (g.ldw + 1));
  __syncthreads();
  const int col = 8 * q + warp;
  double b = lane == col ? 1.0 : 0.0;
#pragma unroll 8
  for (int c = 8 * q; c < kDW; ++c) b = fma(-S[c * kDLd + lane], __shfl_sync(0xffffffffu, b, c), b);
  put_inverse(g, j * kDW + lane, j * kDW + col, col <= lane ? b * ri : 0.0);
  __syncthreads();
}

struct DiagSmem {
  double S[kDW * kDLd];  // the leaf, or its inverse
  double A[16 * kDLd], B[kDW * kDLd], R[kDW];
  int done[kDW];
};

template <class Group>
__device__ void diag_body(const DiagArgs& g, Group grp, DiagSmem& sm) {
  const int G = grp.size(), b = grp.rank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t ld = g.ld, k0 = g.k0;
  const int ldw = g.ldw, size = g.size, nsteps = size / kDW, per = g.inv / kDW;
  double* a = g.a;
  double* w = g.w;
  double *sA = sm.A, *sB = sm.B;
  const int nl = min(G, kDLead);    // CTAs of the next leaf's update
  const int nv = min(G - 1, 4);     // CTAs of V_j
  if (tid < kDW) sm.done[tid] = 0;
  __syncthreads();

  // the first leaf; the 32 x 32 blocks of the inverse off the diagonal start as zero
  if (b == 0) diag_leaf(g, 0, sm.S, sm.done);
  for (int r = G > 1 ? b - 1 : 0; r < size; r += G > 1 ? G - 1 : 1) {
    if (r < 0) break;
    const int g0 = r / g.inv * g.inv;
    for (int c = g0 + tid; c < g0 + g.inv; c += kDThreads)
      if (c / kDW != r / kDW) put_inverse(g, r, c, 0.0);
  }
  grp.sync();

  for (int j = 0; j < nsteps; ++j) {
    const int64_t c0 = k0 + (int64_t)j * kDW, r0 = c0 + kDW;
    const int below = size - (j + 1) * kDW;  // rows of the block below step j
    const int i1 = j > 0 ? (j - 1) / per * per : 0;  // first step of the block of width inv that j - 1 lies in
    // ---- (b) x D^T = A(r, c0 ..) row by row.  Step c takes x_c as it stands and subtracts x_c (r_c L_lc) from the
    //      columns l > c; at the end x_c r_c.  Eight rows a task, sixteen where there are more tasks than CTAs.
    const int lg = below / 8 > G ? 4 : 3, rows = 1 << lg, nsub = below >> lg;
    for (int t = b; t < nsub; t += G) {
      double* src = a + r0 + (int64_t)rows * t + c0 * ld;
      __syncthreads();
      {
        double v[2], vv[4], rc[4];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int idx = tid + u * kDThreads;
          v[u] = idx < rows * kDW ? __ldcg(src + (idx & (rows - 1)) + (int64_t)(idx >> lg) * ld) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          vv[u] = __ldcg(a + c0 + lane + (c0 + warp + 8 * u) * ld);  // D(lane, warp + 8 u)
          rc[u] = __ldcg(w + (int64_t)(j * kDW + warp + 8 * u) * (ldw + 1));
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int idx = tid + u * kDThreads;
          if (idx < rows * kDW) sA[(idx & (rows - 1)) * kDLd + (idx >> lg)] = v[u];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double m = vv[u] * rc[u];
          sB[(warp + 8 * u) * kDLd + lane] = lane > warp + 8 * u ? m : 0.0;
          if (lane == 0) sm.R[warp + 8 * u] = rc[u];
        }
      }
      __syncthreads();
      if (rows == 8) {  // a row a warp: the shorter chain
        double x = sA[warp * kDLd + lane];
#pragma unroll
        for (int c = 0; c < kDW; ++c) x = fma(-__shfl_sync(0xffffffffu, x, c), sB[c * kDLd + lane], x);
        sA[warp * kDLd + lane] = x * sm.R[lane];
      } else {  // two rows a warp, 16 lanes a row with columns q and q + 16: fewer instructions a row
        const int r = 2 * warp + (lane >> 4), q = lane & 15;
        double x0 = sA[r * kDLd + q], x1 = sA[r * kDLd + q + 16];
#pragma unroll
        for (int c = 0; c < kDW; ++c) {
          const double* col = sB + c * kDLd;
          if (c < 16) {
            const double xc = __shfl_sync(0xffffffffu, x0, c, 16);
            x0 = fma(-xc, col[q], x0);
            x1 = fma(-xc, col[q + 16], x1);
          } else {
            x1 = fma(-__shfl_sync(0xffffffffu, x1, c - 16, 16), col[q + 16], x1);
          }
        }
        sA[r * kDLd + q] = x0 * sm.R[q];
        sA[r * kDLd + q + 16] = x1 * sm.R[q + 16];
      }
      __syncthreads();
      for (int idx = tid; idx < rows * kDW; idx += kDThreads)
        src[(idx & (rows - 1)) + (int64_t)(idx >> lg) * ld] = sA[(idx & (rows - 1)) * kDLd + (idx >> lg)];
    }
    //      W_i = V_i T_i in place, i = j - 1, in strips of eight columns (a strip is one task's alone); on the CTAs that
    //      have no rows first
    auto inverse_rows = [&](int i) {
      const int first = i / per * per * kDW, n = (i * kDW - first) / 8;
      for (int t = G - 1 - b; t < n; t += G) {
        const int cb = first + 8 * t;
        double* T = w + (int64_t)(i * kDW) * ldw + cb;
        const double* V = w + (int64_t)(i * kDW) * (ldw + 1);
        __syncthreads();
        const double tv = __ldcg(T + (int64_t)(tid >> 3) * ldw + (tid & 7));
        double vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = __ldcg(V + (int64_t)(warp + 8 * u) * ldw + lane);
        sA[(tid & 7) * kDLd + (tid >> 3)] = tv;
#pragma unroll
        for (int u = 0; u < 4; ++u) sB[(warp + 8 * u) * kDLd + lane] = vv[u];
        __syncthreads();
        double acc = 0.0;
#pragma unroll 8
        for (int k = 0; k < kDW; ++k) acc = fma(sB[lane * kDLd + k], sA[warp * kDLd + k], acc);
        __syncthreads();
        sA[warp * kDLd + lane] = acc;
        __syncthreads();
        put_inverse(g, i * kDW + (tid >> 3), cb + (tid & 7), sA[(tid & 7) * kDLd + (tid >> 3)]);
      }
    };
    if (j > 0) inverse_rows(j - 1);
    if (j == nsteps - 1) {  // V of the last leaf and the log-determinant parts, off the chain
      for (int q = 0; q < 4; ++q)
        if (b == (G > 1 ? 1 + q % nv : 0)) diag_leaf_inverse(g, j, q, sm.S);
      for (int s4 = b; s4 < size / kDSub; s4 += G) {  // uniform over the CTA
        __syncthreads();
        if (tid < kDSub) {
          const int64_t r = k0 + kDSub * s4 + tid;
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
    }
    grp.sync();
    // ---- (c) the next leaf: its rows spread over the first CTAs
    const bool more = j + 1 < nsteps;
    if (more) {
      if (b < nl) {
        __syncthreads();
        double vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) vv[u] = __ldcg(a + r0 + lane + (c0 + warp + 8 * u) * ld);
#pragma unroll
        for (int u = 0; u < 4; ++u) sB[lane * kDLd + warp + 8 * u] = vv[u];
        __syncthreads();
        for (int i = kDW * b / nl + warp; i < kDW * (b + 1) / nl; i += kDThreads / 32) {  // (nl may not divide 32)
          double* pc = a + (r0 + i) + (r0 + lane) * ld;
          const double a0 = lane <= i ? __ldcg(pc) : 0.0;
          double s0 = 0.0, s1 = 0.0;
#pragma unroll
          for (int k = 0; k < kDW; k += 2) {
            s0 = fma(sB[i * kDLd + k], sB[lane * kDLd + k], s0);
            s1 = fma(sB[i * kDLd + k + 1], sB[lane * kDLd + k + 1], s1);
          }
          if (lane <= i) *pc = a0 - (s0 + s1);
        }
      }
      grp.lead_sync();
      if (b == 0) diag_leaf(g, j + 1, sm.S, sm.done);
      for (int q = 0; q < 4; ++q)
        if (b == (G > 1 ? G - 1 - q % nv : 0)) diag_leaf_inverse(g, j, q, sm.S);
    }
    //      Tiles of 32 lanes x 16, two of the 16 a warp: C(l, x) -= sum_k Y(l, k) X(x, k).
    //      A_rc -= L_r L_c^T over 32-row blocks R and 16-wide column strips s <= 2 R + 1, but for the leaf's (R = 0):
    //      block R has 2 R + 2 tiles, numbered from R (R + 1) - 2 on; lanes along the rows.
    //      T_i -= L_i,j-1 W_j-1 for i >= j: lanes along the columns, 16 rows a tile.
    //      The products of a step are summed from zero: taken off C one by one, each would round at C's size.
    //      CTA 0 comes to them three rounds late (the leaf), the CTAs of V_j one or two.
    const int nr = more ? below / kDW : 0, nt = nr > 0 ? nr * (nr + 1) - 2 : 0;
    const int ni = j > 0 ? min(i1 + per, nsteps) - j : 0, nc = j - i1;  // row blocks i, column blocks of W_j-1
    const int ntiles = nt + (j > 0 ? 2 * ni * nc : 0);
    const int late0 = more ? 3 : 0, lateV = more ? (nv > 2 ? 1 : 2) : 0;
    int round = 0, base = 0;
    auto next = [&]() {  // this CTA's next tile, -1: none
      while (base < ntiles) {
        const bool no0 = round < late0, noV = round < lateV;
        const int t = base + b - (no0 ? 1 : 0);
        const bool mine = !(no0 && b == 0) && !(noV && b >= G - nv) && t < ntiles;
        base += G - (no0 ? 1 : 0) - (noV ? nv : 0);
        ++round;
        if (mine) return t;
      }
      return -1;
    };
    double va[2], vb[4], vc[2];
    double* pc = nullptr;
    int64_t cs = 0;
    int lim = 0;  // C(lane, x) belongs to the tile if x <= lim
    auto load = [&](int t) {
      const double *px, *py;
      int64_t ys;
      if (t < nt) {
        int R = (int)sqrtf((float)(t + 2));
        while (R * (R + 1) > t + 2) --R;
        while ((R + 1) * (R + 2) <= t + 2) ++R;
        const int s = t + 2 - R * (R + 1);
        px = a + r0 + 16 * s + c0 * ld;
        py = a + r0 + kDW * R + c0 * ld;
        ys = ld;
        pc = a + r0 + kDW * R + lane + (r0 + 16 * s) * ld;
        cs = ld;
        lim = kDW * R + lane - 16 * s;
      } else {
        const int q = t - nt, row = j * kDW + q / nc * 16, col = (i1 + q % nc) * kDW;
        px = a + k0 + row + (c0 - kDW) * ld;
        py = w + (int64_t)(j - 1) * kDW * ldw + col;
        ys = ldw;
        pc = w + (int64_t)row * ldw + col + lane;
        cs = ldw;
        lim = 15;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) va[u] = __ldcg(px + (tid & 15) + ((tid >> 4) + 16 * u) * ld);
#pragma unroll
      for (int u = 0; u < 4; ++u) vb[u] = __ldcg(py + lane + (warp + 8 * u) * ys);
#pragma unroll
      for (int u = 0; u < 2; ++u) vc[u] = warp + 8 * u <= lim ? __ldcg(pc + (warp + 8 * u) * cs) : 0.0;
    };
    int t = next();
    if (t >= 0) load(t);
    while (t >= 0) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 2; ++u) sA[(tid & 15) * kDLd + (tid >> 4) + 16 * u] = va[u];
#pragma unroll
      for (int u = 0; u < 4; ++u) sB[lane * kDLd + warp + 8 * u] = vb[u];
      double acc0 = 0.0, acc1 = 0.0;
      const double c0v = vc[0], c1v = vc[1];
      double* out = pc + warp * cs;
      const int64_t step = 8 * cs;
      const int left = lim - warp;
      __syncthreads();
      t = next();
      if (t >= 0) load(t);  // in flight during the products
#pragma unroll 8
      for (int k = 0; k < kDW; ++k) {
        const double y = sB[lane * kDLd + k];
        acc0 = fma(sA[warp * kDLd + k], y, acc0);
        acc1 = fma(sA[(warp + 8) * kDLd + k], y, acc1);
      }
      if (left >= 0) *out = c0v - acc0;
      if (left >= 8) out[step] = c1v - acc1;
    }
    grp.sync();
    if (!more) inverse_rows(j);
  }
}

__global__ void __launch_bounds__(kDThreads) diag_block_kernel(const __grid_constant__ DiagArgs g, double* scr) {
  __shared__ DiagSmem sm;
  diag_body(g, GridGroup(scr, g.st), sm);
}

// One 128 x 128 tile a cluster, and y = W z, y^T y and the row exponents of L.
__global__ void __launch_bounds__(kDThreads, 2) diag_tasks_kernel(const SolveTileTask* __restrict__ tasks) {
  __shared__ DiagSmem sm;
  ClusterGroup grp;
  const int G = grp.size(), b = grp.rank(), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const SolveTileTask task = tasks[blockIdx.x / G];
  const DiagTileTask& t = task.tile;
  const DiagArgs g{t.a, t.ld, t.k0, t.w, kDSub, kDSub, nullptr, t.logdet, t.st, kDSub};
  diag_body(g, grp, sm);
  grp.sync();
  if (b == G - 1) {  // the exponents, two threads a row
    const double* row = t.a + t.k0 + (tid >> 1) + t.k0 * t.ld;
    int hi = 0;
#pragma unroll 8
    for (int c = 0; c < kDSub / 2; ++c) {
      const int cc = 2 * c + (tid & 1);
      if (cc <= tid >> 1) hi = max(hi, __double2hiint(__ldcg(row + cc * t.ld)) & 0x7FFFFFFF);
    }
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, 1));
    if (!(tid & 1)) task.rex[tid >> 1] = (hi >> 20) - 1022;
  }
  if (b != 0) return;
  double* zs = sm.S;
  if (tid < kDSub) zs[tid] = task.z[tid];
  __syncthreads();
  double qs = 0.0;
#pragma unroll 4
  for (int r = warp; r < kDSub; r += 8) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) s = fma(__ldcg(t.w + r * kDSub + lane + 32 * q), zs[lane + 32 * q], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) task.z[r] = s;
    qs = fma(s, s, qs);
  }
  __syncthreads();
  if (lane == 0) zs[warp] = qs;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += zs[q];
    *task.quad = s;
  }
}

// The widest cluster with which every tile has its SMs at once: more CTAs shorten a tile, but tiles that queue cost
// more.
cudaError_t launch_diag128_tasks(cudaStream_t s, const SolveTileTask* d_tasks, int ntasks) {
  if (ntasks <= 0) return cudaSuccess;
  int G = 8;
  while (G > 1 && G * ntasks > tc_num_sms()) G /= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(ntasks * G));
  cfg.blockDim = dim3(kDThreads);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim = {(unsigned)G, 1, 1};
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, diag_tasks_kernel, d_tasks);
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
  grid = diag_grid(grid, tc_num_sms());
  e = cudaMemsetAsync(scratch, 0, kDiagScratch * sizeof(double), s);
  if (e != cudaSuccess) return e;
  // (a smaller block is the last of its matrix: only its 128 sub-tile inverses are wanted)
  DiagArgs g{a, ld, k0, w2, kDB, size == kDB ? kDB : kDSub, w_sub, logdet_part, st, size};
  void* args[] = {&g, &scratch};
  // cooperative launch: every CTA is resident at once, so the grid barriers cannot wait on an
  // unscheduled CTA
  return cudaLaunchCooperativeKernel((const void*)diag_block_kernel, grid, kDThreads, args, smem, s);
}

}  // namespace exa
