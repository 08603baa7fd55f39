// Spatial prediction (kriging) at new locations from the FP64 factor of the
// observed field: the conditional mean and variance that the paper's
// exact_predict returns in the sea-surface-temperature tutorial (Section IV).
//
//   a = Sigma^-1 z                    (the factor and the two triangular solves
//                                      of the log-likelihood path)
//   mean_i = c_i^T a,                 c_i = (Sigma(new_i, obs_j))_j, Eq. 3
//   var_i  = sigma^2 - |L^-1 c_i|^2
//
// The mean never stores the cross covariance: each entry is generated from the
// interpolation table where it is used.  The variance needs L^-1 C for a block
// of new points: C (n_pad x 512) is generated, then solved block row by block
// row with the stored inverses of the diagonal tiles (Y_k = W_k C_k, then
// C_rest -= L_rest,k Y_k on FP64 DMMA), accumulating |Y|^2 per column in a
// fixed order.
#include <math.h>
#include <string.h>

#include <algorithm>

#include "bessel.cuh"
#include "ctx.cuh"
#include "digits.cuh"
#include "util.cuh"

namespace exa {

constexpr int kPredTile = 64;   // new points per CTA of the mean kernel
constexpr int kPredCols = 512;  // new points per block of the variance solve on the FP64 units
constexpr int kPredColsDig = 2048;  // ... and on the tensor cores (128 tiles of a 512-row block product: one wave)

// mean_i = sum_j Sigma(new_i, obs_j) a_j.  Thread (p, q) = (tid / 4, tid % 4) sums the
// observations j = q (mod 4) for new point p; the four partials are added in order.  blockIdx.y takes observations
// [y span, (y + 1) span), its sums to mean + y m: 2,048 points alone would keep 32 SMs busy.
__global__ void __launch_bounds__(256) krige_mean_kernel(const double* __restrict__ obs, int64_t n,
                                                         const double* __restrict__ a,
                                                         const double* __restrict__ nl, int64_t m,
                                                         const __grid_constant__ MaternParams P,
                                                         const MaternTable* __restrict__ tab, int64_t span,
                                                         double* __restrict__ mean) {
  __shared__ double sx[256], sy[256], sa[256];
  __shared__ double part[kPredTile][4];
  const int tid = threadIdx.x, p = tid >> 2, q = tid & 3;
  const int64_t i = (int64_t)blockIdx.x * kPredTile + p;
  const double xi = i < m ? nl[2 * i] : 0.0, yi = i < m ? nl[2 * i + 1] : 0.0;
  double acc = 0.0;
  const int64_t start = (int64_t)blockIdx.y * span, end = start + span < n ? start + span : n;
  mean += (int64_t)blockIdx.y * m;
  for (int64_t j0 = start; j0 < end; j0 += 256) {
    const int64_t j = j0 + tid;
    sx[tid] = j < n ? obs[2 * j] : 0.0;
    sy[tid] = j < n ? obs[2 * j + 1] : 0.0;
    sa[tid] = j < n ? a[j] : 0.0;
    __syncthreads();
    const int cnt = (int)((end - j0) < 256 ? (end - j0) : 256);
    for (int t = q; t < cnt; t += 4) {
      acc = fma(matern_value_tab(P, tab, model_dist2(P, xi, yi, sx[t], sy[t])), sa[t], acc);
    }
    __syncthreads();
  }
  part[p][q] = acc;
  __syncthreads();
  if (q == 0 && i < m) mean[i] = ((part[p][0] + part[p][1]) + part[p][2]) + part[p][3];
}

// mean_i = sum over the parts, in order.
__global__ void __launch_bounds__(256) krige_mean_sum_kernel(const double* __restrict__ part, int64_t m, int parts,
                                                             double* __restrict__ mean) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  double s = part[i];
  for (int p = 1; p < parts; ++p) s += part[i + p * m];
  mean[i] = s;
}

// C(j, c) = Sigma(obs_j, new_{c0 + c}) for j < n; zero for padding rows and past the last point.
__global__ void __launch_bounds__(256) cross_cov_kernel(const double* __restrict__ obs, int64_t n, int64_t npad,
                                                        const double* __restrict__ nl, int64_t m, int64_t c0,
                                                        const __grid_constant__ MaternParams P,
                                                        const MaternTable* __restrict__ tab, double* __restrict__ C) {
  const int64_t c = blockIdx.y;
  const int64_t i = c0 + c;
  const bool live = i < m;
  const double xi = live ? nl[2 * i] : 0.0, yi = live ? nl[2 * i + 1] : 0.0;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < npad; j += (int64_t)gridDim.x * blockDim.x) {
    double v = 0.0;
    if (live && j < n) {
      v = matern_value_tab(P, tab, model_dist2(P, obs[2 * j], obs[2 * j + 1], xi, yi));
    }
    C[j + c * npad] = v;
  }
}

// acc[c] += sum_t Y(t, c)^2 over the nb rows of one block (Y column-major, ld = nb); fixed order.
__global__ void col_sumsq_kernel(const double* __restrict__ Y, int nb, int ncols, double* __restrict__ acc) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncols) return;
  double s = 0.0;
  for (int t = 0; t < nb; ++t) {
    const double y = Y[t + (int64_t)c * nb];
    s = fma(y, y, s);
  }
  acc[c] += s;
}

// The same with a warp per column (fixed order).
__global__ void __launch_bounds__(256) col_sumsq_warp_kernel(const double* __restrict__ Y, int rows, int ncols,
                                                             double* __restrict__ acc) {
  const int c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= ncols) return;
  double s = 0.0;
  for (int t = lane; t < rows; t += 32) {
    const double y = Y[t + (int64_t)c * rows];
    s = fma(y, y, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) acc[c] += s;
}

__global__ void krige_var_kernel(const double* __restrict__ acc, double sigma2, int64_t c0, int64_t m, int ncols,
                                 double* __restrict__ var) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c0 + c < m && c < ncols) var[c0 + c] = sigma2 - acc[c];
}

// acc[c] = |L^-1 C(:, c)|^2 for mc columns (a multiple of 64) of C (npad rows, ld npad, overwritten) as digit
// products, block row by block row: Y_k = W_k C_k, corrected once as in the factorisation's panel solve (Y_k += W_k R,
// R = C_k - L_kk Y_k), C_rest -= L_rest,k Y_k.  Y: 512 x mc scratch.  Without the correction the variances were off by
// cond(L_kk) rounding units: 529 points, 3e-15 at nu = 0.5 and 7e-13 at nu = 2.5, range 0.2; 128-wide inverses on the FP64
// units 9e-16 and 2e-14, now 9e-16 and 2e-15.  It takes 2.2 of 29.7 ms for 2,048 points and n = 10,000, where the
// products took 221 ms on the FP64 units.
static cudaError_t variance_digits(exa_ctx* c, int64_t npad, int64_t mc, double* C, double* Y, double* acc) {
  const double* A = (const double*)c->mat.p;
  cudaStream_t s = c->stream;
  cudaError_t e = cudaMemsetAsync(acc, 0, mc * sizeof(double), s);
  for (int64_t k0 = 0, h; k0 < npad && e == cudaSuccess; k0 += h) {
    h = npad - k0 >= kDigMaxK ? kDigMaxK : 128;
    const int64_t rest = npad - k0 - h;
    const double dh = (double)h, dm = (double)mc;
    DigitOperand Dw, Dl, Dwl, Dc, Dr, D;
    digit_layout(Dc, c->mx_split2.p, mc, (int)h, kDigSlices);
    digit_layout(Dr, c->mx_split2.p, mc, (int)h, kDigLow);
    {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * (dm + dh), 4);
      e = split_block_inverse(c, npad, k0, (int)h, Dw, Dl, &Dwl);
      if (e == cudaSuccess) e = launch_digit_split(s, C + k0, npad, 1, mc, (int)h, kDigSlices, Dc, 0, false, Dl.ex, -1);
    }
    DigitGemm g{};
    g.C = Y;
    g.ldc = h;
    g.m = h;
    g.n = mc;
    g.A = Dw;
    g.B = Dc;
    g.K = (int)h;
    g.S = kDigSlices;
    g.shape = kDigRect;
    g.st = c->d_status;
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_GEMM_DIG, dh * dh * dm, 8.0 * dh * dm);
      e = launch_gemm_digits(s, g);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * dm, 1);
      e = launch_digit_split(s, Y, h, 1, mc, (int)h, kDigSlices, Dc);
    }
    if (e == cudaSuccess) {  // R in C_k's place
      DigitGemm r = g;
      r.C = C + k0;
      r.Cin = r.C;
      r.ldc = r.ldcin = npad;
      r.A = Dl;
      r.neg = 1;
      ProfScope ps(c, PK_GEMM_DIG, dh * dh * dm, 16.0 * dh * dm);
      e = launch_gemm_digits(s, r);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_SPLIT, 0.0, 16.0 * dh * dm, 1);
      e = launch_digit_split(s, C + k0, npad, 1, mc, (int)h, kDigLow, Dr, 0, false, Dl.ex, -1);
    }
    if (e == cudaSuccess) {
      DigitGemm r = g;
      r.Cin = Y;
      r.ldcin = h;
      r.A = Dwl;
      r.B = Dr;
      r.S = kDigLow;
      ProfScope ps(c, PK_GEMM_DIG, dh * dh * dm, 16.0 * dh * dm);
      e = launch_gemm_digits(s, r);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_OTHER, 0.0, 8.0 * dh * dm);
      col_sumsq_warp_kernel<<<(unsigned)((mc + 7) / 8), 256, 0, s>>>(Y, (int)h, (int)mc, acc);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess || rest == 0) continue;
    digit_layout(D, c->mx_split.p, rest, (int)h, kDigSlices);
    {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * (dm + (double)rest), 2);
      e = launch_digit_split(s, Y, h, 1, mc, (int)h, kDigSlices, Dc);
      if (e == cudaSuccess) e = launch_digit_split(s, A + k0 + h + k0 * npad, 1, npad, rest, (int)h, kDigSlices, D);
    }
    if (e == cudaSuccess) {
      g.C = C + k0 + h;
      g.Cin = g.C;
      g.ldc = g.ldcin = npad;
      g.m = rest;
      g.A = D;
      g.neg = 1;
      ProfScope ps(c, PK_GEMM_DIG, 2.0 * dh * (double)rest * dm, 16.0 * (double)rest * dm);
      e = launch_gemm_digits(s, g);
    }
  }
  return e;
}

}  // namespace exa

using namespace exa;

extern "C" exa_status exa_predict(exa_ctx* c, const double* d_locs, const double* d_z, const double theta[3],
                                  int64_t n, const double* d_new_locs, int64_t m, double* d_mean, double* d_var) {
  if (!c) return EXA_ERR_ARG;
  c->err[0] = 0;
  c->last_pivot = -1;
  if (n < 1 || m < 0 || !d_locs || !d_z || (m > 0 && (!d_new_locs || !d_mean)))
    return set_err(c, EXA_ERR_ARG, "bad sizes or NULL device pointer");
  exa_status st = check_theta(c, theta);
  if (st != EXA_OK) return st;
  if (m == 0) return EXA_OK;
  // factor, y = L^-1 z (log-likelihood path, FP64)
  exa_result res;
  memset(&res, 0, sizeof(res));
  double* y = nullptr;
  const int nb = c->tile_nb;
  const int64_t npad = round_up(n, nb);
  // new points per block of the variance's products on the tensor cores
  const int64_t mc = std::min<int64_t>(round_up(m, 64), kPredColsDig);
  if (d_var && nb == 128) reserve_inverse_digits(c, npad, true, mc);
  if ((st = loglik_fp64(c, d_locs, d_z, theta, n, &res, &y)) != EXA_OK) return st;
  const int T = (int)(npad / nb);
  double* A = (double*)c->mat.p;
  const double* W = (const double*)c->w_all.p;
  cudaStream_t s = c->stream;
  // a = L^-T y (in place)
  cudaError_t e = solve_backward(c, npad, nb, y);
  if (e != cudaSuccess) return cuda_err(c, e, "prediction solve");
  MaternParams P;
  model_params(c, theta, &P);
  const MaternTable* tab = nullptr;
  if ((st = matern_table(c, P, &tab)) != EXA_OK) return st;
  {
    // parts of the observations, so that at least two CTAs per SM run: by n and m alone, so that a repeated call
    // sums in the same order
    const int64_t blocks = ceil_div(m, kPredTile), want = ceil_div(2 * tc_num_sms(), blocks);
    int64_t span = round_up(ceil_div(n, std::min<int64_t>(want, 64)), 256);
    int64_t parts = ceil_div(n, span);
    if (parts > 1 && ensure(c, c->pr_m, (size_t)(parts * m) * sizeof(double), "prediction sums", true) != EXA_OK) {
      c->err[0] = 0;
      parts = 1;
      span = n;
    }
    ProfScope ps(c, PK_GEN, 0.0, 16.0 * (double)n + 24.0 * (double)m, parts > 1 ? 2 : 1);
    double* out = parts > 1 ? (double*)c->pr_m.p : d_mean;
    krige_mean_kernel<<<dim3((unsigned)blocks, (unsigned)parts), 256, 0, s>>>(d_locs, n, y, d_new_locs, m, P, tab,
                                                                              span, out);
    if (parts > 1) krige_mean_sum_kernel<<<(unsigned)ceil_div(m, 256), 256, 0, s>>>(out, m, (int)parts, d_mean);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return cuda_err(c, e, "prediction mean");
  c->pred_spare = false;  // the buffers are this call's until it ends
  if (d_var && c->wall_kept && reserve_inverse_digits(c, npad, false, mc) &&
      ensure(c, c->pr_c, (size_t)npad * mc * sizeof(double), "prediction cross covariance", true) == EXA_OK &&
      ensure(c, c->pr_y, (size_t)(kDigMaxK + 1) * mc * sizeof(double), "prediction solve block", true) == EXA_OK) {
    c->pred_spare = true;
    double* C = (double*)c->pr_c.p;
    double* Y = (double*)c->pr_y.p;
    double* acc = Y + (size_t)kDigMaxK * mc;
    for (int64_t c0 = 0; c0 < m && e == cudaSuccess; c0 += mc) {
      const int64_t cols = std::min<int64_t>(mc, round_up(m - c0, 64));
      {
        ProfScope ps(c, PK_GEN, 0.0, 8.0 * (double)npad * (double)cols);
        cross_cov_kernel<<<dim3((unsigned)((npad + 255) / 256 < 64 ? (npad + 255) / 256 : 64), (unsigned)cols), 256, 0,
                           s>>>(d_locs, n, npad, d_new_locs, m, c0, P, tab, C);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = variance_digits(c, npad, cols, C, Y, acc);
      if (e == cudaSuccess) {
        krige_var_kernel<<<(unsigned)ceil_div(cols, 128), 128, 0, s>>>(acc, theta[0], c0, m, (int)cols, d_var);
        e = cudaGetLastError();
      }
    }
    if (e != cudaSuccess) return cuda_err(c, e, "prediction variance");
  } else if (d_var) {
    c->err[0] = 0;
    // variance: blocks of kPredCols new points; what was sized for more goes first
    const size_t c_bytes = (size_t)npad * kPredCols * sizeof(double);
    const size_t y_bytes = (size_t)(nb + 1) * kPredCols * sizeof(double);
    if (c->pr_c.bytes > c_bytes || c->pr_y.bytes > y_bytes) free_spare(c, {&c->pr_c, &c->pr_y});
    if ((st = ensure(c, c->pr_c, c_bytes, "prediction cross covariance")) != EXA_OK) return st;
    if ((st = ensure(c, c->pr_y, y_bytes, "prediction solve block")) != EXA_OK) return st;
    double* C = (double*)c->pr_c.p;
    double* Y = (double*)c->pr_y.p;
    double* acc = Y + (size_t)nb * kPredCols;
    for (int64_t c0 = 0; c0 < m && e == cudaSuccess; c0 += kPredCols) {
      {
        ProfScope ps(c, PK_GEN, 0.0, 8.0 * (double)npad * kPredCols);
        cross_cov_kernel<<<dim3((unsigned)((npad + 255) / 256 < 64 ? (npad + 255) / 256 : 64), kPredCols), 256, 0,
                           s>>>(d_locs, n, npad, d_new_locs, m, c0, P, tab, C);
        e = cudaGetLastError();
      }
      if (e == cudaSuccess) e = cudaMemsetAsync(acc, 0, kPredCols * sizeof(double), s);
      for (int k = 0; k < T && e == cudaSuccess; ++k) {
        const int64_t k0 = (int64_t)k * nb, rest = npad - k0 - nb;
        ProfScope ps(c, PK_DGEMM_SMALL, 2.0 * (double)(nb + rest) * nb * kPredCols,
                     8.0 * ((double)(nb + rest) * nb + 2.0 * (double)(nb + rest) * kPredCols), 2 + (rest > 0));
        // Y = W_k C_k   (W_k row-major nb x nb; C_k rows k0.. of C)
        e = launch_dgemm_nt_small(s, nb, kPredCols, nb, 1.0, W + (int64_t)k * nb * nb, nb, 1, C + k0, npad, 1, 0.0,
                                  Y, 1, nb, c->d_status);
        if (e == cudaSuccess) {
          col_sumsq_kernel<<<kPredCols / 128, 128, 0, s>>>(Y, nb, kPredCols, acc);
          e = cudaGetLastError();
        }
        // C_rest -= L_rest,k Y
        if (e == cudaSuccess && rest > 0)
          e = launch_dgemm_nt_small(s, (int)rest, kPredCols, nb, -1.0, A + k0 + nb + k0 * npad, 1, npad, Y, nb, 1,
                                    1.0, C + k0 + nb, 1, npad, c->d_status);
      }
      if (e == cudaSuccess) {
        krige_var_kernel<<<kPredCols / 128, 128, 0, s>>>(acc, theta[0], c0, m, kPredCols, d_var);
        e = cudaGetLastError();
      }
    }
    if (e != cudaSuccess) return cuda_err(c, e, "prediction variance");
  }
  return read_status(c);
}
