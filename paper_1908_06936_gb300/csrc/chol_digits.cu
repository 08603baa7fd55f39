// Step a2 in FP64 on the tensor cores: right-looking Cholesky in 512-wide panels whose contractions run as digit
// products (digits.cu).  Panel k, rows k0 ..:
//   1. the 512 x 512 diagonal block in FP64: L_kk, its inverse W and the 128 sub-tile inverses the solves use
//      (diag_block.cu), on the look-ahead stream beside step 3 of the panel before;
//   2. the panel below it, L_ik = A_ik L_kk^-T: a first solution X = A_ik W^T and one correction,
//      R = A_ik - X L_kk^T, L_ik = X + R W^T.  Multiplying by an explicit inverse alone leaves an error of
//      cond(L_kk) rounding units in A_ik, which grows with the block: on a 512 block of a smooth field it was three
//      times the error of the 128-wide panels; with the correction it is a rounding unit.  R is that much smaller
//      than A_ik, and its product has to hold 1 / cond(L_kk) of itself: four digits.  (With two, the log-determinant of
//      1,024 points was off by 3e-7 at nu = 2.5, range 0.2, and by 4e-2 at nu = 3.5, where now 7e-9 and 8e-6; the panels
//      of 128 rows left 3e-8 and 4e-5.)  The digits are relative to a row's largest value, while column
//      c of A_ik and of W^T goes with the size of row c of L_kk: both products run on A_ic 2^-e_c and W_.c 2^e_c
//      with e_c that row's exponent, so that a badly scaled matrix loses nothing;
//   3. A_ij -= L_ik L_jk^T over the trailing lower triangle: the next diagonal block first, then, while the
//      look-ahead stream factors that, everything else.
#include <algorithm>

#include "ctx.cuh"
#include "digits.cuh"

namespace exa {

constexpr int kNB = kDigMaxK;  // panel width = the longest exact reduction
constexpr int kSub = 128;

static size_t align256(size_t v) { return (v + 255) / 256 * 256; }

static size_t block_bytes(int S) { return align256(digit_bytes(kNB, kNB, S)); }

bool reserve_digits(exa_ctx* c, int64_t npad) {
  const size_t below = npad > kNB ? (size_t)(npad - kNB) : 0;  // rows of the first panel
  struct {
    DevBuf* b;
    size_t bytes;
  } want[] = {{&c->mx_w2, (size_t)kNB * kNB * sizeof(double)},
              {&c->mx_dscr, (diag_block_scratch_doubles() + kSolveScratch) * sizeof(double)},
              {&c->mx_wall, (size_t)(npad / kNB) * kNB * kNB * sizeof(double)},
              {&c->mx_split, below ? align256(digit_bytes(below, kNB, kDigSlices)) : 0},
              {&c->mx_split_b, below ? 2 * block_bytes(kDigSlices) + block_bytes(kDigLow) : 0},
              {&c->mx_split2, below * kNB * sizeof(double)}};
  size_t held = c->held_bytes;
  for (auto& w : want) held += w.bytes > w.b->bytes ? w.bytes - w.b->bytes : 0;
  bool ok = !c->ws_limit || held <= c->ws_limit;
  for (auto& w : want) ok = ok && ensure(c, *w.b, w.bytes, "digit operands", true) == EXA_OK;
  c->operands_spare = true;
  if (!ok) {
    c->err[0] = 0;
    release_digits(c);
  }
  return ok;
}

// The factorisation of `a` (npad a multiple of 128).  *done = false: the workspace could not be had and nothing was
// launched.
exa_status factor_digits(exa_ctx* c, double* a, int64_t ld, int64_t npad, bool* done) {
  *done = false;
  const int T = (int)ceil_div(npad, kNB), T128 = (int)(npad / kSub);
  exa_status st;
  if ((st = ensure(c, c->w_all, (size_t)T128 * kSub * kSub * sizeof(double), "inverted diagonal tiles")) != EXA_OK)
    return st;
  if ((st = ensure(c, c->logdet_part, (size_t)T128 * sizeof(double), "log-det partials")) != EXA_OK) return st;
  if (!reserve_digits(c, npad)) return EXA_OK;
  if ((st = ensure_side(c)) != EXA_OK) return st;
  *done = true;
  double* W = (double*)c->w_all.p;
  double* LD = (double*)c->logdet_part.p;
  c->wall_kept = true;
  double* X = (double*)c->mx_split2.p;
  cudaStream_t ms = c->stream, ss = c->side;
  SideJoin streams(ms, ss, c->la_ev);
  const int sms = tc_num_sms();
  DigitOperand Dw, Dl, Dwl;
  if (T > 1) {
    digit_layout(Dw, c->mx_split_b.p, kNB, kNB, kDigSlices);
    digit_layout(Dl, (uint8_t*)c->mx_split_b.p + block_bytes(kDigSlices), kNB, kNB, kDigSlices);
    digit_layout(Dwl, (uint8_t*)c->mx_split_b.p + 2 * block_bytes(kDigSlices), kNB, kNB, kDigLow);
  }
  // step 1 on stream s, with the digits of W and L_kk that step 2 needs
  auto diagonal = [&](cudaStream_t s, int k, int ctas) -> cudaError_t {
    const int64_t k0 = (int64_t)k * kNB;
    const int w = (int)std::min<int64_t>(kNB, npad - k0);
    const double w3 = (double)w * w * w;
    double* W2 = w == kNB ? (double*)c->mx_wall.p + k0 * kNB : (double*)c->mx_w2.p;
    cudaError_t e;
    {
      ProfScope ps(c, PK_POTRF, (w == kNB ? 2.0 : 1.0) * w3 / 3.0, 8.0 * (3.0 * w * w), 1, s, s != ms);
      e = launch_diag_block(s, a, ld, k0, W + (k0 / kSub) * kSub * kSub, LD + k0 / kSub, W2, (double*)c->mx_dscr.p,
                            c->d_status, ctas, w);
    }
    if (e == cudaSuccess && k + 1 < T) {
      ProfScope ps(c, PK_SPLIT, 0.0, 66.0 * kNB * kNB, 3, s, s != ms);
      e = launch_digit_split(s, a + k0 + k0 * ld, 1, ld, kNB, kNB, kDigSlices, Dl, 0, true);
      if (e == cudaSuccess) e = launch_digit_split(s, W2, kNB, 1, kNB, kNB, kDigSlices, Dw, 0, true, Dl.ex, 1);
      if (e == cudaSuccess) e = launch_digit_split(s, W2, kNB, 1, kNB, kNB, kDigLow, Dwl, 0, true, Dl.ex, 1);
    }
    return e;
  };
  cudaError_t e = diagonal(ms, 0, kDiagCtas);
  for (int k = 0; k + 1 < T && e == cudaSuccess; ++k) {
    const int64_t k0 = (int64_t)k * kNB, r0 = k0 + kNB, m = npad - r0;
    const double dm = (double)m;
    double* panel = a + r0 + k0 * ld;
    // step 2
    DigitOperand D, Dr;
    digit_layout(D, c->mx_split.p, m, kNB, kDigSlices);
    digit_layout(Dr, c->mx_split.p, m, kNB, kDigLow);
    DigitGemm g{};
    g.m = m;
    g.n = g.K = kNB;
    g.shape = kDigRect;
    g.tri = 1;
    g.st = c->d_status;
    {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dm * kNB, 1);
      e = launch_digit_split(ms, panel, 1, ld, m, kNB, kDigSlices, D, 0, false, Dl.ex, -1);
    }
    if (e == cudaSuccess) {  // X = A W^T
      ProfScope ps(c, PK_GEMM_DIG, dm * kNB * kNB, 24.0 * dm * kNB);
      g.C = X;
      g.ldc = m;
      g.A = D;
      g.B = Dw;
      g.S = kDigSlices;
      e = launch_gemm_digits(ms, g);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dm * kNB, 1);
      e = launch_digit_split(ms, X, 1, m, m, kNB, kDigSlices, D);
    }
    if (e == cudaSuccess) {  // R = A - X L_kk^T, in A's place
      ProfScope ps(c, PK_GEMM_DIG, dm * kNB * kNB, 32.0 * dm * kNB);
      g.C = panel;
      g.ldc = ld;
      g.Cin = panel;
      g.ldcin = ld;
      g.B = Dl;
      g.neg = 1;
      e = launch_gemm_digits(ms, g);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_SPLIT, 0.0, 12.0 * dm * kNB, 1);
      e = launch_digit_split(ms, panel, 1, ld, m, kNB, kDigLow, Dr, 0, false, Dl.ex, -1);
    }
    if (e == cudaSuccess) {  // L = X + R W^T
      ProfScope ps(c, PK_GEMM_DIG, dm * kNB * kNB, 20.0 * dm * kNB);
      g.Cin = X;
      g.ldcin = m;
      g.A = Dr;
      g.B = Dwl;
      g.S = kDigLow;
      g.neg = 0;
      e = launch_gemm_digits(ms, g);
    }
    if (e == cudaSuccess) {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dm * kNB, 1);
      e = launch_digit_split(ms, panel, 1, ld, m, kNB, kDigSlices, D);
    }
    if (e != cudaSuccess) break;
    // step 3
    const int64_t w1 = std::min<int64_t>(kNB, m);
    DigitGemm u{};
    u.A = u.B = D;
    u.K = kNB;
    u.S = kDigSlices;
    u.neg = 1;
    u.shape = kDigLower;
    u.st = c->d_status;
    u.C = a + r0 + r0 * ld;
    u.Cin = u.C;
    u.ldc = u.ldcin = ld;
    u.m = u.n = w1;
    {
      ProfScope ps(c, PK_GEMM_DIG, (double)w1 * w1 * kNB, 16.0 * (double)w1 * w1 / 2);
      e = launch_gemm_digits(ms, u);
    }
    if (e != cudaSuccess) break;
    streams.fork();
    const int side = side_share(m, kNB, sms);
    e = diagonal(ss, k + 1, side);
    streams.side_done();
    if (e == cudaSuccess && m > w1) {
      ProfScope ps(c, PK_GEMM_DIG, (dm * dm - (double)w1 * w1) * kNB, 8.0 * (dm * dm - (double)w1 * w1));
      u.m = u.n = m;
      u.skip = w1;
      e = launch_gemm_digits(ms, u, sms - side);
    }
    streams.join();
  }
  if (e != cudaSuccess) return cuda_err(c, e, "Cholesky launch");
  return EXA_OK;
}

const double* block_inverse(exa_ctx* c, int64_t k0, int h) {
  return h == kNB ? (const double*)c->mx_wall.p + k0 * kNB : (const double*)c->w_all.p + k0 * kSub;
}

cudaError_t solve_forward(exa_ctx* c, int64_t npad, int nb, double* z, double* y) {
  const double* a = (const double*)c->mat.p;
  double* tmp = (double*)c->mx_dscr.p + diag_block_scratch_doubles();  // with the block inverses only
  cudaError_t e = cudaSuccess;
  for (int64_t k0 = 0, h; k0 < npad && e == cudaSuccess; k0 += h) {
    h = !c->wall_kept ? nb : npad - k0 >= kNB ? kNB : kSub;
    const double rows = (double)(npad - k0);
    ProfScope ps(c, PK_TRSV, 2.0 * rows * h, 8.0 * rows * h, c->wall_kept ? 3 + (npad - k0 > h) : 1);
    if (c->wall_kept)
      e = launch_block_fwd(c->stream, a + k0 + k0 * npad, npad, (int)h, npad - k0 - h, block_inverse(c, k0, (int)h),
                           z + k0, y + k0, tmp, k0 == 0);
    else
      e = launch_trsv_fwd_step(c->stream, a, npad, npad, nb, (int)(k0 / nb), (const double*)c->w_all.p, y, z,
                               c->d_status);
  }
  return e;
}

cudaError_t solve_backward(exa_ctx* c, int64_t npad, int nb, double* y) {
  const double* a = (const double*)c->mat.p;
  double* tmp = (double*)c->mx_dscr.p + diag_block_scratch_doubles();
  const int64_t full = npad / kNB * kNB;  // the 128-wide blocks start here
  cudaError_t e = cudaSuccess;
  for (int64_t end = npad, h; end > 0 && e == cudaSuccess; end -= h) {
    h = !c->wall_kept ? nb : end > full ? kSub : kNB;
    const int64_t k0 = end - h;
    const double rows = c->wall_kept ? (double)end : (double)(npad - k0);
    ProfScope ps(c, PK_TRSV, 2.0 * rows * h, 8.0 * rows * h, c->wall_kept ? 3 + (k0 > 0) : 2);
    if (c->wall_kept)
      e = launch_block_bwd(c->stream, a + k0, npad, k0, (int)h, block_inverse(c, k0, (int)h), y, tmp, end == npad);
    else
      e = launch_trsv_bwd_step(c->stream, a, npad, npad, nb, (int)(k0 / nb), (const double*)c->w_all.p, y,
                               (double*)c->partial.p + 2 * kRedPartials, c->d_status);
  }
  return e;
}

void release_digits(exa_ctx* c) {
  cudaStreamSynchronize(c->stream);
  for (DevBuf* b : {&c->mx_split, &c->mx_split2, &c->mx_split_b, &c->mx_w2, &c->mx_dscr, &c->mx_wall}) {
    if (b->p) cudaFree(b->p);
    c->held_bytes -= b->bytes;
    b->p = nullptr;
    b->bytes = 0;
  }
  c->operands_spare = c->wall_kept = false;
}

}  // namespace exa
