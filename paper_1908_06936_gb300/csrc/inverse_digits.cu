// Sigma^-1 from the FP64 factor, on the tensor cores (digit products, digits.cu): step a7 and the Fisher information.
//
// Row blocks of X = L^-1 top to bottom, right-looking: with block l done, every later row block takes its share,
//   T_i -= L_il X_l  (all i > l in one product),   X_i = W_i T_i,  X_ii = W_i  (W_i = L_ii^-1),
// and Sigma^-1 = X^T X grows by X_l^T X_l.  X is built in a second n x n buffer; block l's columns of L are not
// needed after step l, so Sigma^-1 replaces L in place.  Blocks are the 512-wide panels, the remainder in 128s (whose
// inverses the factorisation has either way).  On the FP64 units the two halves took n^3 / 3 multiply-adds each at
// 1.05 TFLOP/s: 320 ms at n = 6,400.
#include <algorithm>

#include "ctx.cuh"
#include "digits.cuh"

namespace exa {

constexpr int kNB = kDigMaxK;
constexpr int kSub = 128;

static size_t align256(size_t v) { return (v + 255) / 256 * 256; }

bool reserve_inverse_digits(exa_ctx* c, int64_t npad, bool allocate, int64_t rows) {
  if (rows < npad) rows = npad;
  struct {
    DevBuf* b;
    size_t bytes;
  } want[] = {{&c->mx_split, digit_bytes(npad, kNB, kDigSlices)},
              {&c->mx_split2, digit_bytes(rows, kNB, kDigSlices)},
              {&c->mx_split_b, 2 * align256(digit_bytes(kNB, kNB, kDigSlices)) + align256(digit_bytes(kNB, kNB, kDigLow))}};
  if (!allocate) {
    bool have = true;
    for (auto& w : want) have = have && w.b->bytes >= w.bytes;
    return have;
  }
  size_t held = c->held_bytes;
  for (auto& w : want) held += w.bytes > w.b->bytes ? w.bytes - w.b->bytes : 0;
  bool ok = !c->ws_limit || held <= c->ws_limit;
  c->operands_spare = true;  // given back to what the call cannot do without
  for (auto& w : want) ok = ok && ensure(c, *w.b, w.bytes, "digit operands", true) == EXA_OK;
  if (!ok) c->err[0] = 0;
  return ok;
}

cudaError_t split_block_inverse(exa_ctx* c, int64_t npad, int64_t k0, int h, DigitOperand& Dw, DigitOperand& Dl,
                                DigitOperand* Dwl) {
  const double* a = (const double*)c->mat.p + k0 + k0 * npad;
  const double* w = block_inverse(c, k0, h);
  digit_layout(Dl, c->mx_split_b.p, h, h, kDigSlices);
  const size_t one = align256(digit_bytes(kNB, kNB, kDigSlices));
  digit_layout(Dw, (uint8_t*)c->mx_split_b.p + one, h, h, kDigSlices);
  cudaError_t e = launch_digit_split(c->stream, a, 1, npad, h, h, kDigSlices, Dl, 0, true);
  if (e == cudaSuccess) e = launch_digit_split(c->stream, w, h, 1, h, h, kDigSlices, Dw, 0, true, Dl.ex, 1);
  if (e == cudaSuccess && Dwl) {
    digit_layout(*Dwl, (uint8_t*)c->mx_split_b.p + 2 * one, h, h, kDigLow);
    e = launch_digit_split(c->stream, w, h, 1, h, h, kDigLow, *Dwl, 0, true, Dl.ex, 1);
  }
  return e;
}

// Diagonal block <- W (row-major, h x h), strict upper triangle 0.
__global__ void __launch_bounds__(256) put_inverse_kernel(double* __restrict__ x, int64_t ld, int h,
                                                          const double* __restrict__ w) {
  const int c = blockIdx.x;
  for (int r = threadIdx.x; r < h; r += blockDim.x) x[r + c * ld] = r >= c ? w[(int64_t)r * h + c] : 0.0;
}

// c->mat holds L (npad, ld npad) with the block inverses of its factorisation in c->mx_wall and c->w_all: Sigma^-1 into
// its lower triangle; x: npad^2 scratch.  Needs reserve_inverse_digits.
cudaError_t inverse_digits(exa_ctx* c, int64_t npad, double* x) {
  double* a = (double*)c->mat.p;
  const int64_t ld = npad;
  cudaStream_t s = c->stream;
  cudaError_t e = cudaMemsetAsync(x, 0, (size_t)npad * npad * sizeof(double), s);
  for (int64_t l0 = 0, h; l0 < npad && e == cudaSuccess; l0 += h) {
    h = npad - l0 >= kNB ? kNB : kSub;
    const int64_t n1 = l0 + h, m = npad - n1;
    const double* w = block_inverse(c, l0, (int)h);
    const double dh = (double)h;
    DigitOperand Dl, Dw, D, Dx;
    digit_layout(Dx, c->mx_split2.p, n1, (int)h, kDigSlices);
    if (l0 > 0) {
      // X_l = W_l T_l, column k of W and row k of T scaled by row k's size in L_ll (as in the panel solve)
      digit_layout(D, c->mx_split.p, l0, (int)h, kDigSlices);
      {
        ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * (double)n1, 3);
        e = split_block_inverse(c, npad, l0, (int)h, Dw, Dl);
        if (e == cudaSuccess) e = launch_digit_split(s, x + l0, ld, 1, l0, (int)h, kDigSlices, D, 0, false, Dl.ex, -1);
      }
      DigitGemm g{};
      g.C = x + l0;
      g.ldc = ld;
      g.m = h;
      g.n = l0;
      g.A = Dw;
      g.B = D;
      g.K = (int)h;
      g.S = kDigSlices;
      g.shape = kDigRect;
      g.st = c->d_status;
      ProfScope ps(c, PK_GEMM_DIG, dh * dh * (double)l0, 8.0 * dh * (double)l0);
      if (e == cudaSuccess) e = launch_gemm_digits(s, g);
    }
    if (e != cudaSuccess) break;
    put_inverse_kernel<<<(unsigned)h, 256, 0, s>>>(x + l0 + l0 * ld, ld, (int)h, w);
    {
      ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * (double)n1, 1);
      e = launch_digit_split(s, x + l0, ld, 1, n1, (int)h, kDigSlices, Dx);
    }
    if (e == cudaSuccess && m > 0) {
      // T_i -= L_il X_l for every later row
      digit_layout(D, c->mx_split.p, m, (int)h, kDigSlices);
      {
        ProfScope ps(c, PK_SPLIT, 0.0, 24.0 * dh * (double)m, 1);
        e = launch_digit_split(s, a + n1 + l0 * ld, 1, ld, m, (int)h, kDigSlices, D);
      }
      DigitGemm g{};
      g.C = x + n1;
      g.Cin = g.C;
      g.ldc = g.ldcin = ld;
      g.m = m;
      g.n = n1;
      g.A = D;
      g.B = Dx;
      g.K = (int)h;
      g.S = kDigSlices;
      g.neg = 1;
      g.shape = kDigRect;
      g.st = c->d_status;
      ProfScope ps(c, PK_GEMM_DIG, 2.0 * dh * (double)m * (double)n1, 16.0 * (double)m * (double)n1);
      if (e == cudaSuccess) e = launch_gemm_digits(s, g);
    }
    if (e == cudaSuccess) e = cudaMemset2DAsync(a + l0, ld * sizeof(double), 0, h * sizeof(double), n1, s);
    if (e == cudaSuccess) {
      DigitGemm g{};
      g.C = a;
      g.Cin = a;
      g.ldc = g.ldcin = ld;
      g.m = g.n = n1;
      g.A = g.B = Dx;
      g.K = (int)h;
      g.S = kDigSlices;
      g.shape = kDigLower;
      g.st = c->d_status;
      ProfScope ps(c, PK_GEMM_DIG, dh * (double)n1 * (double)n1, 8.0 * (double)n1 * (double)n1);
      e = launch_gemm_digits(s, g);
    }
  }
  return e;
}

}  // namespace exa
