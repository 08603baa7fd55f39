// FP64 products on the tensor cores: operands cut into BF16 digits, exact partial sums.
#pragma once

#include "exa_internal.cuh"

struct exa_ctx;

namespace exa {

constexpr int kDigSlices = 8;    // 7-bit digits per value of a full-precision operand (55 bits below the row maximum)
constexpr int kDigLow = 4;       // digits of a correction operand (27 bits below its row maximum)
constexpr int kDigMaxK = 512;    // longest reduction of one pass (its digit sums stay below 2^24)
constexpr int kDigTN = 64;       // output tile: 128 x kDigTN

// `rows` x K values as digit planes.  Plane p = kc * S + s (16 columns from 16 kc, digit s) holds every row's
// 16 BF16 digits, 32 bytes a row, in the order the tensor cores read: 8-row groups of 256 bytes, each two
// 128-byte halves (columns 0-7 and 8-15) of 8 rows x 16 bytes.  Row r is scaled by 2^ex[r] (kDigBad: the row
// holds an infinity or a NaN).  sq[r] = sum_k of the digit products with s + t = S of the row with itself,
// which the product leaves out (see gemm_digits_kernel).
struct DigitOperand {
  uint8_t* dig = nullptr;
  int* ex = nullptr;
  int* sq = nullptr;
  int64_t rows = 0;    // rows of every plane (a multiple of 8)
};
constexpr int kDigBad = 1 << 28;  // above any sum of exponents, below overflow

// Bytes of an operand of `rows` x K with S digits, and its layout at `base` (256-byte aligned).
size_t digit_bytes(int64_t rows, int K, int S);
void digit_layout(DigitOperand& op, void* base, int64_t rows, int K, int S);
// Rows [0, rows) of src (element (r, k) at src[r rs + k cs]) to operand rows [out_row0, ...), which is a
// multiple of 8; K a multiple of 16, at most kDigMaxK; S = kDigSlices or kDigLow.  lower: values with k > r count
// as 0 and are not read.  colex: column k is multiplied by 2^(colsign colex[k]) first (entries kDigBad: unspecified).
cudaError_t launch_digit_split(cudaStream_t s, const double* src, int64_t rs, int64_t cs, int64_t rows, int K, int S,
                               const DigitOperand& op, int64_t out_row0 = 0, bool lower = false,
                               const int* colex = nullptr, int colsign = 0);

enum : int { kDigRect = 0, kDigLower = 1, kDigTasks = 2 };
struct DigitGemm {
  // C(i, j) = Cin(i, j) +- sum_k A(a_row0 + i, k) B(b_row0 + j, k), C and Cin column-major; Cin = nullptr: 0.
  double* C;
  int64_t ldc;
  const double* Cin;
  int64_t ldcin;
  int64_t m, n;              // m a multiple of 128, n of kDigTN
  DigitOperand A, B;
  int64_t a_row0, b_row0;    // multiples of 8
  int K;                     // multiple of 16, at most kDigMaxK
  int S;                     // digits of both operands
  int neg;                   // the product's sign: 0 +, 1 -
  int shape;                 // kDigRect, or kDigLower (m = n, A = B, a_row0 = b_row0): entries i >= j only
  int tri;                   // B is lower triangular (B(j, k) = 0 for k > j): the reduction of column tile j stops there
  int64_t skip;              // kDigLower: leave out the leading skip x skip block (a multiple of 128, at most 2048)
  DevStatus* st;
};
// max_ctas > 0 caps the persistent grid.
cudaError_t launch_gemm_digits(cudaStream_t s, const DigitGemm& g, int max_ctas = 0);

// Grouped forms (batched replicates).  One 128 x kDigTN tile of C: rows a_row.. of A against rows b_row.. of B.
// diag >= 0: the tile lies on the diagonal of a symmetric output (rows of A and B alike), its first column diag columns
// right of its first row's, and only entries on or below the diagonal are written; kDigPlain: all entries; kDigStore:
// C = A B^T without reading C.
enum : int { kDigPlain = -1, kDigStore = -2 };
struct DigitTask {
  double* C;
  int64_t ldc;
  int a_row, b_row;
  int diag, pad;
};
cudaError_t launch_gemm_digits_tasks(cudaStream_t s, const DigitTask* d_tasks, long long ntasks, int K, int S,
                                     const DigitOperand& A, const DigitOperand& B, bool neg, DevStatus* st);
// One piece of a grouped split (the arguments of launch_digit_split).
struct DigitSplitTask {
  const double* src;
  int64_t rs, cs, rows, out_row0;
  const int* colex;
  int colsign, lower;
};
cudaError_t launch_digit_split_tasks(cudaStream_t s, const DigitSplitTask* d_tasks, int ntasks, int64_t max_rows,
                                     int K, int S, const DigitOperand& op);

}  // namespace exa
