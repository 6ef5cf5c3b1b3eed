// FP64-accurate complex GEMM on the bf16 tensor cores (zgemm_tc.cu).
#pragma once
#include <cuda_bf16.h>

#include "pw_internal.cuh"

namespace pw {
namespace oz {

// 7-bit digits per operand entry: 49 bits of each row-scaled entry, or 56, which carry FP64 entries
// within 2^3 of the row's largest whole.  Error of a sum of K products a_k b_k: below 2^-44 (seven
// digits) or 2^-51 of |a_max| |b_max| per element; FMAs err relative to the running sum.  Emulated at
// K = 4000, relative to |a| |b|: entries of even size 8 digits 3e-18, FMAs 8e-18; both decaying over 6
// decades 7e-17 and 1e-16, over 10 both 1e-16 (7 digits 5e-16 to 6e-15); where one decays and the other
// grows, products of even size add up to far less than |a| |b| and FMAs keep what eight digits do not
// (4 decades: 2e-17 and 3e-20).
constexpr int kDigits = 7, kDigitsFull = 8;

// Digit planes of a K-major realified operand: dig[s * plane + row * pitch + k], s < digits,
// rows x k2 bf16 values (k2 = 2 x complex K), and one power-of-two exponent per complex row
// (A form) or per column (B form): entry = 2^exp * sum_s digit_s 2^(-7 (s + 1)).
struct Digits {
  const __nv_bfloat16* dig;
  int rows;       // realified rows: 2 x complex rows (A form) or columns of op(B) (B form)
  int k2;         // realified K
  int64_t pitch;  // elements per row (multiple of 8)
  int64_t plane;  // elements per digit plane
  const int* exp;
  int digits;     // kDigits or kDigitsFull
};

// Bytes of digit planes for `rows` realified rows of realified length k2.
size_t digit_bytes(int rows, int k2, int digits = kDigits);
int64_t digit_pitch(int k2);

// Slices op(X) (R x K complex; element (r, l) = X[r * sr + l * sl], conjugated if cj) into digit
// planes: A form (aform != 0) gives the real matrix of 2R rows [Re -Im; Im Re] per complex
// entry, B form gives R rows of interleaved (Re, Im) along K.  amax: R scratch words.  A row with an
// entry that is not finite makes its row (column) of a product NaN.
cudaError_t slice(const double2* X, int64_t sr, int64_t sl, int cj, int R, int K, int aform, __nv_bfloat16* dig,
                  int64_t pitch, int64_t plane, unsigned long long* amax, int* exp, cudaStream_t st, int digits = kDigits);

// Split count of a GEMM with realified M2 x N output over realified K k2 (whole K chunks).
int split_count(int M2, int N, int k2, int lower);

// C (M x N complex) = op(A) op(B), both operands with the same number of digits, with the epilogue `epi`: A in A form (rows 2M), B in B form
// (rows N), both of realified length 2K.  lower != 0: only the 64 x 64 complex tiles on or
// below the diagonal (M == N).  nsplit > 1 reduces through `part` (nsplit * N * 2M doubles).
// *err (device) is set if a bounded wait expired; test_no_copies makes the producer issue no
// copies with a short wait limit, so that the first wait expires (failure-path test).
cudaError_t gemm(const Digits& A, const Digits& B, int M, int N, int K, const Epi<double>& epi, int lower,
                 int nsplit, double* part, int* err, int test_no_copies, cudaStream_t st);

bool available();

}  // namespace oz
}  // namespace pw
