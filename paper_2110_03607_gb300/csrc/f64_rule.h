// Which FP64 products C = A . B^T take the digits on the tensor cores (kernels_f64_tc.cu).
#pragma once

namespace hotrg {

// M x N over K terms.  The FP64 pipe does 0.6e12 multiply-adds a second, so 2^24 of them take 28 us there, about as
// long as the launches and the first tiles of the other path.  A product that is done in groups of columns is
// judged as a whole, so that its bits do not depend on the groups.
inline bool f64_digits_pay(double M, double N, double K, bool upper_only) {
  return M >= 32.0 && N >= 16.0 && K >= 32.0 && M * N * K * (upper_only ? 0.5 : 1.0) >= 16777216.0;
}

// Grams of 2D steps, K = chi_c chi_j <= 32 x 32 terms, stay on the pipe: at a degenerate cut the kept vector follows
// the rounding of the Gram (ordered 2D phase, chi = 24, step 11: a pair 2.8e-15 lambda_1 apart), and such runs go on
// as they did; digits would save 0.1 ms of a Gram of 576 rows.
inline bool f64_gram_digits_pay(double M, double K, bool upper_only) {
  return K > 1024.0 && f64_digits_pay(M, M, K, upper_only);
}

}  // namespace hotrg
