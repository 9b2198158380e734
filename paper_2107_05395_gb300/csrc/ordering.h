// Whether a banded matrix may be eliminated in another order than from its first row
// down (host C++ only).  The two-ended and partitioned solves take no pivots in orders
// that the plain factorisation of A says nothing about: a matrix whose LU is harmless
// can have a tiny pivot from the other end or inside a chunk.  For the two classes
// below every order is stable without pivoting, so those solves may be taken without
// being asked for:
//   * weakly diagonally dominant by rows or by columns, with a non-zero diagonal: what is
//     left after any row is eliminated is dominant again, and no entry grows beyond twice
//     the largest of A;
//   * symmetric positive definite (symmetric, and every pivot of A = LU positive): nothing
//     grows, and no pivot is smaller than A's smallest eigenvalue.
// The pivots themselves differ from one order to another: [[1, 1], [1, 2]] has 1, 1 from
// the first row down and 2, 1/2 from the last row up.
#pragma once

#include <cmath>
#include <cstdint>

namespace sb {

// diag[(o + P) * N + i] = A[i][i + o], zero outside the matrix.
inline bool any_order_stable(int P, int64_t N, const double* diag) {
  auto A = [&](int64_t i, int o) -> double {
    return (i < 0 || i >= N || i + o < 0 || i + o >= N) ? 0.0 : diag[(size_t)(o + P) * N + i];
  };
  bool rows = true, cols = true, sym = true;
  for (int64_t i = 0; i < N; ++i) {
    double r = 0.0, c = 0.0;
    for (int o = 1; o <= P; ++o) {
      r += std::fabs(A(i, o)) + std::fabs(A(i, -o));
      c += std::fabs(A(i + o, -o)) + std::fabs(A(i - o, o));
      sym = sym && A(i, o) == A(i + o, -o);
    }
    const double d = std::fabs(A(i, 0));
    rows = rows && d > 0.0 && d >= r;
    cols = cols && d > 0.0 && d >= c;
  }
  if (rows || cols) return true;
  if (!sym) return false;
  // pivots of the LDL^T recurrence (section 4.1's, with beta_i = gamma_{i-1} alpha_{i-1})
  double al1 = 0.0, al2 = 0.0, be1 = 0.0;  // alpha_{i-1}, alpha_{i-2}, entry (i-1, i-2) after elimination
  for (int64_t i = 0; i < N; ++i) {
    const double e = P == 2 ? A(i, -2) : 0.0;
    const double l2 = i >= 2 ? e / al2 : 0.0;
    const double be = i >= 1 ? A(i, -1) - l2 * be1 : 0.0;
    const double al = A(i, 0) - (i >= 2 ? l2 * e : 0.0) - (i >= 1 ? be * be / al1 : 0.0);
    if (!(al > 0.0) || !std::isfinite(al)) return false;
    al2 = al1;
    al1 = al;
    be1 = be;
  }
  return true;
}

}  // namespace sb
