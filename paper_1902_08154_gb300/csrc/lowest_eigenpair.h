// lowest_eigenpair.h -- the lowest eigenpair of a small symmetric matrix, on the
// host (the subspace matrix of the Davidson iteration in davidson.cu).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

namespace qp {

// The lowest eigenpair of the symmetric m x m matrix a (row-major): Householder
// reduction to a tridiagonal matrix, its lowest eigenvalue by bisection on the
// sign count of the LDL^T pivots (Sturm sequence), the eigenvector by inverse
// iteration and the reflections, the eigenvalue again as its Rayleigh quotient.
// The whole spectrum by Jacobi rotations, of which one pair was used, took
// most of the solver's time at 20 and more vectors.
inline double lowest_eigenpair(int m, const std::vector<double>& a0, double* y) {
  if (m == 1) {
    y[0] = 1.0;
    return a0[0];
  }
  std::vector<double> a(a0), v((size_t)m * m, 0.0), beta(m, 0.0), d(m), e(m, 0.0), p(m);
  for (int k = 0; k + 2 < m; k++) {  // reflection k acts on the indices k + 1 .. m - 1
    double* u = &v[(size_t)k * m];
    // the column below its leading element, summed by itself: as a difference
    // it vanishes for couplings of 1e-8 of that element, which are not small
    double tail = 0.0;
    for (int i = k + 2; i < m; i++) tail += a[(size_t)i * m + k] * a[(size_t)i * m + k];
    const double x0 = a[(size_t)(k + 1) * m + k], xx = x0 * x0 + tail;
    if (!(tail > 0.0)) continue;
    const double alpha = x0 > 0 ? -std::sqrt(xx) : std::sqrt(xx);
    for (int i = k + 1; i < m; i++) u[i] = a[(size_t)i * m + k];
    u[k + 1] -= alpha;
    const double b = 2.0 / (tail + u[k + 1] * u[k + 1]);
    beta[k] = b;
    double up = 0.0;
    for (int i = k + 1; i < m; i++) {
      double q = 0.0;
      for (int j = k + 1; j < m; j++) q += a[(size_t)i * m + j] * u[j];
      p[i] = b * q;
      up += u[i] * p[i];
    }
    for (int i = k + 1; i < m; i++) p[i] -= 0.5 * b * up * u[i];
    for (int i = k + 1; i < m; i++)
      for (int j = k + 1; j < m; j++) a[(size_t)i * m + j] -= u[i] * p[j] + p[i] * u[j];
    a[(size_t)(k + 1) * m + k] = alpha;
  }
  double lo = INFINITY, hi = INFINITY, scale = 0.0;
  for (int i = 0; i < m; i++) {
    d[i] = a[(size_t)i * m + i];
    if (i + 1 < m) e[i] = a[(size_t)(i + 1) * m + i];
  }
  for (int i = 0; i < m; i++) {
    const double rad = (i ? std::fabs(e[i - 1]) : 0.0) + std::fabs(e[i]);
    lo = std::fmin(lo, d[i] - rad);
    hi = std::fmin(hi, d[i]);  // the lowest eigenvalue is at most the lowest diagonal entry
    scale = std::fmax(scale, std::fabs(d[i]) + rad);
  }
  const double tiny = scale * 1e-300 + 1e-300;
  for (int it = 0; it < 200 && hi - lo > 2.3e-16 * std::fmax(std::fabs(lo), std::fabs(hi)); it++) {
    const double mid = 0.5 * (lo + hi);
    if (mid <= lo || mid >= hi) break;
    double q = d[0] - mid;
    bool neg = q < 0.0;
    for (int i = 1; i < m && !neg; i++) {
      if (std::fabs(q) < tiny) q = tiny;
      q = d[i] - mid - e[i - 1] * e[i - 1] / q;
      neg = q < 0.0;
    }
    if (neg) hi = mid;
    else lo = mid;
  }
  // inverse iteration: (T - lo) by Gaussian elimination with row exchanges
  const double mu = lo, small = scale * 2.3e-16 + 1e-300;
  std::vector<double> c0(m), c1(m), c2(m), mult(m);
  std::vector<char> swp(m, 0);
  for (int i = 0; i < m; i++) {
    c0[i] = d[i] - mu;
    c1[i] = e[i];
    c2[i] = 0.0;
  }
  for (int i = 0; i + 1 < m; i++) {
    double below = e[i];  // entry (i + 1, i)
    if (std::fabs(below) > std::fabs(c0[i])) {
      swp[i] = 1;
      const double r0 = c0[i], r1 = c1[i];
      c0[i] = below;
      c1[i] = c0[i + 1];
      c2[i] = c1[i + 1];
      below = r0;
      mult[i] = below / c0[i];
      c0[i + 1] = r1 - mult[i] * c1[i];
      c1[i + 1] = -mult[i] * c2[i];
    } else {
      if (std::fabs(c0[i]) < small) c0[i] = small;
      mult[i] = below / c0[i];
      c0[i + 1] -= mult[i] * c1[i];
    }
  }
  if (std::fabs(c0[m - 1]) < small) c0[m - 1] = small;
  for (int i = 0; i < m; i++) y[i] = 1.0 + 0.01 * i;
  for (int it = 0; it < 4; it++) {
    if (it)  // the first right-hand side is taken as eliminated already
      for (int i = 0; i + 1 < m; i++) {
        if (swp[i]) std::swap(y[i], y[i + 1]);
        y[i + 1] -= mult[i] * y[i];
      }
    double big = 0.0;
    for (int i = m - 1; i >= 0; i--) {
      double b = y[i];
      if (i + 1 < m) b -= c1[i] * y[i + 1];
      if (i + 2 < m) b -= c2[i] * y[i + 2];
      y[i] = b / c0[i];
      big = std::fmax(big, std::fabs(y[i]));
    }
    for (int i = 0; i < m; i++) y[i] /= big;
  }
  for (int k = m - 3; k >= 0; k--) {
    if (beta[k] == 0.0) continue;
    const double* u = &v[(size_t)k * m];
    double q = 0.0;
    for (int i = k + 1; i < m; i++) q += u[i] * y[i];
    for (int i = k + 1; i < m; i++) y[i] -= beta[k] * q * u[i];
  }
  double nn = 0.0;
  for (int i = 0; i < m; i++) nn += y[i] * y[i];
  nn = 1.0 / std::sqrt(nn);
  for (int i = 0; i < m; i++) y[i] *= nn;
  double theta = 0.0;
  for (int i = 0; i < m; i++)
    for (int j = 0; j < m; j++) theta += y[i] * a0[(size_t)i * m + j] * y[j];
  return theta;
}

}  // namespace qp
