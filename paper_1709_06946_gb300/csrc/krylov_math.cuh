// Small dense FP64 algebra of the Krylov iterations, compiled for the host and
// the device (the device copy runs inside the Lanczos control kernel).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace pse {

// Symmetric tridiagonal eigen-decomposition by the implicit QL method with
// shifts from the leading 2x2 block (Wilkinson).  d[0..n): diagonal, replaced
// by the eigenvalues; e[0..n): off-diagonal in e[0..n-1), destroyed; Z: n x n
// row-major, Z[i*n+k] = component i of eigenvector k.  Returns false when an
// eigenvalue needs more than 100 sweeps.
__host__ __device__ inline bool tql_eigen(int n, double *d, double *e, double *Z) {
  for (int i = 0; i < n; ++i)
    for (int k = 0; k < n; ++k) Z[i * n + k] = i == k ? 1.0 : 0.0;
  if (n > 0) e[n - 1] = 0.0;
  const double eps = 2.220446049250313e-16;
  for (int l = 0; l < n; ++l) {
    for (int iter = 0;; ++iter) {
      int m = l;
      for (; m < n - 1; ++m) {
        double dd = fabs(d[m]) + fabs(d[m + 1]);
        if (fabs(e[m]) <= eps * dd) break;
      }
      if (m == l) break;
      if (iter > 100) return false;
      double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
      double rr = hypot(g, 1.0);
      g = d[m] - d[l] + e[l] / (g + (g >= 0 ? rr : -rr));
      double s = 1.0, c = 1.0, pp = 0.0;
      bool deflated = false;
      for (int i = m - 1; i >= l; --i) {
        double f = s * e[i], b = c * e[i];
        rr = hypot(f, g);
        e[i + 1] = rr;
        if (rr == 0.0) {  // underflow: split the problem
          d[i + 1] -= pp;
          e[m] = 0.0;
          deflated = true;
          break;
        }
        s = f / rr;
        c = g / rr;
        g = d[i + 1] - pp;
        rr = (d[i] - g) * s + 2.0 * c * b;
        pp = s * rr;
        d[i + 1] = g + pp;
        g = c * rr - b;
        for (int k = 0; k < n; ++k) {  // rotate columns i, i+1 of Z
          double zf = Z[k * n + i + 1];
          Z[k * n + i + 1] = s * Z[k * n + i] + c * zf;
          Z[k * n + i] = c * Z[k * n + i] - s * zf;
        }
      }
      if (deflated) continue;
      d[l] -= pp;
      e[l] = g;
      e[m] = 0.0;
    }
  }
  return true;
}

// cvec = T^{1/2} e1 for the symmetric tridiagonal T = tridiag(beta, alpha, beta)
// of order n (eigenvalues clamped at zero); work: 2n + n^2 doubles.
__host__ __device__ inline bool tridiag_sqrt_e1(int n, const double *alpha, const double *beta, double *work,
                                                double *cvec) {
  double *d = work, *e = work + n, *Z = work + 2 * n;
  for (int i = 0; i < n; ++i) {
    d[i] = alpha[i];
    e[i] = i < n - 1 ? beta[i] : 0.0;
  }
  if (!tql_eigen(n, d, e, Z)) return false;
  for (int i = 0; i < n; ++i) {
    double s = 0.0;
    for (int k = 0; k < n; ++k) s += Z[i * n + k] * sqrt(d[k] > 0.0 ? d[k] : 0.0) * Z[k];
    cvec[i] = s;
  }
  return true;
}

// Rational form of the square root on the spectral window [hi / SQRT_WINDOW, hi]:
//   sqrt(x) = sqrt(hi) x sum_k w_k / (x + hi s_k),
// the contour quadrature with the Jacobi-elliptic map of Hale, Higham and Trefethen
// (SIAM J. Numer. Anal. 46, 2505, 2008, their method for the square root).  With
// n nodes its relative error is about exp(-2 pi^2 n / (ln SQRT_WINDOW + 3)): 31 nodes
// and a window of 10^6 reach the FP64 rounding level.
constexpr int SQRT_NODES = 31;
constexpr double SQRT_WINDOW = 1e6;

// Nodes s[0..n) and weights w[0..n) (host).  With m = 1 - 1/window, K = K(m) and
// t_k = sc((k + 1/2) K / n | m): s = t^2 / window and, from sc' = dn / cn^2 =
// sqrt((1 + t^2/window)(1 + t^2)), w = 2 K sc' / (pi n sqrt(window)).  sc comes from
// the theta series of the complementary nome (about 6e-8 here: three terms).
inline void sqrt_nodes(int n, double window, double *s, double *w) {
  const double pi = 3.14159265358979323846;
  auto agm = [](double a, double b) {
    for (int i = 0; i < 40 && fabs(a - b) > 1e-16 * a; ++i) {
      const double m = 0.5 * (a + b);
      b = sqrt(a * b);
      a = m;
    }
    return 0.5 * (a + b);
  };
  const double kc2 = 1.0 / window;                                  // complementary parameter
  const double K = pi / (2.0 * agm(1.0, sqrt(kc2)));                // K(1 - kc2)
  const double K1 = pi / (2.0 * agm(1.0, sqrt(1.0 - kc2)));         // K(kc2)
  const double q = exp(-pi * K / K1);
  double th2 = 0.0, th3 = 1.0;
  for (int j = 0; j < 6; ++j) {
    th2 += 2.0 * pow(q, (j + 0.5) * (j + 0.5));
    if (j > 0) th3 += 2.0 * pow(q, (double)j * j);
  }
  for (int k = 0; k < n; ++k) {
    const double y = pi * (k + 0.5) * K / n / (2.0 * K1);           // sn(iu | kc2) = i sc(u | m)
    double th1 = 0.0, th4 = 1.0;
    for (int j = 0; j < 6; ++j) {
      const double sg = j % 2 ? -1.0 : 1.0;
      th1 += 2.0 * sg * pow(q, (j + 0.5) * (j + 0.5)) * sinh((2 * j + 1) * y);
      if (j > 0) th4 += 2.0 * sg * pow(q, (double)j * j) * cosh(2 * j * y);
    }
    const double t = th3 * th1 / (th2 * th4);
    s[k] = t * t * kc2;
    w[k] = 2.0 * K / (pi * n) * sqrt(kc2) * sqrt((1.0 + t * t * kc2) * (1.0 + t * t));
  }
}

// 1 / d and sqrt(x) in FP64, to two units in the last place.  On the device, for arguments well
// inside the FP32 range, an FP32 seed (7 digits) and two Newton steps (14, then FP64's
// 16): the FP64 unit issues one warp instruction in sixteen cycles and the library forms
// are serial chains of several tens of them.
__host__ __device__ inline double recip(double d) {
#ifdef __CUDA_ARCH__
  const float f = (float)d;
  if (fabsf(f) > 1e-30f && fabsf(f) < 1e30f) {
    double r = (double)(1.0f / f);
    r = fma(r, fma(-d, r, 1.0), r);
    return fma(r, fma(-d, r, 1.0), r);
  }
#endif
  return 1.0 / d;
}
__host__ __device__ inline double root(double x) {
#ifdef __CUDA_ARCH__
  const float f = (float)x;
  if (f > 1e-30f && f < 1e30f) {
    double y = (double)rsqrtf(f);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    const double s = x * y;
    return fma(0.5 * y, fma(-s, s, x), s);
  }
#endif
  return sqrt(x);
}

// x = (T + shift)^{-1} e1 for T = tridiag(beta, alpha, beta) of order n, eliminated from
// the last row up (one reciprocal per row; T of order one); x[i] at x[i * stride].
// Returns true when every pivot is positive, i.e. when T + shift is positive definite.
__host__ __device__ inline bool shifted_solve_e1(int n, const double *alpha, const double *beta, double shift,
                                                 double *x, int stride) {
  double d = alpha[n - 1] + shift;
  bool spd = d > 0.0;
  for (int i = n - 1; i > 0; --i) {
    const double b = beta[i - 1], f = b * recip(d);
    x[i * stride] = -f;  // x_i = -f x_{i-1}
    d = alpha[i - 1] + shift - b * f;
    spd = spd && d > 0.0;
  }
  double v = recip(d);
  x[0] = v;
  for (int i = 1; i < n; ++i) {
    v *= x[i * stride];
    x[i * stride] = v;
  }
  return spd;
}

}  // namespace pse
