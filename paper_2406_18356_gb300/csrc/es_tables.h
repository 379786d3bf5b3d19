// The exponential-of-semicircle kernel's FP64 weight tables: how a plan makes
// them (host) and how the kernels read them (device, and host for the tests).
#pragma once

#include <cmath>
#include <vector>

#ifdef __CUDACC__
#define MS_HD __host__ __device__ __forceinline__
#else
#define MS_HD inline
#endif

namespace ms {

constexpr int kW = 7;          // ES kernel support in cells
constexpr int kHalfW = 3;      // (W - 1) / 2

// The gridding kernel: its shape and, for FP64 plans, the device tables of
// its taps' weights (nullptr: evaluated directly): kEsSegs segments of the
// inner taps (5 x 7 polynomial coefficients, the segment's centre, one pad),
// then of the outer taps (9 coefficients, the centre, one pad).  Odd strides,
// so that lanes in different segments read different banks.
struct EsKernel {
  double beta = 0;
  const double* tab = nullptr;
};
constexpr int kEsSegs = 64, kEsInner = 37, kEsOuter = 11;
constexpr int kEsTable = kEsSegs * (kEsInner + kEsOuter);
constexpr double kEsOuterRange = 0.7;   // of v = sqrt(1 - z^2) at |z| >= 5/7
constexpr double kEsMaxBeta = 32.0;     // the polynomials hold for 0 < beta <= this

// Matrix [n][n] from the values of a function at the n Chebyshev nodes x_i =
// cos(pi (2i + 1) / 2n) of [-1, 1] to the monomial coefficients of its
// interpolating polynomial (Newton's divided differences of unit vectors).
inline std::vector<double> chebyshev_fit(int n, std::vector<double>* nodes) {
  const long double pi = 3.141592653589793238462643383279502884L;
  std::vector<long double> x(n);
  for (int i = 0; i < n; ++i) x[i] = std::cos(pi * (2 * i + 1) / (2.0L * n));
  if (n % 2) x[n / 2] = 0.0L;
  nodes->assign(x.begin(), x.end());
  std::vector<double> m(n * n);
  for (int u = 0; u < n; ++u) {
    std::vector<long double> d(n, 0.0L), p(n, 0.0L);
    d[u] = 1.0L;
    for (int k = 1; k < n; ++k)
      for (int i = n - 1; i >= k; --i) d[i] = (d[i] - d[i - 1]) / (x[i] - x[i - k]);
    for (int i = n - 1; i >= 0; --i) {   // p <- p (x - x_i) + d_i
      for (int k = n - 1; k >= 1; --k) p[k] = p[k - 1] - x[i] * p[k];
      p[0] = d[i] - x[i] * p[0];
    }
    for (int k = 0; k < n; ++k) m[k * n + u] = (double)p[k];
  }
  return m;
}

// The FP64 weight tables (see EsKernel) of the ES kernel with shape beta.  A
// segment's polynomial interpolates the differences from its centre value
// (relative to it, through expm1, so that they keep their digits); the inner
// taps i and 6 - i mirror each other, and the outer function's segments are
// one polynomial of exp(beta x) times their centre values.
inline std::vector<double> es_tables(double beta) {
  std::vector<double> t(kEsTable, 0.0), x7, x9;
  const std::vector<double> f7 = chebyshev_fit(7, &x7), f9 = chebyshev_fit(9, &x9);
  const double c2 = 4.0 / (kW * kW), h = 0.5 / kEsSegs, ho = 0.5 * kEsOuterRange / kEsSegs;
  // out[k] = a c_k / h^k, c the fit of d (d = 0 at the centre), out[0] = a
  auto put = [](const std::vector<double>& fit, int n, const double* d, double a, double h,
                double* out) {
    double hk = 1.0;
    out[0] = a;
    for (int k = 1; k < n; ++k) {
      double s = 0.0;
      hk *= h;
      for (int i = 0; i < n; ++i) s += fit[k * n + i] * d[i];
      out[k] = a * s / hk;
    }
  };
  double d9[9];
  for (int i = 0; i < 9; ++i) d9[i] = std::expm1(beta * ho * x9[i]);
  for (int g = 0; g < kEsSegs; ++g) {
    const double c = -0.5 + (2 * g + 1) * h;
    double* q = &t[g * kEsInner];
    q[kEsInner - 2] = c;
    for (int i = 1; i <= kHalfW; ++i) {
      const double tc = c + (kHalfW - i), z2 = tc * tc * c2, sc = std::sqrt(1.0 - z2);
      double d[7];
      for (int n = 0; n < 7; ++n) {
        const double x = h * x7[n], ds = -c2 * x * (2.0 * tc + x);   // s(tc + x) - s(tc)
        d[n] = std::expm1(beta * ds / (std::sqrt(1.0 - z2 + ds) + sc));
      }
      put(f7, 7, d, std::exp(-beta * z2 / (1.0 + sc)), h, q + (i - 1) * 7);
      double* mirror = &t[(kEsSegs - 1 - g) * kEsInner] + (kW - 2 - i) * 7;
      for (int k = 0; k < 7 && i < kHalfW; ++k) mirror[k] = (k & 1 ? -1 : 1) * q[(i - 1) * 7 + k];
    }
    double* o = &t[kEsSegs * kEsInner + g * kEsOuter];
    o[kEsOuter - 2] = (2 * g + 1) * ho;
    put(f9, 9, d9, std::exp(beta * (o[kEsOuter - 2] - 1.0)), ho, o);
  }
  return t;
}

// FP64 weights from the plan's tables (EsKernel): the inner five taps are
// degree-6 polynomials of f on 64 segments of its range, the outer two
// exp(beta (v - 1)), a degree-8 polynomial on 64 segments of v = sqrt(1 - z^2)
// in [0, 0.7) (smooth there; in f they have a square-root end point).  Their
// errors are roundings: the inner taps' at most 1.9e-16 of the kernel's peak
// for beta from 1e-6 to 32 (1.6e-16 at the default 16.1), the outer taps' below
// 2e-16 besides that of v at the support's edge, where the direct evaluation
// loses the same digits.  A scheduler issues one FP64 instruction per 76
// cycles, and the library's exp, sqrt and division spend most of the
// operator's on the 14 weights of a row: some 170 of them this way.  Measured
// at 128 px, 31,744 rows (with the smaller work items): the residual image 374
// -> 203 us, degridding 20.9 and gridding 30.9 us of it; 5.9M rows 16.1 -> 9.0
// ms.
MS_HD void es_weights_tab(double f, const double* tab, double* w) {
  int seg = (int)(((float)f + 0.5f) * kEsSegs);
  seg = seg < 0 ? 0 : (seg >= kEsSegs ? kEsSegs - 1 : seg);
  const double* c = tab + seg * kEsInner;
  const double x = f - c[kEsInner - 2];
#pragma unroll
  for (int i = 1; i < kW - 1; ++i) {
    const double* q = c + (i - 1) * 7;
    double a = q[6];
#pragma unroll
    for (int k = 5; k >= 0; --k) a = fma(a, x, q[k]);
    w[i] = a;
  }
#pragma unroll
  for (int i = 0; i < kW; i += kW - 1) {
    const double t = f + (double)(kHalfW - i);
    double s = fma(t * (-4.0 / (kW * kW)), t, 1.0);
    s = s > 0.0 ? s : 0.0;
    const double v = sqrt(s);
    const int g = (int)((float)v * (float)(kEsSegs / kEsOuterRange));
    const double* q = tab + kEsSegs * kEsInner + (g < kEsSegs ? g : kEsSegs - 1) * kEsOuter;
    const double y = v - q[kEsOuter - 2];
    double a = q[8];
#pragma unroll
    for (int k = 7; k >= 0; --k) a = fma(a, y, q[k]);
    w[i] = a;
  }
}


}  // namespace ms
