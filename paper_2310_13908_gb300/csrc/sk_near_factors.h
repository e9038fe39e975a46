// sk_near_factors.h -- power-series coefficients of the kernel factors
// s1/p, s2/p^3 and s3/p^5 (derivation: sk_series.cuh), and from them the table of
// local polynomials that the FP64 near sums use. Compile-time values only (a
// CPU test compiles it with the host compiler).
#pragma once

#ifdef __CUDACC__
#define SK_HD __host__ __device__
#else
#define SK_HD
#endif

namespace sk {

constexpr double INV_SQRT_PI = 0.56418958354775628695;  // 1/sqrt(pi)
constexpr double PI_D = 3.14159265358979323846;

SK_HD constexpr double ecoef(int k) {
  if (k < 0) return 0.0;
  double v = 1.0;
  for (int i = 1; i <= k; ++i) v /= (double)i;
  return (k & 1) ? -v : v;
}

template <int N>
struct Poly {
  double c[N];
};

// which = 1: s1/p, 2: s2/p^3, 3: s3/p^5 (prefactor included)
template <int WHICH, int N>
SK_HD constexpr Poly<N> series_coefs() {
  Poly<N> P{};
  for (int n = 0; n < N; ++n) {
    double v = 0.0;
    if (WHICH == 1)
      v = (8.0 / 3.0) * INV_SQRT_PI * (2.0 * ecoef(n) - 4.0 * ecoef(n - 1) + ecoef(n - 2)) /
          (2.0 * n + 1.0);
    else if (WHICH == 2)
      v = (16.0 / 3.0) * INV_SQRT_PI * (6.0 * ecoef(n) - 6.0 * ecoef(n - 1) + ecoef(n - 2)) /
          (2.0 * n + 3.0);
    else
      v = (32.0 / 9.0) * INV_SQRT_PI * (12.0 * ecoef(n) - 8.0 * ecoef(n - 1) + ecoef(n - 2)) /
          (2.0 * n + 5.0);
    P.c[n] = v;
  }
  return P;
}

// The factors for x < NEAR_X_MAX (the FP64 near pairs of SK_FP32C at the default
// rho_T = 0.5): local polynomials about the middles of NEAR_N intervals, from
// the series above. With |t| <= 1/64 the terms from t^5 on are below 2^-36 of
// the factor and run in FP32, so that a factor takes 5 FP64 instructions
// instead of 12 (the FP64 pipe bounds the near sums; the gathered loads of
// the coefficients hit L1).
constexpr int NEAR_N = 8;
constexpr double NEAR_X_MAX = 0.25;
struct NearFactors {
  double c[3][5][NEAR_N];  // s1/p, s2/p^3, s3/p^5
  float t[3][3][NEAR_N];
};
template <int WHICH>
SK_HD constexpr void near_factor_coefs(NearFactors& f) {
  const Poly<18> P = series_coefs<WHICH, 18>();
  for (int i = 0; i < NEAR_N; ++i) {
    const double m = (i + 0.5) * (NEAR_X_MAX / NEAR_N);
    for (int k = 0; k < 8; ++k) {  // coefficient of t^k: sum_n P_n C(n, k) m^(n - k)
      double s = 0.0;
      for (int n = 17; n >= k; --n) {
        double b = P.c[n];
        for (int q = 0; q < k; ++q) b = b * (double)(n - q) / (double)(q + 1);
        s = s * m + b;
      }
      if (k < 5)
        f.c[WHICH - 1][k][i] = s;
      else
        f.t[WHICH - 1][k - 5][i] = (float)s;
    }
  }
}
SK_HD constexpr NearFactors near_factors() {
  NearFactors f{};
  near_factor_coefs<1>(f);
  near_factor_coefs<2>(f);
  near_factor_coefs<3>(f);
  return f;
}

}  // namespace sk
