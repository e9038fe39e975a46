// sk_factors64.h -- table of the FP64 kernel factors of the regularized pairs
// (host construction; sk_pair64.cu evaluates it).
//
// With x = rho^2 the pair sums need F_n(x) = s(rho) / rho^n: n = 1 for s1,
// n = 3 for s2 (Sec. 3.4), n = 5 for the stresslet's s3. All three are entire
// in x and, from s_i'(p) = poly(p) e^{-p^2} (sk_series.cuh), satisfy
//
//   x F' + (n/2) F = E(x),   E(x) = A (x^2 - a x + b) e^{-x},
//
//   n = 1: A = 4/(3 sqrt pi),  a = 4, b = 2
//   n = 3: A = 8/(3 sqrt pi),  a = 6, b = 6
//   n = 5: A = 16/(9 sqrt pi), a = 8, b = 12.
//
// In powers of t about an interval's middle m this is the recurrence
//   F_{k+1} = (E_k - (k + n/2) F_k) / (m (k + 1)),
// E_k the Taylor coefficients of E there. A rounding error of F_0 grows like
// m^{-k}, and |t| <= m in every interval, so the sum keeps F_0's accuracy.
// F_0 comes from the power series at 0 (x < 2) or the closed form, in long
// double; the table holds values rounded once to double (float for the tail).
//
// Intervals: y = 1 + x in [1, 256), 2^F64_SUB_BITS per octave of y, so that the
// interval of a pair is the top bits of the double y. Half an interval is at
// most 2^-8 y: the terms from t^4 on are below 2^-30 of F and are kept in FP32.
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

namespace sk {

constexpr int F64_SUB_BITS = 7;
constexpr int F64_OCTAVES = 8;
constexpr int F64_N = F64_OCTAVES << F64_SUB_BITS;  // intervals
constexpr int F64_HEAD = 4;                         // FP64 coefficients t^0 .. t^3
// FP32 coefficients from t^4 on: to t^6 for n = 1, 3 and t^7 for n = 5 (the
// first term left out is below 2^-54 of F at the interval's edge)
constexpr int F64_TAIL_SL = 3, F64_TAIL_DL = 4;

// Byte layout of one layer's table: heads [function][F64_HEAD][F64_N] double,
// then tails [function][tail][F64_N] float. Functions: s1, s2 (single layer);
// s3 (double layer). The double layer's table follows the single layer's.
constexpr size_t f64_table_bytes(bool dl) {
  return (dl ? 1 : 2) * (size_t)F64_N *
         (F64_HEAD * sizeof(double) + (dl ? F64_TAIL_DL : F64_TAIL_SL) * sizeof(float));
}
constexpr size_t F64_TABLES_BYTES = f64_table_bytes(false) + f64_table_bytes(true);

// Power series of the three functions at 0: F_n(x) = sum_k c_k x^k, c_k the coefficient
// of x^k in 2A (x^2 - a x + b) e^{-x} over 2k + n. At x < 2 the 40 terms leave out less
// than 2^-110 of F.
constexpr int F64_SERIES = 40;
struct F64Series {
  long double c[3][F64_SERIES];
};
inline F64Series f64_series() {
  const long double isp = 0.564189583547756286948079451560772586L;  // 1/sqrt(pi)
  F64Series s;
  for (int f = 0; f < 3; ++f) {
    const int n = 2 * f + 1;
    const long double a = n == 1 ? 4 : n == 3 ? 6 : 8, b = n == 1 ? 2 : n == 3 ? 6 : 12;
    const long double A2 = (n == 1 ? 8.0L / 3 : n == 3 ? 16.0L / 3 : 32.0L / 9) * isp;
    long double e0 = 1, e1 = 0, e2 = 0;  // e_k, e_{k-1}, e_{k-2}; e_k = (-1)^k/k!
    for (int k = 0; k < F64_SERIES; ++k) {
      s.c[f][k] = A2 * (b * e0 - a * e1 + e2) / (2 * k + n);
      e2 = e1;
      e1 = e0;
      e0 = -e0 / (k + 1);
    }
  }
  return s;
}

// What the three functions share at the middle m of an interval. (long double is
// software on Arm: with 60 series terms, exponential and error function for each function
// the table took 16.4 ms of a process's first context there; 5.6 ms like this.)
struct F64Point {
  long double m, im, p, ex, er;  // m, 1/m, sqrt m, e^-m, erf p
};
inline F64Point f64_point(long double m) {
  F64Point q;
  q.m = m;
  q.im = 1 / m;
  q.p = std::sqrt(m);
  const bool tail = m < 80;  // beyond: e^-m times any factor's polynomial is below 2^-90
  q.ex = tail ? std::exp(-m) : 0;
  q.er = tail ? std::erf(q.p) : 1;
  return q;
}

// F_n at q, n = 1, 3, 5.
inline long double f64_factor(int n, const F64Point& q, const F64Series& series) {
  if (q.m < 2.0L) {
    const long double* c = series.c[n / 2];
    long double s = c[F64_SERIES - 1];
    for (int k = F64_SERIES - 2; k >= 0; --k) s = s * q.m + c[k];
    return s;
  }
  const long double isp = 0.564189583547756286948079451560772586L;
  const long double x = q.m, p = q.p, g = q.ex * isp;
  if (n == 1) return (q.er - 2.0L / 3 * p * (2 * x - 5) * g) / p;
  if (n == 3) return (q.er - 2.0L / 3 * p * ((4 * x - 14) * x + 3) * g) / (p * x);
  return (q.er - 2.0L / 9 * p * (((8 * x - 36) * x + 6) * x + 9) * g) / (p * x * x);
}

// Taylor coefficients F_0 .. F_{K-1} of F_n about q.
inline void f64_taylor(int n, const F64Point& q, const F64Series& series, int K, long double* F) {
  const long double isp = 0.564189583547756286948079451560772586L;
  const long double A = (n == 1 ? 4.0L / 3 : n == 3 ? 8.0L / 3 : 16.0L / 9) * isp;
  const long double a = n == 1 ? 4 : n == 3 ? 6 : 8, b = n == 1 ? 2 : n == 3 ? 6 : 12;
  const long double q0 = (q.m - a) * q.m + b, q1 = 2 * q.m - a;  // x^2 - a x + b = q0 + q1 t + t^2
  long double e0 = A * q.ex, e1 = 0, e2 = 0;  // A e^{-m} (-1)^k / k!, k, k-1, k-2
  F[0] = f64_factor(n, q, series);
  for (int k = 0; k + 1 < K; ++k) {
    const long double E = q0 * e0 + q1 * e1 + e2, ik = 1.0L / (k + 1);
    F[k + 1] = (E - (k + 0.5L * n) * F[k]) * (q.im * ik);
    e2 = e1;
    e1 = e0;
    e0 = -e0 * ik;
  }
}

// Both layers' tables into out (F64_TABLES_BYTES).
inline void f64_build_tables(char* out) {
  const F64Series series = f64_series();
  for (int i = 0; i < F64_N; ++i) {
    const int oct = i >> F64_SUB_BITS, sub = i & ((1 << F64_SUB_BITS) - 1);
    const long double y =
        std::ldexp(1.0L + (sub + 0.5L) / (1 << F64_SUB_BITS), oct);  // middle of the interval
    const F64Point q = f64_point(y - 1);
    for (int n = 1; n <= 5; n += 2) {
      const bool dl = n == 5;
      const int nf = dl ? 1 : 2, f = dl ? 0 : n / 2, tail = dl ? F64_TAIL_DL : F64_TAIL_SL;
      double* head = reinterpret_cast<double*>(out + (dl ? f64_table_bytes(false) : 0));
      float* tl = reinterpret_cast<float*>(head + (size_t)nf * F64_HEAD * F64_N);
      long double F[F64_HEAD + 4];
      f64_taylor(n, q, series, F64_HEAD + tail, F);
      for (int k = 0; k < F64_HEAD; ++k)
        head[((size_t)f * F64_HEAD + k) * F64_N + i] = (double)F[k];
      for (int k = 0; k < tail; ++k)
        tl[((size_t)f * tail + k) * F64_N + i] = (float)F[F64_HEAD + k];
    }
  }
}

}  // namespace sk
