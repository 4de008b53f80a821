// Piecewise polynomials of the pair bracket for the FP64 kernels (pair64.cu).
//
// With s = u^2 = r^2 / (2 x_s)^2 the functions of Eq. p3m_gravity's short-range
// half do not depend on the simulation's parameters:
//   b(s) = [erfc(u) + 2u/sqrt(pi) e^{-u^2}] / u^3      B = b / (2 x_s)^3 (no softening)
//   q(s) = s^{-3/2}                                    the point-mass and Plummer shapes
//   h(s) = q(s) - b(s) = 4/sqrt(pi) int_0^1 x^2 e^{-s x^2} dx   (regular at s = 0)
// and their s-derivatives give B'(r)/r.  b and q (and derivatives) are tabulated on
// 64 intervals per octave of s, h and h' on intervals of 1/16, each interval holding
// a polynomial of degree 6 in s - (interval middle).
//
// The tables hold B and B'(r)/r themselves: each simulation's split scale is multiplied in
// when they are filled, before the value at the middle is rounded.
//
// The coefficients are the Taylor series at the middle, cut to degree 6 by Chebyshev
// telescoping.  The series come from the differential equation
// s b' = -(3/2) b - (2/sqrt(pi)) e^{-s}; the value at the middle is summed in
// double-double arithmetic (Dekker 1971, Knuth).  Against 30-digit values the polynomials
// are within 1.4e-16 of the point-mass bracket s^{-3/2} everywhere (relative).
#pragma once

#include <cmath>

#include "common.cuh"

namespace p3m {

constexpr int kTabDeg = 6;                  // degree of every polynomial
constexpr int kTabRow = kTabDeg + 1;        // doubles per interval
constexpr int kTabLogBits = 6;              // 2^6 intervals per octave of s
constexpr int kTabLogShift = 23 - kTabLogBits;
constexpr int kTabLogMinExp = -12;          // logarithmic tables cover s in [2^-12, 2^4)
constexpr int kTabLogMaxExp = 4;
constexpr int kTabLogRows = (kTabLogMaxExp - kTabLogMinExp) << kTabLogBits;
constexpr int kTabLogFirst = (127 + kTabLogMinExp) << kTabLogBits;  // (float bits of s) >> kTabLogShift of row 0
constexpr int kTabUniPerUnit = 16;          // uniform tables: intervals per unit of s, s in [0, 8)
constexpr int kTabUniRows = 8 * kTabUniPerUnit;
constexpr int kTabDoubles = (2 * kTabLogRows + 2 * kTabUniRows) * kTabRow;  // f, f', h, h'
constexpr int kTabTaylor = 10;              // Taylor terms before the telescoping

struct DD {  // value hi + lo
  double hi, lo;
};

#define P3M_HD __host__ __device__ __forceinline__

P3M_HD DD dd_sum(double a, double b) {  // exact
  const double s = a + b, t = s - a;
  return DD{s, (a - (s - t)) + (b - t)};
}
P3M_HD DD dd_prod(double a, double b) {  // exact
  const double p = a * b;
  return DD{p, fma(a, b, -p)};
}
P3M_HD DD dd_norm(double hi, double lo) {
  const double s = hi + lo;
  return DD{s, lo - (s - hi)};
}
P3M_HD DD dd_add(DD a, DD b) {
  const DD s = dd_sum(a.hi, b.hi);
  return dd_norm(s.hi, s.lo + (a.lo + b.lo));
}
P3M_HD DD dd_mul(DD a, DD b) {
  const DD p = dd_prod(a.hi, b.hi);
  return dd_norm(p.hi, p.lo + (a.hi * b.lo + a.lo * b.hi));
}
P3M_HD DD dd_div(DD a, DD b) {
  const double q = a.hi / b.hi;
  const DD p = dd_mul(DD{q, 0.0}, b);
  const double r = (a.hi - p.hi) + (a.lo - p.lo);
  return dd_norm(q, r / b.hi);
}

// Coefficients of the two power series below, made once on the host (make_series_dd), so
// that no division stands in the chain of a summation.
constexpr int kTabSeries = 86;
struct SeriesDD {
  DD s[kTabSeries];  // 1 / (3 5 7 ... (2 j + 3))
  DD e[kTabSeries];  // 1 / j!
};
inline SeriesDD make_series_dd() {
  SeriesDD t;
  t.s[0] = dd_div(DD{1.0, 0.0}, DD{3.0, 0.0});
  t.e[0] = DD{1.0, 0.0};
  for (int j = 1; j < kTabSeries; ++j) {
    t.s[j] = dd_div(t.s[j - 1], DD{2.0 * j + 3.0, 0.0});
    t.e[j] = dd_div(t.e[j - 1], DD{(double)j, 0.0});
  }
  return t;
}
P3M_HD int series_terms(double m) { return 20 + (int)(4.0 * m); }  // remainders below 1e-20 for m < 16

P3M_HD DD dd_step(DD s, double y, DD c) {  // s y + c
  const DD p = dd_prod(s.hi, y);
  const DD t = dd_sum(p.hi, c.hi);
  return dd_norm(t.hi, t.lo + (fma(s.lo, y, p.lo) + c.lo));
}

// S_0(m) = int_0^1 x^2 e^{m (1 - x^2)} dx = sum_j (2m)^j / (3 5 ... (2j + 3)) and E = e^m, all
// terms positive.
P3M_HD void series_se(const SeriesDD& t, double m, DD& S, DD& E) {
  const int n = series_terms(m);
  S = t.s[n];
  E = t.e[n];
  for (int j = n - 1; j >= 0; --j) {
    S = dd_step(S, 2.0 * m, t.s[j]);
    E = dd_step(E, m, t.e[j]);
  }
}

// S_k(m) = int_0^1 x^(2k+2) e^{m (1 - x^2)} dx = (1 + 2m S_{k+1}) / (2k + 3), downwards.
P3M_HD void series_sk(double m, double (&S)[kTabTaylor + 1]) {
  double s = 0.0;
  for (int k = kTabTaylor + series_terms(m); k > kTabTaylor; --k) s = fma(2.0 * m, s, 1.0) / (2.0 * k + 3.0);
#pragma unroll
  for (int k = kTabTaylor; k >= 0; --k) {
    s = fma(2.0 * m, s, 1.0) * (1.0 / (2.0 * k + 3.0));
    S[k] = s;
  }
}

P3M_HD DD pow_m32(double m) {  // m^{-3/2}
  const double y = 1.0 / sqrt(m);
  const DD y2 = dd_prod(y, y);
  const DD my2 = dd_mul(y2, DD{m, 0.0});
  const double e = (1.0 - my2.hi) - my2.lo;
  const DD r = dd_norm(y, 0.5 * y * e);
  return dd_mul(dd_mul(r, r), r);
}

// Cut the polynomial c[0 .. kTabTaylor] in t, |t| <= w, to degree kTabDeg by dropping its
// highest Chebyshev terms one by one.
P3M_HD void telescope(double (&c)[kTabTaylor + 1], double w) {  // w: a power of two
  double wk = 1.0;
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) {
    c[k] *= wk;
    wk *= w;
  }
#pragma unroll
  for (int n = kTabTaylor; n > kTabDeg; --n) {
    // x^n - T_n(x) / 2^(n-1) holds the powers n - 2, n - 4, ...
    double v = c[n];
#pragma unroll
    for (int j = n; j >= 2; j -= 2) {
      v *= -((double)(j * (j - 1)) / (double)((n - j + 2) * (n + j - 2)));
      c[j - 2] -= v;
    }
    c[n] = 0.0;
  }
  const double iw = 1.0 / w;
  wk = 1.0;
#pragma unroll
  for (int k = 0; k <= kTabDeg; ++k) {
    c[k] *= wk;
    wk *= iw;
  }
}

// Interval `row` of the logarithmic tables: plummer = false: b and b', true: q and q',
// times sf and sfd.
P3M_HD void table_log_row(const SeriesDD& t, int row, bool plummer, DD sf, double sfd, double* f, double* fd) {
  const double octave = ldexp(1.0, kTabLogMinExp + (row >> kTabLogBits));
  const int i = row & ((1 << kTabLogBits) - 1);
  const double w = octave / (2 << kTabLogBits);
  const double m = octave + (2 * i + 1) * w;
  const DD q = pow_m32(m);
  double a[kTabTaylor + 2];
  double src = 0.0;  // (2/sqrt(pi)) e^{-m}: the inhomogeneous term of b's equation
  DD v = q;
  if (!plummer) {
    DD S, E;
    series_se(t, m, S, E);
    const DD h = dd_mul(dd_div(S, E), DD{0x1.20dd750429b6dp+1, 0x1.1ae3a914fed8p-55});  // 4/sqrt(pi)
    v = dd_add(q, DD{-h.hi, -h.lo});
    src = 0x1.20dd750429b6dp+0 / E.hi;
  }
  a[0] = v.hi;
  const double im = 1.0 / m;
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) {
    a[k + 1] = -((k + 1.5) * a[k] + src) * (im * (1.0 / (k + 1)));
    src *= -1.0 / (k + 1);
  }
  double c[kTabTaylor + 1];
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) c[k] = (k == 0 ? dd_mul(v, sf).hi : a[k] * sf.hi);
  telescope(c, w);
#pragma unroll
  for (int k = 0; k <= kTabDeg; ++k) f[k] = c[k];
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) c[k] = (k + 1) * a[k + 1] * sfd;
  telescope(c, w);
#pragma unroll
  for (int k = 0; k <= kTabDeg; ++k) fd[k] = c[k];
}

// Interval `row` of the uniform tables: h and h', times sf and sfd.
P3M_HD void table_uni_row(const SeriesDD& t, int row, DD sf, double sfd, double* f, double* fd) {
  const double w = 0.5 / kTabUniPerUnit;
  const double m = (2 * row + 1) * w;
  double S[kTabTaylor + 1];
  series_sk(m, S);
  DD S0, E;
  series_se(t, m, S0, E);
  const DD h = dd_mul(dd_div(S0, E), DD{0x1.20dd750429b6dp+1, 0x1.1ae3a914fed8p-55});
  double a[kTabTaylor + 1], c[kTabTaylor + 1];
  double fact = 0x1.20dd750429b6dp+1 / E.hi;  // (4/sqrt(pi)) e^{-m} (-1)^k / k!
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) {
    a[k] = k == 0 ? h.hi : fact * S[k];
    fact *= -1.0 / (k + 1);
  }
#pragma unroll
  for (int k = 0; k <= kTabTaylor; ++k) c[k] = (k == 0 ? dd_mul(h, sf).hi : a[k] * sf.hi);
  telescope(c, w);
#pragma unroll
  for (int k = 0; k <= kTabDeg; ++k) f[k] = c[k];
#pragma unroll
  for (int k = 0; k < kTabTaylor; ++k) c[k] = (k + 1) * a[k + 1] * sfd;
  c[kTabTaylor] = 0.0;
  telescope(c, w);
#pragma unroll
  for (int k = 0; k <= kTabDeg; ++k) fd[k] = c[k];
}

}  // namespace p3m
