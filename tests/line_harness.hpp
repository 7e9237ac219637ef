// A whole 1D right-hand side of the Euler equations (NC = 3; NC = 4 with a
// tangential momentum, a row of a 2D grid) on the host, three ways: the paper's
// formulas in 128-bit floating point, the same in FP64 on cell differences, and
// the integer path of csrc/weno_fixed.cuh.  FP64 inputs are the same for all.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <random>
#include <vector>

#include "weno_fixed.cuh"
#ifdef __x86_64__
typedef __float128 Q;
#else
typedef long double Q;
#endif
using namespace weno::fx;

inline double root(double x) { return std::sqrt(x); }
inline Q root(Q x) {
  Q r = std::sqrt((double)x);
  for (int k = 0; k < 2; ++k) r = (r + x / r) / 2;
  return r;
}
template <class T>
T mag(T x) { return x < 0 ? -x : x; }

// f - v2 of eqs. (11)-(22), p = 1, with a sensitivity term of 0
template <class T>
T correction(const T *d) {
  T s[4], t[4] = {3 * d[1] - d[0], d[1] + d[2], 3 * d[2] - d[3], 3 * d[4] - 5 * d[3]}, b[4], top = 0;
  for (int k = 0; k < 4; ++k) s[k] = d[k + 1] - d[k];
  for (int k = 0; k < 4; ++k) b[k] = (T)13 / 3 * s[k] * s[k] + t[k] * t[k];
  b[3] = (b[0] + b[1] + b[2] + b[3]) / 4;
  const T r5 = s[3] - s[0] + 3 * (s[1] - s[2]), tau = 4 * r5 * r5, D[4] = {1, 9, 9, 1};
  const T r[4] = {5 * d[1] - 2 * d[0], d[1] + 2 * d[2], 4 * d[2] - d[3], 6 * d[2] - 5 * d[3] + 2 * d[4]};
  for (int k = 0; k < 4; ++k) top = std::max(top, std::max(b[k], tau));
  if (top == 0) return 0;
  T num = 0, den = 0;
  for (int k = 0; k < 4; ++k) {
    const T a = D[k] * (1 + (tau / top) / (b[k] / top + (T)1e-80));
    num += a * r[k];
    den += a;
  }
  return num / den / 6;
}

template <int NC>
struct Line {
  std::vector<double> U[NC];
  double gm1;
  int n() const { return (int)U[0].size(); }
};
// cell i of n takes (rho, u, v, p) = at(i)
template <int NC, class At>
Line<NC> line(int n, double gm1, At at) {
  Line<NC> s;
  s.gm1 = gm1;
  for (int i = 0; i < n; ++i) {
    double w[4] = {};
    at(i, w);
    if (NC == 3) w[2] = 0;
    const double E = w[3] / gm1 + 0.5 * w[0] * (w[1] * w[1] + w[2] * w[2]);
    const double U[4] = {w[0], w[0] * w[1], NC == 4 ? w[0] * w[2] : E, E};
    for (int q = 0; q < NC; ++q) s.U[q].push_back(U[q]);
  }
  return s;
}

template <class T>
struct Cell {
  T rho, m, n, E, u, v, p, H, F[4];
};
template <class T, int NC>
Cell<T> cell(const Line<NC> &s, int i) {
  Cell<T> c;
  c.rho = s.U[0][i];
  c.m = s.U[1][i];
  c.n = NC == 4 ? s.U[2][i] : 0.0;
  c.E = s.U[NC - 1][i];
  c.u = c.m / c.rho;
  c.v = c.n / c.rho;
  c.p = (T)s.gm1 * (c.E - (c.m * c.u + c.n * c.v) / 2);
  c.H = (c.E + c.p) / c.rho;
  c.F[0] = c.m;
  c.F[1] = c.m * c.u + c.p;
  c.F[2] = NC == 4 ? c.n * c.u : c.H * c.m;
  c.F[NC - 1] = c.H * c.m;
  return c;
}
template <class T>
struct Face {
  T un, ut, H, c, ic, b1, b2, q2;
};
template <class T>
Face<T> roe(const Cell<T> &L, const Cell<T> &R, double gm1) {
  const T a = root(L.rho), b = root(R.rho);
  Face<T> f;
  f.un = (a * L.u + b * R.u) / (a + b);
  f.ut = (a * L.v + b * R.v) / (a + b);
  f.H = (a * L.H + b * R.H) / (a + b);
  f.q2 = f.un * f.un + f.ut * f.ut;
  f.c = root((T)gm1 * (f.H - f.q2 / 2));
  f.ic = 1 / f.c;
  f.b1 = (T)gm1 * f.ic * f.ic;
  f.b2 = f.b1 * f.q2 / 2;
  return f;
}
// Largest |u - c|, |u|, (|u|,) |u + c|
template <int NC>
void speeds(const Line<NC> &s, double *A) {
  for (int m = 0; m < NC; ++m) A[m] = 0;
  for (int i = 0; i < s.n(); ++i) {
    const Cell<double> x = cell<double>(s, i);
    const double c = std::sqrt((s.gm1 + 1) * x.p / x.rho);
    A[0] = std::max(A[0], std::fabs(x.u - c));
    A[1] = std::max(A[1], std::fabs(x.u));
    A[NC - 1] = std::max(A[NC - 1], std::fabs(x.u + c));
  }
  if (NC == 4) A[2] = A[1];
}
// The fields' h less their centre values at the face of pairs x[0..5], by the formulas in T
template <class T, int NC>
void fields(const Line<NC> &s, const Cell<T> *x, const Face<T> &f, const double *A, int i0, T *h) {
  T w[NC][5], g[NC][5];
  for (int j = 0; j < 5; ++j) {
    T dU[4], dF[4];
    for (int q = 0; q < NC; ++q) {
      dU[q] = (T)s.U[q][i0 + j + 1] - (T)s.U[q][i0 + j];
      dF[q] = x[j + 1].F[q] - x[j].F[q];
    }
    for (int k = 0; k < 2; ++k) {
      const T *d = k ? dF : dU;
      const T mt = NC == 4 ? d[2] : 0;
      const T z = f.b2 * d[0] - f.b1 * (f.un * d[1] + (f.ut * mt - d[NC - 1]));
      const T tc = (f.un * d[0] - d[1]) * f.ic;
      const T o[4] = {z + tc, d[0] - z, NC == 4 ? mt - f.ut * d[0] : z - tc, z - tc};
      for (int m = 0; m < NC; ++m) (k ? g : w)[m][j] = o[m];
    }
  }
  for (int m = 0; m < NC; ++m) {
    T p[5], n[5];
    for (int j = 0; j < 5; ++j) {
      p[j] = (T)A[m] * w[m][j] + g[m][j];
      n[4 - j] = (T)A[m] * w[m][j] - g[m][j];
    }
    h[m] = -(T)A[m] * w[m][2] + correction<T>(p) + correction<T>(n);
  }
}
// The same by the integer path.
template <int NC>
void fields_fixed(const Line<NC> &s, const Cell<double> *x, const Face<double> &f, const double *A,
                  int i0, double *h) {
  const int a = exponent(std::max(A[0], A[NC - 1])) - 1022, a1 = imax(exponent(A[1]) - 1022, a - 300);
  u64 P[2][NC][5];
  int E[NC], B0 = 0, B2 = 0, top = 0;
  for (int q = 0; q < NC; ++q) {
    int eu = 0, ef = 0;
    for (int j = 0; j < 5; ++j) {
      eu = imax(eu, packed_exponent(P[0][q][j] = pack(s.U[q][i0 + j + 1] - s.U[q][i0 + j])));
      ef = imax(ef, packed_exponent(P[1][q][j] = pack(x[j + 1].F[q] - x[j].F[q])));
    }
    E[q] = aligned(eu, ef, a);
    if (q == 0) B0 = aligned(eu, ef, a1);
    if (NC == 4 && q == 2) B2 = aligned(eu, ef, a1);
    top = imax(top, imax(eu, ef));
  }
  for (int m = 0; m < NC; ++m) h[m] = 0;
  if (top == 0) return;
  const LeftRows<NC> rows =
      left_rows<NC>(E, B0, B2, a, a1, f.b2, f.b1, f.un * f.ic, f.b1 * f.un, f.b1 * f.ut, f.ic, f.ut);
  // fields left to FP64
  const int floor = exponent(std::sqrt(x[2].rho)) + exponent(std::sqrt(x[3].rho)) - exponent(f.ic) - 1023;
  unsigned left = strong_fields<NC>(rows, a, a1, f.ic, f.ut, floor);
  if (left)
    left &= uneven_fields<NC>([&](int k, int q, int j) { return P[k][q][j]; }, a, a1, rows.um, rows.ue,
                              rows.us, f.b2, f.b1, f.un * f.ic, f.b1 * f.un, f.b1 * f.ut, f.ic, f.ut);
  double wide[NC];
  if (left) fields<double, NC>(s, x, f, A, i0, wide);
  i64 d[2][NC][5];
  for (int k = 0; k < 2; ++k)
    for (int j = 0; j < 5; ++j) {
      u64 v[NC];
      for (int q = 0; q < NC; ++q) v[q] = P[k][q][j];
      const int as = k ? a : 0, as1 = k ? a1 : 0;
      const Proj p = project<NC>(rows, E, as, as1, v);
      d[k][0][j] = p.z + p.tc;
      d[k][1][j] = entropy<NC>(rows, as, as1, p);
      if constexpr (NC == 4) d[k][2][j] = project_shear(rows, B0, as1, v[0], v[2]);
      d[k][NC - 1][j] = p.z - p.tc;
    }
  for (int m = 0; m < NC; ++m) {
    const bool slow = m > 0 && m < NC - 1;
    const int k0 = (!slow ? rows.um + a : m == 1 ? rows.ue + a1 : rows.us + a1) - 1592;
    if (left >> m & 1) {
      h[m] = wide[m];
      continue;
    }
    i64 *w = d[0][m], *g = d[1][m], X[5], G[5], p[5], n[5];
    for (int j = 0; j < 5; ++j) {
      X[j] = times_speed(speed(A[m], slow ? a1 : a), w[j]);
      G[j] = g[j];
      p[j] = (X[j] + G[j]) >> 2;
      n[4 - j] = (X[j] - G[j]) >> 2;
    }
    int cp, cm;
    const bool sp = smooth_term<false>(p, cp), sm = smooth_term<false>(n, cm);
    if (sp && sm) {
      h[m] = from_fixed(smooth_sum(G, cp + cm), k0 + 2) / 6;
      continue;
    }
    const int sh = field_shift(X, G);
    if (sh == 64) continue;
    shift_field(X, sh);
    shift_field(G, sh);
    bool lost = false;
    const i64 S = rough_sum(X, G, [&](const i64(&e)[5]) {
      return recon6<false>(e[0], e[1], e[2], e[3], e[4], Flt(), &lost); });
    h[m] = from_fixed(S, k0 + 6 - sh) / 6;
    if (lost) {
      fields<double, NC>(s, x, f, A, i0, wide);
      h[m] = wide[m];
    }
  }
}
template <class T, int NC>
void back(const Face<T> &f, const T *h, const Cell<T> &L, const Cell<T> &R, T *F) {
  const T h14 = h[0] + h[NC - 1], S = 2 * h[1] + h14, D = h[NC - 1] - h[0], h3 = NC == 4 ? 2 * h[2] : 0;
  const T X[4] = {S, f.un * S + f.c * D, f.ut * S + h3, f.H * h14 + (f.un * f.c * D + (f.q2 * h[1] + f.ut * h3))};
  for (int q = 0; q < NC; ++q) F[q] = X[NC == 3 && q == 2 ? 3 : q] / 4 + (L.F[q] + R.F[q]) / 2;
}
// Largest value and the largest error by the FP64 formulas and by the integer path of each
// component's flux differences.
template <int NC>
struct Errors {
  double top[NC] = {}, fp64[NC] = {}, fixed[NC] = {};
};
template <int NC>
Errors<NC> errors(const Line<NC> &s) {
  double A[NC];
  speeds(s, A);
  std::vector<Cell<double>> x;
  std::vector<Cell<Q>> y;
  for (int i = 0; i < s.n(); ++i) {
    x.push_back(cell<double>(s, i));
    y.push_back(cell<Q>(s, i));
  }
  Errors<NC> e;
  double F[2][NC] = {}, prev[2][NC];
  Q FQ[NC] = {}, prevQ[NC];
  for (int L = 2; L + 3 < s.n(); ++L) {
    std::copy(&F[0][0], &F[0][0] + 2 * NC, &prev[0][0]);
    std::copy(FQ, FQ + NC, prevQ);
    const Face<double> f = roe(x[L], x[L + 1], s.gm1);
    const Face<Q> fq = roe(y[L], y[L + 1], s.gm1);
    double h[NC];
    Q hq[NC];
    fields<double, NC>(s, &x[L - 2], f, A, L - 2, h);
    back<double, NC>(f, h, x[L], x[L + 1], F[0]);
    fields_fixed<NC>(s, &x[L - 2], f, A, L - 2, h);
    back<double, NC>(f, h, x[L], x[L + 1], F[1]);
    fields<Q, NC>(s, &y[L - 2], fq, A, L - 2, hq);
    back<Q, NC>(fq, hq, y[L], y[L + 1], FQ);
    if (L == 2) continue;
    for (int q = 0; q < NC; ++q) {
      const Q d = FQ[q] - prevQ[q];
      e.top[q] = std::max(e.top[q], (double)mag(d));
      e.fp64[q] = std::max(e.fp64[q], (double)mag(d - ((Q)F[0][q] - prev[0][q])));
      e.fixed[q] = std::max(e.fixed[q], (double)mag(d - ((Q)F[1][q] - prev[1][q])));
    }
  }
  return e;
}
