// weno_fixed.cuh -- the sixth-order reconstruction of eqs. (11)-(22) on the
// integer pipes.
//
// What bounds the stage kernels is FP64 issue: an SM of GB300 starts about
// 1.95 FP64 operations per clock, but (measured) 62 integer multiply-adds
// (58 with a 64-bit result) and beside them 62 logic or shift operations, or
// 118 additions.  A 64-bit integer step therefore costs a few percent of an
// FP64 one, and the reconstruction -- 71 % of the FP64 work of a 2D stage when
// it ran there -- needs neither FP64's range inside a stencil nor its
// rounding: it is homogeneous of degree one, its answer is an average of
// candidates within the stencil's variation, and so an error of a few units
// of 2^-57 of the largest difference, in every difference, is below the
// rounding FP64 gives it (2^-53 per operation) as long as the differences that
// the weights choose are not far smaller than the largest.  Beside a strong
// jump they can be; such faces are left to FP64 (uneven_fields).
//
// Measured at 2048^2, FP64, one step: 33.5 ms with the reconstruction and the
// projections on the FP64 pipe, 16.0 ms with the reconstruction here, 9.16 ms
// with the projections (project) and the smooth stencils (smooth_term) too,
// 7.87 ms with the scheme's constants from the host and the speed maxima
// filtered in FP32, 7.95 ms with a scale for each group of fields and with what
// a common unit does not serve left to FP64.  What is left is bound by both: FP64
// pipe 56 %, integer (alu) 38 %, 48 % of the issue slots (1024^2, 11.8k instructions
// and 211 FP64 operations per cell and stage).
//
// Number formats (tests/test_kernel_fixed.py compiles this header for the host
// and measures the error against quadruple precision):
//  * differences and what is linear in them (second differences, candidate
//    fluxes, the fifth difference): 64-bit integers in units of 2^-57 of the
//    power of two above the largest of the ten differences of a field -- exact
//    sums;
//  * indicators and tau: a 64-bit mantissa with its top bit set and an
//    exponent;
//  * weights: their reciprocals 1/b_k and 1/(4 tau), aligned to the largest,
//    since alpha_k of eqs. (20)-(21) is proportional to d_k (1/b_k + 1/(4 tau))
//    for p = 1: a weighted mean needs its weights to a fixed fraction of the
//    largest one only.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define WENO_FX __device__ __forceinline__
#else
#include <cmath>
#define WENO_FX inline
#endif

namespace weno {
namespace fx {

typedef unsigned long long u64;
typedef long long i64;

#ifdef __CUDA_ARCH__
// 64-bit shifts that give 0 for a count of 64 or more
WENO_FX u64 shr(u64 x, int n) {
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}
WENO_FX u64 shl(u64 x, int n) {
  u64 r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}
WENO_FX int clz32(uint32_t x) { return __clz((int)x); }
WENO_FX uint32_t rcp_seed(uint32_t fbits) {  // bits of about 1 / f, f in [1, 2)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fbits)));
  return __float_as_uint(r);
}
// (by halves: a test of the exponent bits of a bit-cast double is turned into
// an FP64 comparison)
WENO_FX u64 dbits(double x) {
  return ((u64)(uint32_t)__double2hiint(x) << 32) | (uint32_t)__double2loint(x);
}
WENO_FX double bitsd(u64 b) { return __longlong_as_double((i64)b); }
#else
WENO_FX u64 shr(u64 x, int n) { return n >= 64 ? 0 : x >> n; }
WENO_FX u64 shl(u64 x, int n) { return n >= 64 ? 0 : x << n; }
WENO_FX int clz32(uint32_t x) { return x ? __builtin_clz(x) : 32; }
WENO_FX uint32_t rcp_seed(uint32_t fbits) {
  float f, r;
  std::memcpy(&f, &fbits, 4);
  r = 1.0f / f;
  std::memcpy(&fbits, &r, 4);
  return fbits;
}
WENO_FX u64 dbits(double x) {
  u64 b;
  std::memcpy(&b, &x, 8);
  return b;
}
WENO_FX double bitsd(u64 b) {
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}
#endif

WENO_FX uint32_t lo32(u64 x) { return (uint32_t)x; }
WENO_FX uint32_t hi32(u64 x) { return (uint32_t)(x >> 32); }
WENO_FX int imax(int a, int b) { return a > b ? a : b; }
WENO_FX u64 abs64(i64 x) { return x < 0 ? 0 - (u64)x : (u64)x; }

// a b / 2^64, low by at most 2 (the product of the low words and the carries
// out of the lower 64 bits are left out): three multiply-adds.
WENO_FX u64 mulhi64(u64 a, u64 b) {
  const u64 c1 = (u64)hi32(a) * lo32(b), c2 = (u64)lo32(a) * hi32(b);
  return (u64)hi32(a) * hi32(b) + hi32(c1) + hi32(c2);
}
// a^2 / 2^64 for a < 2^63.
WENO_FX u64 sqrhi(u64 a) {
  const u64 c = (u64)(hi32(a) * 2u) * lo32(a);
  return (u64)hi32(a) * hi32(a) + hi32(c);
}

// Leading zeros of a 64-bit number (64 for 0) with one FLO.
WENO_FX int clz64(u64 x) {
  const uint32_t h = hi32(x), w = h ? h : lo32(x);
  return clz32(w) + (h ? 0 : 32);
}

// 2^127 / X for X >= 2^63, low by at most 2^-60 of it and never high (so it
// stays below 2^64): the
// special-function unit's FP32 reciprocal of the top 24 bits, taken a little
// low so that e = 1 - x r is positive (0 < e < 2^-20), then r (1 + e + e^2)
// in 64-bit arithmetic.
WENO_FX u64 rcp64(u64 X) {
  const uint32_t rb = rcp_seed((hi32(X) >> 8) | 0x3F000001u);
  const uint32_t r = rb * 256u + (0x80000000u - 0x400u);  // r / 2^32 < 1 / x, x = X / 2^63
  const u64 d = (u64)hi32(X) * r + hi32((u64)lo32(X) * r);  // x r in units of 2^-63
  const u64 e = 0x7FFFFFFFFFFFFFFFull - d;          // a unit low, for what d leaves out
  const uint32_t eh = (uint32_t)(e >> 12);          // e in units of 2^-51 (31 bits)
  const u64 g = e + (hi32((u64)eh * eh) >> 7);      // + e^2: 2^-102+32 = 2^-70 -> 2^-63
  const u64 w = (u64)r * lo32(g);
  return ((u64)r * (0x80000000u + hi32(g)) + hi32(w)) << 1;
}

// Fixed-point value of x: x 2^(57 - (es - 1022)), truncated towards zero, with
// es at least the biased exponent of x and at least 64 (then a zero x, and
// any x below 2^-57 of the unit, gives 0).
WENO_FX i64 to_fixed(double x, int es) {
  const u64 b = dbits(x);
  const u64 m = (b << 11) | 0x8000000000000000ull;
  const int e = (int)((b >> 52) & 0x7FF);
  const u64 v = shr(m, 7 + es - e);
  return (i64)b < 0 ? -(i64)v : (i64)v;
}

// 13 s^2 + 3 t^2 = 3 (4 beta) of |s|, |t| < 2^62, as raw 2^(64 - 2 n).
struct Ind {
  u64 raw;  // 0 or at least 2^59.5
  int n;
};
WENO_FX Ind indicator(i64 s, i64 t) {
  const u64 sa = abs64(s), ta = abs64(t);
  Ind o;
  o.n = clz64(sa | ta) - 2;
  const u64 S = sqrhi(shl(sa, o.n)), T = sqrhi(shl(ta, o.n));
  o.raw = 13ull * S + 3ull * T;
  return o;
}

// A positive number m 2^e with the top bit of m set.
struct Flt {
  u64 m;
  int e;
};
// raw 2^e, raw = 0 or above 2^56; a zero counts as 2^56.
WENO_FX Flt normal(u64 raw, int e) {
  Flt f;
  const uint32_t h = hi32(raw) > 0x01000000u ? hi32(raw) : 0x01000000u;
  const int n = clz32(h);
  f.m = shl(((u64)h << 32) | lo32(raw), n);
  f.e = e - n;
  return f;
}
// raw 2^e + s, aligned to the larger of the two.
WENO_FX Flt normal_plus(u64 raw, int e, const Flt &s) {
  const int d = raw ? s.e - e : 8192;
  const u64 v = shr(raw, d > 0 ? d + 1 : 1) + shr(s.m, d > 0 ? 1 : 1 - d);
  return normal(v, (d > 0 ? s.e : e) + 1);
}

// Six times the correction f - v2 of eqs. (14)-(22) (p = 1) of the stencil
// with differences d_j, |d_j| < 2^58, in their units:
//   c = r_1 + sum_k w_k (r_k - r_1), w_k = D_k z_k / sum D_j z_j,
//   z_k = 1/b_k + 1/T, b_k = 3 (4 beta_k), T = 3 (4 tau), D = (1, 9, 9, 1).
// SENS: whether the sensitivity term e = 3 (4 eps mu^2) of eq. (21) is added
// to the b_k.  At epsilon <= 2^-126 it is below a quarter of the unit squared
// wherever mu_0 is below the largest difference, and it could only decide
// between candidates that agree to a few units; it is then left out, and an
// indicator that is 0 in these units counts as 2^-4.
// Where one is 0 (three equal cells: d0 = d1 = 0, d1 = d2 = 0 or d2 = d3 = 0) the
// others' weights are 2^-4 / T of its own at most, below a unit of the candidates
// from |r5| = 2^29 on.  Below (cubic data to its rounding) the weights hang on
// the sensitivity term and on what the units leave of r5: *lost, for FP64 to take
// over, whose differences of equal cells are 0 and the others' exact.
template <bool SENS>
WENO_FX i64 recon6(i64 d0, i64 d1, i64 d2, i64 d3, i64 d4, const Flt &e, bool *lost = nullptr) {
  const i64 s0 = d1 - d0, s1 = d2 - d1, s2 = d3 - d2, s3 = d4 - d3;
  const Ind i0 = indicator(s0, 2 * d1 + s0);           // t_0 = 3 d1 - d0
  const Ind i1 = indicator(s1, d1 + d2);               // t_1
  const Ind i2 = indicator(s2, 2 * d2 - s2);           // t_2 = 3 d2 - d3
  const Ind id = indicator(s3, s3 + 2 * (s3 - d3));    // t_3 = 3 d4 - 5 d3
  const i64 q = s1 - s2;
  const i64 r5 = (s3 - s0) + 3 * q;                    // fifth difference
  // b_3 = mean of the four (eq. (16)), aligned to the largest
  const int a01 = i0.n < i1.n ? i0.n : i1.n, a2d = i2.n < id.n ? i2.n : id.n;
  const int nm = a01 < a2d ? a01 : a2d;
  const u64 raw3 = shr(i0.raw, 2 * (i0.n - nm) + 2) + shr(i1.raw, 2 * (i1.n - nm) + 2) +
                   shr(i2.raw, 2 * (i2.n - nm) + 2) + shr(id.raw, 2 * (id.n - nm) + 2);
  Flt b0, b1, b2, b3;
  if (SENS) {
    b0 = normal_plus(i0.raw, 64 - 2 * i0.n, e);
    b1 = normal_plus(i1.raw, 64 - 2 * i1.n, e);
    b2 = normal_plus(i2.raw, 64 - 2 * i2.n, e);
    b3 = normal_plus(raw3, 64 - 2 * nm, e);
  } else {
    b0 = normal(i0.raw, 64 - 2 * i0.n);
    b1 = normal(i1.raw, 64 - 2 * i1.n);
    b2 = normal(i2.raw, 64 - 2 * i2.n);
    b3 = normal(raw3, 64 - 2 * nm);
  }
  // T = 12 r5^2
  const u64 ra = abs64(r5);
  const int nt = clz64(ra) - 1;
  if (lost && nt > 33 && nm < 62 && imax(imax(i0.n, i1.n), i2.n) == 62) *lost = true;
  const u64 sq = sqrhi(shl(ra, nt));
  const Flt T = normal(3ull * sq, ra ? 66 - 2 * nt : -16384);  // 0: far below every b_k
  // y_k = D_k z_k with the largest of D_k / b_k and 8 / T in [2^60, 2^61)
  const int e0 = b0.e < b3.e ? b0.e : b3.e, e1 = (b1.e < b2.e ? b1.e : b2.e) - 3;
  const int e01 = e0 < e1 ? e0 : e1, em = (e01 < T.e - 3 ? e01 : T.e - 3) - 3;
  const u64 w8 = shr(rcp64(T.m), T.e - 3 - em), w1 = w8 >> 3, w9 = w8 + w1;  // 8/T, 1/T, 9/T
  const u64 v1 = shr(rcp64(b1.m), b1.e - 3 - em), v2 = shr(rcp64(b2.m), b2.e - 3 - em);
  const u64 z0 = shr(rcp64(b0.m), b0.e - em) + w1, z3 = shr(rcp64(b3.m), b3.e - em) + w1;
  const u64 z1 = v1 + (v1 >> 3) + w9, z2 = v2 + (v2 >> 3) + w9;
  const u64 den = (z0 + z3) + (z1 + z2);  // < 6.75 2^61
  // sum_k D_k z_k (r_k - r_1) / den with the sum formed on r_k - r_1 + 2^62 >= 0
  const int nd = clz32(hi32(den));
  const u64 y0 = shl(z0, nd), y2 = shl(z2, nd), y3 = shl(z3, nd);  // y0 + y2 + y3 < 2^64
  const i64 p0 = 2 * (s0 - s1), p3 = q + 2 * (s3 - s2);
  const u64 B = 0x8000000000000000ull;
  const u64 N = mulhi64(y0, B + 2 * (u64)p0) + mulhi64(y2, B + 2 * (u64)q) +
                mulhi64(y3, B + 2 * (u64)p3);
  const i64 Ns = (i64)(N - ((y0 + y2 + y3) >> 1));
  const u64 c = mulhi64(abs64(Ns), rcp64(shl(den, nd)));
  return (d1 + 2 * d2) + (Ns < 0 ? -(i64)c : (i64)c);
}

// recon6's *lost for either sign of a scalar's differences x +- g, told before the
// reconstructions (a flag after them keeps the FP64 differences in registers all
// the while: 96 instead of 64, 13695 x 5 Burgers cells 60.4 -> 64.6 us a step).
WENO_FX bool lost_pair(const i64 (&x)[5], const i64 (&g)[5]) {
  bool flat = false;
#pragma unroll
  for (int j = 0; j < 4; ++j) flat = flat || (x[j] | g[j] | x[j + 1] | g[j + 1]) == 0;
  if (!flat) return false;
  const i64 a = (x[0] + x[4]) - 4 * (x[1] + x[3]) + 6 * x[2];
  const i64 b = (g[0] + g[4]) - 4 * (g[1] + g[3]) + 6 * g[2];
  i64 p = 0, n = 0;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    p |= x[j] + g[j];
    n |= x[j] - g[j];
  }
  return (p != 0 && abs64(a + b) < (1ull << 29)) || (n != 0 && abs64(a - b) < (1ull << 29));
}

// The largest biased exponent of the ten differences.
WENO_FX int top_exponent(const double (&xw)[5], const double (&dg)[5]) {
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const uint32_t a = hi32(dbits(xw[j])) & 0x7FFFFFFFu, b = hi32(dbits(dg[j])) & 0x7FFFFFFFu;
    m = m > a ? m : a;
    m = m > b ? m : b;
  }
  return (int)(m >> 20);
}

// c 2^(es - 1022 - 57) / 6: a correction of recon6 back in the data's units.
WENO_FX double scale_back(int es) {
  return bitsd(dbits(1.0 / 6.0) + ((u64)(i64)(es - 1079) << 52));
}

// ---------------------------------------------------------------------------
// Projection on the face's left eigenvectors, on the integer pipes.
//
// The kernels stage differences between adjacent cells packed in 64 bits: the
// signed 53-bit mantissa of the double above a 10-bit exponent code (0: the
// value is 0; kWide: not finite, or not 0 and outside 2^-511 .. 2^511, which
// the integer path leaves to FP64), so a face aligns one with a mask and a
// shift.  Per face and component q the exponent E_q is the largest of the
// stencil's five pairs; the eigenvectors' coefficients get the scale that
// brings the largest coefficient times its component below 2^61 both ways, and
// a coefficient times a component is a 64 x 64-bit product of 32-bit limbs, three
// multiply-adds.
// ---------------------------------------------------------------------------
constexpr int kWide = 1023;
WENO_FX u64 pack(double x) {
  const u64 b = dbits(x);
  const int e = (int)((b >> 52) & 0x7FF);
  const u64 m = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const bool in = e >= 512 && e <= 1533, zero = (b << 1) == 0;
  return zero ? 0 : ((((i64)b < 0 ? 0 - m : m) << 10) | (u64)(in ? e - 511 : kWide));
}
WENO_FX int packed_exponent(u64 w) { return (int)(w & 0x3FF); }
// Shift right with the sign; a count of 64 or more (or below 0) leaves the sign.
WENO_FX i64 shr_signed(i64 v, int n) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return v >> ((unsigned)n > 63u ? 63 : n);
#endif
}
WENO_FX i64 packed_value(u64 w, int n) { return shr_signed((i64)(w & ~0x3FFull), n); }

// A number as two limbs, 2^32 h + 2 l (its lowest bit dropped): all products
// of limbs are signed 32 x 32 -> 64 bits.
struct Limb {
  int h, l;
};
WENO_FX Limb limb(i64 v) {
  Limb o;
  o.h = (int)(v >> 32);
  o.l = (int)(lo32((u64)v) >> 1);
  return o;
}
// Sum of products in units of 2^64 (hi) and 2^33 (cr): of four with factors
// below 2^61 (the products of the low limbs, left out, are then a relative
// 2^-58).
struct Acc {
  i64 hi, cr;
};
WENO_FX i64 over63(const Acc &a) { return (a.hi << 1) + (a.cr >> 30); }  // sum / 2^63
WENO_FX void mac(Acc &s, const Limb &a, const Limb &b) {
  s.hi += (i64)a.h * b.h;
  s.cr += (i64)a.h * b.l;
  s.cr += (i64)a.l * b.h;
}

// The integer form of a coefficient: x 2^(1083 + E - um) with E an exponent
// code (|result| < 2^61 for um >= exponent(x) + E).
WENO_FX Limb coefficient(double x, int E, int um) {
  const u64 b = dbits(x);
  const int e = (int)((b >> 52) & 0x7FF);
  const u64 m = e ? (b << 11) | 0x8000000000000000ull : 0;
  const u64 v = shr(m, um - e - E + 3);
  return limb((i64)b < 0 ? -(i64)v : (i64)v);
}
WENO_FX int exponent(double x) { return (int)((hi32(dbits(x)) >> 20) & 0x7FF); }
// A GLF speed A < 2^a as A 2^(63 - a).
WENO_FX Limb speed(double A, int a) {
  const u64 b = dbits(A);
  const int e = (int)(b >> 52);
  return limb((i64)shr(e ? (b << 11) | 0x8000000000000000ull : 0, a + 1023 - e));
}
// A w / 2^a for |w| < 2^62.
WENO_FX i64 times_speed(const Limb &A, i64 w) {
  Acc v = {0, 0};
  mac(v, A, limb(w));
  return over63(v);
}

// Exponent code of a component: the largest of its states' and its fluxes' over 2^a.
WENO_FX int aligned(int eu, int ef, int a) { return imax(eu, ef ? ef - a : 0); }

// The left eigenvectors of a face in the form project4 (NC = 4) and project3
// (NC = 3) apply them: with z = b2 r - t2 m_n - t3 m_t + b1 E and
// tc = t1 r - ic m_n the fields are z + tc, r - z, (m_t - ut r,) z - tc.
// Three scales, each that of the terms its sums are made of, so that no field
// is cut where FP64 would keep it: um of z and tc (r is no term of theirs:
// beside a dense cell its scale would be far above them), ue of the entropy
// field r - z, us of the shear field.  A projected state is x 2^(1592 - u), a
// field below 2^61.6; fluxes are 2^a (z and tc) and 2^a1 (the two fields that
// move with the flow, whose speed may be far below the sound speed) times as
// large.  E: the components' exponents with 2^a, B0 and B2 of components 0 and
// 2 with 2^a1.  emax: the largest exponent among the coefficients (2047: not
// finite).
template <int NC>
struct LeftRows {
  Limb zr, zn, zt, zE, tr, tn, sr;
  int um, ue, us, emax;
};
template <int NC>
WENO_FX LeftRows<NC> left_rows(const int (&E)[NC], int B0, int B2, int a, int a1, double b2,
                               double b1, double t1, double t2, double t3, double ic, double ut,
                               int least = 0) {
  LeftRows<NC> o;
  const int e1 = exponent(b1), e2 = exponent(b2), f1 = exponent(t1), f2 = exponent(t2),
            f3 = exponent(t3), fc = exponent(ic), fu = exponent(ut);
  o.emax = imax(imax(imax(e1, e2), imax(f1, f2)), imax(fc, NC == 4 ? imax(f3, fu) : 0));
  o.um = imax(imax(imax(e2, f1) + E[0], least), imax(imax(f2, fc) + E[1], e1 + E[NC - 1]));
  o.us = 0;
  if (NC == 4) {
    o.um = imax(o.um, f3 + E[2]);
    o.us = imax(fu + B0, 1023 + B2);
    o.zt = coefficient(-t3, E[2], o.um);
    o.sr = coefficient(-ut, B0, o.us);
  }
  o.ue = imax(o.um + a - a1, 1023 + B0);
  o.zr = coefficient(b2, E[0], o.um);
  o.zn = coefficient(-t2, E[1], o.um);
  o.zE = coefficient(b1, E[NC - 1], o.um);
  o.tr = coefficient(t1, E[0], o.um);
  o.tn = coefficient(-ic, E[1], o.um);
  return o;
}
// A difference vector's projections from its packed components v[q], and apart
// (it lives no longer than its own field) s = m_t - ut r; a = a1 = 0 for
// states, the speeds' exponents for physical fluxes.  r is in units of the
// entropy field (entropy).
struct Proj {
  i64 z, tc, r;
};
template <int NC>
WENO_FX Proj project(const LeftRows<NC> &c, const int (&E)[NC], int a, int a1, const u64 (&v)[NC]) {
  Limb d[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) d[q] = limb(packed_value(v[q], E[q] + a + 2 - packed_exponent(v[q])));
  Acc z = {0, 0}, t = {0, 0};
  mac(z, c.zr, d[0]);
  mac(z, c.zn, d[1]);
  if (NC == 4) mac(z, c.zt, d[2]);
  mac(z, c.zE, d[NC - 1]);
  mac(t, c.tr, d[0]);
  mac(t, c.tn, d[1]);
  return Proj{over63(z), over63(t), packed_value(v[0], c.ue + a1 - 1018 - packed_exponent(v[0]))};
}
template <int NC>
WENO_FX i64 entropy(const LeftRows<NC> &c, int a, int a1, const Proj &p) {
  return p.r - shr_signed(p.z, c.ue + a1 - c.um - a);
}
WENO_FX i64 project_shear(const LeftRows<4> &c, int B0, int a1, u64 rho, u64 mt) {
  Acc u = {0, 0};
  mac(u, c.sr, limb(packed_value(rho, B0 + a1 + 2 - packed_exponent(rho))));
  return over63(u) + packed_value(mt, c.us + a1 - 1018 - packed_exponent(mt));
}
#ifndef __CUDACC__
// One speed exponent and one scale for all fields (host tests).
template <int NC>
WENO_FX LeftRows<NC> left_rows(const int (&E)[NC], double b2, double b1, double t1, double t2,
                               double t3, double ic, double ut) {
  return left_rows<NC>(E, E[0], E[2], 0, 0, b2, b1, t1, t2, t3, ic, ut, 1023 + E[0]);
}
template <int NC>
WENO_FX Proj project(const LeftRows<NC> &c, const int (&E)[NC], int a, const u64 (&v)[NC]) {
  return project<NC>(c, E, a, a, v);
}
WENO_FX i64 project_shear(const LeftRows<4> &c, const int (&E)[4], int a, u64 rho, u64 mt) {
  return project_shear(c, E[0], a, rho, mt);
}
#endif

// Where one unit a field is not enough.  The unit is 2^-57 of the stencil's
// largest difference; the weights may choose a candidate whose differences are
// far smaller, and FP64 holds those to 2^-53 of their own.  That shows only
// where the unit is also above the rounding of the face's flux: h is off by a
// few units in any case, and 2^-53 rho c of it by the rounding of the pressure.
// So a field is left to FP64 where its scale is more than 2^kStrong rho c (the
// shear field's, a momentum's: rho c times the larger of c and ut) and two adjacent
// differences (three of the four candidates are made of two) are both more than
// 2^kUneven below it, in the terms that they are sums of.  With 8 and 4 no
// state tried (jumps of pressure and density up to 1e18, random cells up to
// 1e12 apart) is further off than 2.4 times the FP64 formulas, as with 4 and 4;
// of 3000 random pairs of states one in a hundred is off by 6 times (4: 2, 10:
// 15).  Tubes and quadrants with pressures of 0.1 to 2 stay here (with 4 a few
// faces did not, and as such a face takes its warp 20 us longer, a step of 64 x
// 1600 cells took 210 us, 149 without them).
constexpr int kStrong = 8, kUneven = 4;
// Fields that may need FP64 as far as their scales tell, as a mask; floor: the
// exponent of rho c, not biased.
template <int NC>
WENO_FX unsigned strong_fields(const LeftRows<NC> &c, int a, int a1, double ic, double ut, int floor) {
  const int least = floor + kStrong + 1535;
  unsigned m = c.um + a > least ? 1u | (1u << (NC - 1)) : 0u;
  m |= c.ue + a1 > least ? 2u : 0u;
  if (NC == 4) m |= c.us + a1 > least + imax(exponent(ut), 2046 - exponent(ic)) - 1023 ? 4u : 0u;
  return m;
}
// Those of them with two adjacent small differences.
template <int NC, class Diff>
WENO_FX unsigned uneven_fields(Diff diff, int a, int a1, int um, int ue, int us, double b2,
                               double b1, double t1, double t2, double t3, double ic, double ut) {
  const int none = -65536, fu = exponent(ut);
  const int c[4] = {imax(exponent(b2), exponent(t1)), imax(exponent(t2), exponent(ic)),
                    NC == 4 ? exponent(t3) : exponent(b1), exponent(b1)};
  int lz = none, le = none, ls = none;  // the pair before
  unsigned m = 0;
#pragma unroll 1
  for (int j = 0; j < 5; ++j) {
    int zu = none, zf = none, r0 = none, r2 = none;
#pragma unroll
    for (int q = 0; q < NC; ++q) {
      const int u = packed_exponent(diff(0, q, j)), f = packed_exponent(diff(1, q, j));
      const int xu = u ? u : none, xf = f ? f : none;
      zu = imax(zu, xu + c[q]);
      zf = imax(zf, xf + c[q]);
      if (q == 0) r0 = imax(xu, xf - a1);
      if (NC == 4 && q == 2) r2 = imax(xu, xf - a1);
    }
    const int z = imax(zu, zf - a), e = imax(imax(zu, zf - a1), 1023 + r0), s = imax(fu + r0, 1023 + r2);
    if (j > 0) {
      if (imax(z, lz) < um - kUneven) m |= 1u | (1u << (NC - 1));
      if (imax(e, le) < ue - kUneven) m |= 2u;
      if (NC == 4 && imax(s, ls) < us - kUneven) m |= 4u;
    }
    lz = z;
    le = e;
    ls = s;
  }
  return m;
}
// The same for a scalar's ten differences with the largest exponent es, 2^kUneven
// above the centre values (a scalar has no pressure whose rounding would cover
// more).
WENO_FX bool uneven(const double (&xw)[5], const double (&dg)[5], int es, double centre) {
  if (es <= exponent(centre) + kUneven) return false;
  bool m = false;
  int last = 0;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const int e = imax(exponent(xw[j]), exponent(dg[j]));
    m = m || (j > 0 && imax(e, last) < es - kUneven);
    last = e;
  }
  return m;
}

// The stencil differences g + x of f^+ become those of the mirrored f^-:
// x - g in reverse order.
WENO_FX void mirror(i64 (&x)[5], i64 (&g)[5]) {
  const i64 x0 = x[0], x1 = x[1], g0 = g[0], g1 = g[1];
  x[0] = x[4];
  x[4] = x0;
  x[1] = x[3];
  x[3] = x1;
  g[0] = -g[4];
  g[4] = -g0;
  g[1] = -g[3];
  g[3] = -g1;
  g[2] = -g[2];
}

// Shift of a field's differences that brings the largest |g +- x| to
// [2^57, 2^58): left by n - 6 (n = 64: they are all 0).
WENO_FX int field_shift(const i64 (&x)[5], const i64 (&g)[5]) {
  uint32_t mh = 0, ml = 0;
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const i64 p = x[j] + g[j], n = x[j] - g[j], sp = p >> 63, sn = n >> 63;
    mh |= hi32((u64)(p ^ sp)) | hi32((u64)(n ^ sn));
    ml |= lo32((u64)(p ^ sp)) | lo32((u64)(n ^ sn));
  }
  return clz64(((u64)mh << 32) | ml);
}
WENO_FX void shift_field(i64 (&x)[5], int n) {
#pragma unroll
  for (int j = 0; j < 5; ++j) x[j] = (i64)shl((u64)x[j], n - 1) >> 5;
}

// FP32 operations that no compiler contracts: every kernel takes the same
// decision, and the same term, for the same stencil.
#ifdef __CUDA_ARCH__
WENO_FX float fmul(float a, float b) { return __fmul_rn(a, b); }
WENO_FX float fadd(float a, float b) { return __fadd_rn(a, b); }
WENO_FX float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
WENO_FX float fmul(float a, float b) { return a * b; }
WENO_FX float fadd(float a, float b) { return a + b; }
WENO_FX float ffma(float a, float b, float c) { return std::fma(a, b, c); }
#endif
// A 64-bit integer over 2^32 in FP32.
WENO_FX float to_float(i64 x) {
  return ffma((float)lo32((u64)x), 0x1p-32f, (float)(int)hi32((u64)x));
}
WENO_FX float rcpf(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

// Smooth stencils.  With the linear candidate average rm = sum D_k r_k / 20,
//   c = rm + sum_k D_k G_k (r_k - rm) / (20 + sum_k D_k G_k), G_k = T / b_k,
// the second term is far below a unit, or a few units, wherever the stencil
// resolves its data (G is the eighth power of the phase per cell, r_k - rm its
// third).  Computed in FP32 on the exact second differences, their exact
// differences and the exact fifth one, so that nothing cancels but in forming
// r_k - rm, whose largest is at least half the largest of its terms: the error
// is below 2^-21 of max G max |r_k - rm|, which is 2 units (2^-58 of the bound
// on the projected differences) where that product is at most 2^22 units, from
// about 70 cells a wavelength on.
// |d_j| < 2^61: a field's differences over 4.  Returns whether it is, and the
// term in units.  (About 80 FP32 operations a flux, where the weights take
// several hundred integer ones.)
// SENS: a sensitivity term would lower G, so the term then has to vanish (at
// most half a unit); without it (epsilon <= 2^-126) the same holds unless
// every b_k is above 2^18 units squared, 2^25 times what it could be.
template <bool SENS>
WENO_FX bool smooth_term(const i64 (&d)[5], int &corr) {
  const i64 s0 = d[1] - d[0], s1 = d[2] - d[1], s2 = d[3] - d[2], s3 = d[4] - d[3];
  const float a0 = to_float(s0), a1 = to_float(s1), a2 = to_float(s2), a3 = to_float(s3);
  const float f1 = to_float(d[1]), f2 = to_float(d[2]), f3 = to_float(d[3]);
  const i64 q = s1 - s2, l = s3 - s0;
  const float e2 = to_float(q), f5 = ffma(3.0f, e2, to_float(l));
  // l + 3 q is the fifth difference.  It can cancel to far below both, so where
  // it fits 64 bits it is formed in them: FP32's 2^-24 of q would be noise in
  // T, 1e6 units in the term of a cubic.
  const float r5 = fabsf(f5) < 0x1p30f ? to_float((i64)((u64)l + 3 * (u64)q)) : f5;
  const float t0 = ffma(2.0f, f1, a0), t1 = fadd(f1, f2), t2 = ffma(2.0f, f2, -a2),
              t3 = ffma(3.0f, a3, fmul(-2.0f, f3));
  const float b0 = ffma(fmul(13.0f, a0), a0, fmul(fmul(3.0f, t0), t0));
  const float b1 = ffma(fmul(13.0f, a1), a1, fmul(fmul(3.0f, t1), t1));
  const float b2 = ffma(fmul(13.0f, a2), a2, fmul(fmul(3.0f, t2), t2));
  const float bd = ffma(fmul(13.0f, a3), a3, fmul(fmul(3.0f, t3), t3));
  const float b3 = fmul(0.25f, fadd(fadd(b0, b1), fadd(b2, bd)));
  // (2^-126 / 2^-120: an indicator of 0 beside r5 = 0 gives G = 9 / 64, so that
  // recon6 decides there unless the candidates agree to 2^6 units)
  const float T = ffma(fmul(12.0f, r5), r5, 0x1p-126f), T9 = fmul(9.0f, T), tiny = 0x1p-120f;
  const float g0 = fmul(T, rcpf(fadd(b0, tiny))), g1 = fmul(T9, rcpf(fadd(b1, tiny)));
  const float g2 = fmul(T9, rcpf(fadd(b2, tiny))), g3 = fmul(T, rcpf(fadd(b3, tiny)));
  // r_k - r_1, their mean m, and r_k - rm
  const float e0 = fmul(2.0f, to_float(s0 - s1));
  const float e3 = ffma(2.0f, to_float(s3 - s2), e2);
  const float m = fmul(0.05f, ffma(9.0f, e2, fadd(e0, e3)));
  const float h0 = fadd(e0, -m), h2 = fadd(e2, -m), h3 = fadd(e3, -m);
  const float gs = fadd(fadd(g0, g1), fadd(g2, g3));  // 20 times a mean of the G_k
  const float hm = fmaxf(fmaxf(fabsf(h0), fabsf(h2)), fmaxf(fabsf(h3), fabsf(m)));
  const float most = fmul(gs, hm);
  if (SENS) {
    corr = 0;
    return most <= 8 * 0x1p-32f;
  }
  const float c = fmul(ffma(g0, h0, ffma(g2, h2, ffma(g3, h3, -fmul(g1, m)))),
                       rcpf(fadd(20.0f, gs)));
  const bool ok = most <= 16 * 0x1p-10f &&
                  (most <= 8 * 0x1p-32f || fminf(fminf(b0, b1), fminf(b2, b3)) >= 0x1p-46f);
  corr = ok ? (int)ffma(c, 0x1p32f, c < 0.0f ? -0.5f : 0.5f) : 0;
  return ok;
}

// c^+ + c^- less 6 alpha dw_2 of a smooth field: the linear parts add up to
// (7 (g_1 - g_3) - (g_0 - g_4)) / 5 (alpha drops out of the central flux).
// In units of 4, as the terms.
WENO_FX i64 smooth_sum(const i64 (&g)[5], int corr) {
  const i64 v = (g[1] >> 2) - (g[3] >> 2);
  const i64 u = 2 * v - ((g[0] >> 2) - (g[4] >> 2));  // v + u / 5
  Acc p = {0, 0};  // u times 2^63 / 5
  mac(p, Limb{0x19999999, 0x4CCCCCCD}, limb(u));
  return v + over63(p) + corr;
}

// c^+ + c^- less 6 alpha dw_2 by the weights, one flux after the other.
template <class Recon>
WENO_FX i64 rough_sum(i64 (&x)[5], i64 (&g)[5], Recon recon) {
  i64 S = 0;
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    i64 d[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) d[j] = x[j] + g[j];
    S += recon(d) - 3 * d[2];
    mirror(x, g);
  }
  return S;
}

// S 2^k, rounded to nearest, by shifts (a conversion from a 64-bit integer
// issues to the FP64 pipe).
WENO_FX double from_fixed(i64 S, int k) {
  const u64 a = abs64(S);
  const int n = clz64(a);
  const u64 v = shl(a, n), r = (v >> 11) + ((v >> 10) & 1);  // the leading bit adds to the exponent
  const u64 b = r + ((u64)(i64)(1085 + k - n) << 52);
  return bitsd(S == 0 ? 0 : (S < 0 ? b | 0x8000000000000000ull : b));
}

}  // namespace fx
}  // namespace weno
