// kf_fp64.cuh -- the Kalman step in double precision (KF_FP64 and the redo
// passes of KF_ADAPTIVE), written for GB300's FP64 pipe.
//
// What bounds it: an SM executes two FP64 lanes per clock, so one FP64 warp
// instruction holds its scheduler's pipe for 64 to 76 cycles (a probe of
// dependent and independent chains: additions, products, fused
// multiply-adds, comparisons and conversions from and to float alike, with
// one lane active or with 32), while an integer or FP32 instruction takes
// two or less.  Only the number of FP64 instructions matters, so this file
// spends integer and FP32 instructions to save them:
//  * conversions to and from float by integer shifts (8-12 cycles);
//  * comparisons on the bit patterns;
//  * 1/x, 1/sqrt(x) and sqrt(x) from an FP32 seed and one third-order step
//    (3 to 5 FP64 instructions; the library's take 6 to 9);
//  * sin and cos from a 256-entry table (13 FP64 instructions, the library's
//    27), the turning angle from the same table (9 instead of 45);
//  * the transport C' = J C J^T through J's factored form J = J_s + u (ds/dp)
//    (89 multiply-adds for a cylinder, 70 for a plane), and the update
//    without the columns and products the general form spends on them.
// Sums, products and fused multiply-adds are correctly rounded double operations
// and none is done in less: the seeds only choose where the double iteration
// starts.  1/x and sqrt(x) come out correctly rounded but for a few near-ties,
// 1/sqrt(x) within 1 ulp; sin and cos carry the table's and two sums' roundings;
// a quotient is a product with the reciprocal, within 1 ulp (correctly rounded
// quotients for the arc and S(h) change a whole step's rms error against
// quadruple precision by less than 1 %).
//
// Every rounding is written out (as in kf_num.cuh), so all kernels that call
// these functions agree bit for bit.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kf_num.cuh"

namespace kf {
namespace f64 {

__device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// ------------------------------------------------------- bits, conversions

// A float that is neither zero, denormal, infinite nor NaN, as a double.
__device__ __forceinline__ double from_normal(float f) {
  const int i = __float_as_int(f);
  return __hiloint2double(((i >> 3) & (int)0x8fffffff) + 0x38000000, i << 29);
}

// (double)f by shifts, exact for every float: below the normal range f is
// scaled up by 2^32 first, by a product that keeps denormals whether or not the
// unit is built with -ftz=true; infinities and NaN stay what they are.
__device__ __forceinline__ double from_float(float f) {
  const int e = __float_as_int(f) & 0x7f800000;
  float up;
  asm("mul.rn.f32 %0, %1, 0f4F800000;" : "=f"(up) : "f"(f));
  const int i = __float_as_int(e == 0 ? up : f);
  const int bias = e == 0 ? 0x36000000 : e == 0x7f800000 ? 0x70000000 : 0x38000000;
  const int hi = ((i >> 3) & (int)0x8fffffff) + bias;
  return __hiloint2double((i << 1) == 0 ? i : hi, i << 29);
}

// The high word of |x|: the exponent and 20 bits of the mantissa.
__device__ __forceinline__ unsigned top(double x) {
  return (unsigned)__double2hiint(x) & 0x7fffffffu;
}

// x cut to float, for a normal float's range of |x|.
__device__ __forceinline__ float cut_normal(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const unsigned m = __funnelshift_l((unsigned)__double2loint(x), hi - 0x38000000u, 3);
  return __uint_as_float((m & 0x7fffffffu) | (hi & 0x80000000u));
}
// The same with values below that range cut to zero (keeping the sign).
__device__ __forceinline__ float cut(double x) {
  return top(x) < 0x38100000u ? __int_as_float(__double2hiint(x) & (int)0x80000000)
                              : cut_normal(x);
}

// (float)x, rounded to nearest even: the bits cut off plus just under half a
// unit (half, if the last bit kept is odd) carry into it.  Zero, and
// what is not a normal float, take the instruction, which keeps denormal
// results in every unit.
__device__ __forceinline__ float to_float(double x) {
  if (top(x) - 0x38100000u >= 0x0fe00000u) {
    float f;
    asm("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(x));
    return f;
  }
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = __funnelshift_l(lo, hi - 0x38000000u, 3) & 0x7fffffffu;
  const unsigned rest = lo << 3;
  const unsigned up = rest > 0x80000000u - (m & 1u) ? 1u : 0u;
  return __uint_as_float((m + up) | (hi & 0x80000000u));
}

__device__ __forceinline__ unsigned long long bits(double x) {
  return (unsigned long long)__double_as_longlong(x);
}
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;
// x > 0 and x >= 0; false for NaN
__device__ __forceinline__ bool gt0(double x) { return bits(x) - 1ull < kInfBits; }
__device__ __forceinline__ bool ge0(double x) {
  return bits(x) <= kInfBits || bits(x) == 0x8000000000000000ull;
}
// |x| > c for a positive constant c given by its bits; false for NaN
__device__ __forceinline__ bool abs_gt(double x, unsigned long long c) {
  const unsigned long long a = bits(x) & 0x7fffffffffffffffull;
  return a > c && a <= kInfBits;
}

// --------------------------------------------------- 1/x, 1/sqrt(x), sqrt(x)
// Outside the range where the FP32 seed is a normal number (zero, infinity,
// NaN, extreme scales) the library's operation.
static __device__ __noinline__ double rcp_any(double x) { return __ddiv_rn(1.0, x); }
static __device__ __noinline__ double rsqrt_any(double x) { return ::rsqrt(x); }
static __device__ __noinline__ double sqrt_any(double x) { return __dsqrt_rn(x); }

// |x| within 2^-100 .. 2^100
__device__ __forceinline__ bool seedable(double x) { return top(x) - 0x39b00000u < 0x0c800000u; }

// e = 1 - x r is below 2^-21, and r (1 + e + e^2) leaves e^3.
__device__ __forceinline__ double rcp(double x) {
  if (!seedable(x)) return rcp_any(x);
  float s;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(cut_normal(x)));
  const double r = from_normal(s);
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1/sqrt(x) = y (1 - e)^(-1/2) with e = 1 - x y^2: y + y e (1/2 + 3/8 e),
// the next term 5/16 e^3.
__device__ __forceinline__ double rsqrt(double x) {
  if (__double2hiint(x) < 0 || !seedable(x)) return rsqrt_any(x);
  float s;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(cut_normal(x)));
  const double y = from_normal(s);
  const double e = fma(-mul(x, y), y, 1.0);
  return fma(mul(y, e), fma(e, 0.375, 0.5), y);
}

// sqrt(x) = g (1 - e)^(-1/2) with g = x y and e as above.  t = y (x - g^2) is
// g e and undoes g's own rounding, so the result is the correctly rounded root
// but for arguments within 2^-20 ulp of a tie (e from g y leaves half of that
// rounding: 0.75 ulp).  A float's digits are enough for the e beside 1/2.
// |x| within 2^-60 .. 2^60, where x - g^2 is a normal float.
__device__ __forceinline__ double sqrt(double x) {
  if ((unsigned)__double2hiint(x) - 0x3c300000u >= 0x07800000u) return sqrt_any(x);
  float s;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(cut_normal(x)));
  const double y = from_normal(s), g = mul(x, y);
  const double d = fma(-g, g, x);
  const double e = from_normal(__fmul_rn(__fmul_rn(cut(d), s), s));  // 2^-127 for 0
  return fma(mul(y, d), fma(e, 0.375, 0.5), g);
}

// ------------------------------------------------------------- sin and cos
// sin and cos of k pi/128, k = 0..255, evaluated at compile time by Taylor
// series in double-double arithmetic (Knuth's two-sum, Dekker's product) and
// rounded to double.  Read as double2 (table_entry), so the table is aligned
// like one: doubles alone would ask for 8 bytes, and a 16-byte load faults on
// an address that is no multiple of 16.
struct alignas(alignof(double2)) SinCosTable {
  double v[256][2];
};

namespace table {
struct dd {
  double hi, lo;
};
constexpr dd two_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return {s, (a - (s - bb)) + (b - bb)};
}
constexpr dd quick(double a, double b) {
  const double s = a + b;
  return {s, b - (s - a)};
}
constexpr dd two_prod(double a, double b) {
  const double p = a * b, c = 134217729.0;  // 2^27 + 1
  const double a1 = c * a - (c * a - a), a2 = a - a1, b1 = c * b - (c * b - b), b2 = b - b1;
  return {p, ((a1 * b1 - p) + a1 * b2 + a2 * b1) + a2 * b2};
}
constexpr dd mul(dd x, dd y) {
  const dd p = two_prod(x.hi, y.hi);
  return quick(p.hi, p.lo + (x.hi * y.lo + x.lo * y.hi));
}
constexpr dd add(dd x, dd y) {
  const dd s = two_sum(x.hi, y.hi);
  return quick(s.hi, s.lo + (x.lo + y.lo));
}
constexpr dd div(dd x, double d) {
  const double q = x.hi / d;
  const dd p = two_prod(q, d);
  return quick(q, (((x.hi - p.hi) - p.lo) + x.lo) / d);
}
// sin (first = 1) or cos (first = 0) of j pi/128 for j <= 32: the series
// summed from its last term, t <- 1 - x^2 / (m (m - 1)) t.
constexpr double series(int j, int first) {
  const dd pi{3.141592653589793, 1.2246467991473532e-16};
  const dd x = div(mul(pi, dd{(double)j, 0.0}), 128.0);
  const dd x2 = mul(x, x);
  dd t{1.0, 0.0};
  for (int m = first + 24; m > first; m -= 2) {
    const dd u = mul(div(x2, (double)(m * (m - 1))), t);
    t = add(dd{1.0, 0.0}, dd{-u.hi, -u.lo});
  }
  return first ? mul(x, t).hi : t.hi;
}
constexpr SinCosTable make() {
  SinCosTable t{};
  for (int j = 0; j < 64; ++j) {
    const double s = j <= 32 ? series(j, 1) : series(64 - j, 0);
    const double c = j <= 32 ? series(j, 0) : series(64 - j, 1);
    t.v[j][0] = s, t.v[j][1] = c;
    t.v[j + 64][0] = c, t.v[j + 64][1] = -s;
    t.v[j + 128][0] = -s, t.v[j + 128][1] = -c;
    t.v[j + 192][0] = -c, t.v[j + 192][1] = s;
  }
  return t;
}
}  // namespace table

__device__ constexpr SinCosTable kSinCos = table::make();

constexpr double kStepHi = 0.02454369260617026, kStepLo = 9.567553118338697e-19;  // pi/128

struct sc {
  double s, c;
};

__device__ __forceinline__ sc table_entry(int k) {
  const double2 t = __ldg(reinterpret_cast<const double2 *>(&kSinCos.v[k & 255][0]));
  return {t.x, t.y};
}

static __device__ __noinline__ sc sincos_any(double x) {
  sc r;
  ::sincos(x, &r.s, &r.c);
  return r;
}

// x = k pi/128 + r with |r| <= pi/256, then
//   sin x = S + (C sin r + S (cos r - 1)),  cos x = C + (C (cos r - 1) - S sin r).
// sin r / r = 1 + c3 r^2 + c5 r^4 with minimax c3, c5 on the range (relative
// error 3e-17, found by the Remez exchange), cos r - 1 by its Taylor series to
// r^6 (1.3e-20).  pi/128 enters as a double and its remainder, so r keeps its
// relative precision near the multiples.
// From |x| = 64 on (and for NaN) the library's.
__device__ __forceinline__ sc sincos(double x) {
  if (top(x) >= 0x40500000u) return sincos_any(x);
  const float kf = rintf(cut(x) * 40.743665431525206f);  // 128 / pi
  const double k = from_float(kf);
  const double r = fma(k, -kStepLo, fma(k, -kStepHi, x));
  const sc t = table_entry((int)kf);
  const double z = mul(r, r);
  const double sr = fma(mul(r, z), fma(z, 0x1.1110b41d9fc27p-7, -0x1.5555555542e06p-3), r);
  const double cr = mul(z, fma(z, fma(z, -1.0 / 720.0, 1.0 / 24.0), -0.5));
  return {fma(t.s, cr, fma(t.c, sr, t.s)), fma(t.c, cr, fma(-t.s, sr, t.c))};
}

static __device__ __noinline__ double atan2_any(double y, double x) { return ::atan2(y, x); }

// atan2(y, x) when its sine and cosine are known (y and x over their norm):
// atan2f names the nearest table angle k pi/128, s = sin(h - k pi/128) comes
// from the table's entries, and its arcsine from the series to s^7 (|s| <=
// 0.0123: the next term is 2e-17 of it).  9 FP64 instructions; the library's
// atan2 takes 45, a correction of atan2f through sincos 16.
__device__ __forceinline__ double angle(double y, double x, double sh, double ch) {
  // the larger operand within 2^-100 .. 2^100 (a float cuts the other to zero
  // only where the angle to an axis is below 2^-26), no NaN; else the library's
  const unsigned m = top(y) > top(x) ? top(y) : top(x);
  if (m - 0x39b00000u >= 0x0c800000u) return atan2_any(y, x);
  const float kf = rintf(atan2f(cut(y), cut(x)) * 40.743665431525206f);
  const double k = from_float(kf);
  const sc t = table_entry((int)kf);
  const double s = fma(sh, t.c, -mul(ch, t.s)), z = mul(s, s);
  const double d = fma(mul(s, z), fma(z, fma(z, 15.0 / 336.0, 3.0 / 40.0), 1.0 / 6.0), s);
  return fma(k, kStepHi, fma(k, kStepLo, d));
}

// S(h) = sin(h)/h and dS/dh from sin(h) and cos(h); below |h| = 0.05, where
// cos(h) - S(h) cancels, the Taylor series (the first terms left out are
// below 1e-18 and 3e-17 of the sums), else with 1/h.
struct Sinc {
  double S, dS;
};
__device__ __forceinline__ bool sinc_by_series(double h) { return top(h) < 0x3fa99999u; }
__device__ __forceinline__ Sinc sinc_series(double h) {
  const double z = mul(h, h);
  return {fma(z, fma(z, fma(z, fma(z, 1.0 / 362880.0, -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0),
              1.0),
          mul(h, fma(z, fma(z, fma(z, 1.0 / 45360.0, -1.0 / 840.0), 1.0 / 30.0), -1.0 / 3.0))};
}
__device__ __forceinline__ Sinc sinc_quotient(double ih, double sh, double ch) {
  const double S = mul(sh, ih);
  return {S, mul(sub(ch, S), ih)};
}
__device__ __forceinline__ Sinc sinc(double h, double sh, double ch) {
  return sinc_by_series(h) ? sinc_series(h) : sinc_quotient(rcp(h), sh, ch);
}

// Azimuth wrapped to (-pi, pi] (as wrap_phi, kf_device.cuh).  The number of
// turns comes from the float angle and can be one off within a float's
// rounding of +-pi, which is put right there.
__device__ __forceinline__ double wrap_phi(double a) {
  const double n = top(a) < 0x41600000u ? from_float(rintf(cut(a) * 0.15915494309189535f))
                                        : rint(mul(a, 0.15915494309189535));  // from 2^23 on
  const double w = fma(n, -2.4492935982947064e-16, fma(n, -6.283185307179586, a));
  if (top(w) < 0x400921fbu) return w;  // below pi in the high word
  if (w <= -3.141592653589793) return add(add(w, 6.283185307179586), 2.4492935982947064e-16);
  if (w > 3.141592653589793) return sub(sub(w, 6.283185307179586), 2.4492935982947064e-16);
  return w;
}

// ------------------------------------------------------------------- pieces
// Each piece of a step is a function of its own, so that the step of one
// thread (below) and the step that four warps share (kf_fp64_group.cuh)
// round alike.

// d omega / d k
__device__ __forceinline__ double curvature_rate(double q, double bz) {
  return mul(mul(q, -0.299792458e-2), bz);
}

// cos and sin of the chord's direction phi + h.
__device__ __forceinline__ sc turned(const sc &ph, const sc &h) {
  return {fma(ph.c, h.s, mul(ph.s, h.c)), fma(ph.c, h.c, -mul(ph.s, h.s))};
}

// The update's gain (two measured components, h0 the first one's weight):
// K0 = t a00 + u Si01, K1 = t a01 + u Si11 for a component with C' entries t
// and u in the measured columns.  bad: S is not positive definite.
struct Gain {
  double a00, a01, Si01, Si11;
  bool bad;
};
template <bool UNIT0>
__device__ __forceinline__ Gain gain(double T0, double T1, double U1, double h0, double V00,
                                     double V01, double V11) {
  const double S00 = UNIT0 ? add(T0, V00) : fma(mul(h0, h0), T0, V00);
  const double S01 = UNIT0 ? add(T1, V01) : fma(h0, T1, V01);
  const double S11 = add(U1, V11);
  const double det = fma(S00, S11, -mul(S01, S01));
  Gain g;
  g.bad = !(gt0(S00) && gt0(det));
  const double inv = rcp(det);
  const double Si00 = mul(S11, inv);
  g.Si01 = -mul(S01, inv);
  g.Si11 = mul(S00, inv);
  g.a00 = UNIT0 ? Si00 : mul(h0, Si00);
  g.a01 = UNIT0 ? g.Si01 : mul(h0, g.Si01);
  return g;
}
struct Pair {
  double a, b;
};
__device__ __forceinline__ Pair gain_of(const Gain &g, double t, double u) {
  return {fma(t, g.a00, mul(u, g.Si01)), fma(t, g.a01, mul(u, g.Si11))};
}
// k.a x + k.b y + c, and without c: the state's update, and a measured
// column, K V.
__device__ __forceinline__ double dot_add(const Pair &k, double x, double y, double c) {
  return fma(k.a, x, fma(k.b, y, c));
}
__device__ __forceinline__ double dot(const Pair &k, double x, double y) {
  return fma(k.a, x, mul(k.b, y));
}
// C'_im - K_i (H C')_m with k = (h0 K0, K1) of row i, t and u of row m.
__device__ __forceinline__ double reduced(const Pair &k, double t, double u, double c) {
  return fma(-k.a, t, fma(-k.b, u, c));
}

// --------------------------------------------------------------- p2z pieces
// The path to the plane: s, the half turning angle h, ds/dz, ds/dtheta.
// Not ok: parallel to the plane.
struct PlanePath {
  double s, h, dsz, dst;
  bool ok;
};
__device__ __forceinline__ PlanePath plane_path(const sc &th, double dz, double w) {
  PlanePath r;
  r.ok = abs_gt(th.c, 0x3f1a36e2eb1c432dull);  // 1e-4
  const double ict = rcp(th.c), tanth = mul(th.s, ict);
  r.s = mul(dz, tanth);
  r.h = mul(mul(0.5, w), r.s);
  r.dsz = -tanth;
  r.dst = mul(mul(dz, ict), ict);
  return r;
}

// Chord L and the factors of the partials along k at fixed path: with the
// chord's direction (c, s), d(x, y)/dk = a (c, s) + b (-s, c); kap = d phi/dk,
// hs2 = s kap / 2.
struct Bend {
  double L, a, b;
};
__device__ __forceinline__ double half_s_kap(double s, double kap) {
  return mul(mul(0.5, s), kap);
}
__device__ __forceinline__ Bend bend(double s, double hs2, const Sinc &c) {
  return {mul(s, c.S), mul(hs2, c.dS), mul(hs2, c.S)};
}

// A row e_i + a e_k + b e_phi of J_s times a column (c_i, c_k, c_phi) of C.
__device__ __forceinline__ double row(double a, double b, double ci, double ck, double cf) {
  return fma(b, cf, fma(a, ck, ci));
}

// --------------------------------------------------------------- p2r pieces
// The crossing (cos h, sin h, chord) = (den, yh, d) / hypot(den, yh), as in
// propagate_to_r (kf_device.cuh) with half the curvature wh = omega/2 and
// yh = wh d.  Not ok: starts outside, or never reaches the cylinder (the rest
// is then a crossing on the spot, which four warps carry through the step to
// no effect and without a division by zero).
struct Cross {
  double d, den, yh, ch, sh, L;
  bool ok;
};
__device__ __forceinline__ Cross cross(double x, double y, const sc &ph, double w, double wh,
                                       double R) {
  Cross r{};
  r.d = fma(R, R, -fma(x, x, mul(y, y)));
  const double A = fma(x, ph.c, mul(y, ph.s)), B = fma(y, ph.c, -mul(x, ph.s));
  r.yh = mul(wh, r.d);
  const double D = fma(A, A, mul(fma(w, B, fma(-wh, r.yh, 1.0)), r.d));
  r.ok = gt0(r.d) && ge0(D);
  if (!r.ok) {
    r.den = r.ch = 1.0;
    return r;
  }
  r.den = add(A, sqrt(D));
  const double inv = rsqrt(fma(r.den, r.den, mul(r.yh, r.yh)));
  r.ch = mul(r.den, inv);
  r.sh = mul(r.yh, inv);
  r.L = mul(r.d, inv);
  return r;
}

// The path for the half turning angle h: 2 h / omega (iwh = 2 / omega), or the
// straight line's.
__device__ __forceinline__ double arc(const Cross &c, double h, double w, double iwh) {
  return top(w) > 0x3d719799u ? mul(h, iwh) : mul(c.d, rcp(c.den));  // 1e-12
}

// Surface frame at the crossing, n = (ca, sa), t = (-sa, ca), with the chord's
// direction (nm, tm) in it; the gradient of the path is ds = -ic m with
// m = n.J_s = (ca, sa, ., mk, mf, .).
struct Frame {
  double x, y, ca, sa, nm, tm, mf;
};
__device__ __forceinline__ Frame frame(const sc &e, double L, double x, double y, double iR) {
  Frame r;
  r.x = fma(L, e.c, x);
  r.y = fma(L, e.s, y);
  r.ca = mul(r.x, iR);
  r.sa = mul(r.y, iR);
  r.nm = fma(r.ca, e.c, mul(r.sa, e.s));
  r.tm = fma(r.ca, e.s, -mul(r.sa, e.c));
  r.mf = -mul(L, r.tm);
  return r;
}
// The track's direction (nu, tu) in the frame, the chord's turned by h; ic =
// 1 / nu, tau = tu / nu and the t row v = t.J_s - tau m but for its entry vk.
struct Slope {
  double ic, tau, vx, vy, vf;
};
__device__ __forceinline__ Slope slope(const Frame &f, double ch, double sh, double L) {
  Slope r;
  const double nu = fma(f.nm, ch, -mul(f.tm, sh)), tu = fma(f.tm, ch, mul(f.nm, sh));
  r.ic = rcp(nu);
  r.tau = mul(tu, r.ic);
  r.vx = fma(-r.tau, f.ca, -f.sa);
  r.vy = fma(-r.tau, f.sa, f.ca);
  r.vf = fma(-r.tau, f.mf, mul(L, f.nm));
  return r;
}
// (mk, vk): the entries of m and v along k.
__device__ __forceinline__ Pair along_k(double a, double b, double nm, double tm, double tau) {
  const double mk = fma(a, nm, -mul(b, tm));
  return {mk, fma(-tau, mk, fma(a, tm, mul(b, nm)))};
}
// A row (m0, m1, mk, mf) over (x, y, k, phi) times a column: the part without
// k (known before the turning angle is), and the whole.
__device__ __forceinline__ double part(double m0, double m1, double mf, double c0, double c1,
                                       double c4) {
  return fma(mf, c4, fma(m1, c1, mul(m0, c0)));
}

// Measurement direction at the hit, u = (-hy, hx) / |h|, and V = P V_hit P^T.
struct HitFrame {
  double ux, uy, V00, V01;
};
__device__ __forceinline__ HitFrame hit_frame(double hx, double hy, const double (&hc)[6]) {
  HitFrame r;
  const double ir = rsqrt(fma(hx, hx, mul(hy, hy)));
  r.ux = -mul(hy, ir);
  r.uy = mul(hx, ir);
  r.V00 = fma(r.ux, fma(r.ux, hc[0], mul(r.uy, hc[1])),
              mul(r.uy, fma(r.ux, hc[1], mul(r.uy, hc[2]))));
  r.V01 = fma(r.ux, hc[3], mul(r.uy, hc[4]));
  return r;
}

// ------------------------------------------------------------------- steps

// The Kalman update of both step kinds, on the five components that carry
// variance: index M0 of p and C is the first measured component (with weight
// h0, 1 on a plane), M1 the second, 3, 4, 5 the others.  C holds C', p the
// propagated state, r0, r1 the residual.  The measured rows and columns use
// C'' H^T = K V, which cancels no digits; the rest C' - K (H C').  Returns
// kSNotPD and leaves p and C alone if S is not positive definite.
template <int M0, int M1, bool UNIT0>
__device__ __forceinline__ unsigned update(double (&p)[6], double (&C)[21], double h0, double V00,
                                           double V01, double V11, double r0, double r1) {
  constexpr int kAll[5] = {M0, M1, 3, 4, 5};
  const Gain g = gain<UNIT0>(C[tri(M0, M0)], C[tri(M1, M0)], C[tri(M1, M1)], h0, V00, V01, V11);
  if (g.bad) return kSNotPD;
  Pair K[6];
#pragma unroll
  for (int e = 0; e < 5; ++e) {
    const int i = kAll[e];
    K[i] = gain_of(g, C[tri(i, M0)], C[tri(i, M1)]);
    p[i] = dot_add(K[i], r0, r1, p[i]);
  }
  // the unmeasured block first: it needs C's measured columns as they were
#pragma unroll
  for (int i = 3; i < 6; ++i) {
    const Pair k{UNIT0 ? K[i].a : mul(h0, K[i].a), K[i].b};
#pragma unroll
    for (int m = 3; m <= i; ++m)
      C[tri(i, m)] = reduced(k, C[tri(m, M0)], C[tri(m, M1)], C[tri(i, m)]);
  }
  const double ih = UNIT0 ? 1.0 : rcp(h0);
  const double W00 = UNIT0 ? V00 : mul(V00, ih), W01 = UNIT0 ? V01 : mul(V01, ih);
#pragma unroll
  for (int e = 0; e < 5; ++e) {
    const int i = kAll[e];
    C[tri(i, M0)] = dot(K[i], W00, W01);
    if (i != M0) C[tri(i, M1)] = dot(K[i], V01, V11);
  }
  return 0u;
}

// One p2z step: propagate to the plane z = zt and update with (hx, hy).
// p and C are left alone when the track is parallel to the plane.
//
// J = J_s + u ds with u = d p'/ds = (cos, sin, ., 0, omega, 0) after the step
// and ds = (ds/dz, ds/dtheta) the only entries of the path-length gradient;
// J_s has rows x: e_x + Xk e_k + Xf e_phi, y: e_y + Yk e_k + Yf e_phi,
// phi: e_phi + kap e_k.  So with c = C ds^T and B = J_s C J_s^T,
// C'_ab = B_ab + u_a (e_b + u_b dd) + u_b e_a, e = J_s c, dd = ds c.
__device__ __forceinline__ unsigned p2z_step(double (&p)[6], double (&C)[21], double q, double bz,
                                             double zt, double hx, double hy, double vxx,
                                             double vxy, double vyy) {
  const double dw = curvature_rate(q, bz), w = mul(dw, p[3]);
  const PlanePath pa = plane_path(sincos(p[5]), sub(zt, p[2]), w);
  if (!pa.ok) return kNoIntersect;
  const sc hh = sincos(pa.h);
  const double kap = mul(pa.s, dw);
  const Bend be = bend(pa.s, half_s_kap(pa.s, kap), sinc(pa.h, hh.s, hh.c));
  const sc e = turned(sincos(p[4]), hh), f = turned(e, hh);
  const double Xk = fma(be.a, e.c, -mul(be.b, e.s)), Yk = fma(be.a, e.s, mul(be.b, e.c));
  const double Xf = -mul(be.L, e.s), Yf = mul(be.L, e.c);
  p[0] = fma(be.L, e.c, p[0]);
  p[1] = fma(be.L, e.s, p[1]);
  p[2] = zt;
  p[4] = fma(2.0, pa.h, p[4]);

  double c[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) c[j] = fma(pa.dsz, C[tri(2, j)], mul(pa.dst, C[tri(5, j)]));
  const double dd = fma(pa.dsz, c[2], mul(pa.dst, c[5]));
  const double ex = row(Xk, Xf, c[0], c[3], c[4]), ey = row(Yk, Yf, c[1], c[3], c[4]);
  const double ef = fma(kap, c[3], c[4]);
  const double gx = fma(f.c, dd, ex), gy = fma(f.s, dd, ey), gf = fma(w, dd, ef);
  auto X = [&](int j) { return row(Xk, Xf, C[tri(0, j)], C[tri(3, j)], C[tri(4, j)]); };
  auto Y = [&](int j) { return row(Yk, Yf, C[tri(1, j)], C[tri(3, j)], C[tri(4, j)]); };
  auto F = [&](int j) { return fma(kap, C[tri(3, j)], C[tri(4, j)]); };
  const double xk = X(3), xf = X(4), yk = Y(3), yf = Y(4), fk = F(3), ff = F(4);
  const double xx = row(Xk, Xf, X(0), xk, xf), xy = row(Yk, Yf, X(1), xk, xf);
  const double yy = row(Yk, Yf, Y(1), yk, yf);
  const double xt = fma(f.c, c[5], X(5)), yt = fma(f.s, c[5], Y(5)), ft = fma(w, c[5], F(5));
  C[tri(0, 0)] = fma(f.c, gx, fma(f.c, ex, xx));
  C[tri(1, 0)] = fma(f.c, gy, fma(f.s, ex, xy));
  C[tri(1, 1)] = fma(f.s, gy, fma(f.s, ey, yy));
  C[tri(4, 0)] = fma(f.c, gf, fma(w, ex, fma(kap, xk, xf)));
  C[tri(4, 1)] = fma(f.s, gf, fma(w, ey, fma(kap, yk, yf)));
  C[tri(4, 4)] = fma(w, gf, fma(w, ef, fma(kap, fk, ff)));
  C[tri(3, 0)] = fma(f.c, c[3], xk);
  C[tri(3, 1)] = fma(f.s, c[3], yk);
  C[tri(4, 3)] = fma(w, c[3], fk);
  C[tri(5, 0)] = xt;
  C[tri(5, 1)] = yt;
  C[tri(5, 4)] = ft;
#pragma unroll
  for (int j = 0; j < 6; ++j) C[tri(2, j)] = 0.0;  // z' is the plane's

  unsigned st = update<0, 1, true>(p, C, 1.0, vxx, vxy, vyy, sub(hx, p[0]), sub(hy, p[1]));
  p[4] = wrap_phi(p[4]);
  if (!gt0(p[3])) st |= kBadK;
  return st;
}

// One p2r step: propagate to the first outward crossing of r = R and update
// with the hit's azimuth and z.  p and C are left alone when the track starts
// outside the cylinder or does not reach it.
//
// In the surface frame (Frame, Slope) J's rows are t: v, z: e_z + zt e_theta + cz m,
// phi: e_phi + kap e_k + cf m, so C' needs only the two products C m^T and
// C v^T.
__device__ __forceinline__ unsigned p2r_step(double (&p)[6], double (&C)[21], double q, double bz,
                                             double R, double hx, double hy, double hz,
                                             const double (&hc)[6]) {
  const double dw = curvature_rate(q, bz), w = mul(dw, p[3]), wh = mul(0.5, w);
  const sc ph = sincos(p[4]);
  const Cross cr = cross(p[0], p[1], ph, w, wh, R);
  if (!cr.ok) return kNoIntersect;
  const sc th = sincos(p[5]);
  const double ist = rcp(th.s), cot = mul(th.c, ist);
  const double h = angle(cr.yh, cr.den, cr.sh, cr.ch), s = arc(cr, h, w, rcp(wh));
  const double kap = mul(s, dw);
  const Bend be = bend(s, half_s_kap(s, kap), sinc(h, cr.sh, cr.ch));
  const Frame ax = frame(turned(ph, {cr.sh, cr.ch}), cr.L, p[0], p[1], rcp(R));
  const Slope sl = slope(ax, cr.ch, cr.sh, cr.L);
  p[0] = ax.x;
  p[1] = ax.y;
  p[2] = fma(s, cot, p[2]);
  p[4] = fma(2.0, h, p[4]);

  const Pair ak = along_k(be.a, be.b, ax.nm, ax.tm, sl.tau);
  const double mk = ak.a, vk = ak.b;
  const double cz = -mul(cot, sl.ic), cf = -mul(w, sl.ic), zt = -mul(mul(s, ist), ist);
  double cm[6], cv[6];  // C m^T, C v^T
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const double c0 = C[tri(0, j)], c1 = C[tri(1, j)], c3 = C[tri(3, j)], c4 = C[tri(4, j)];
    cm[j] = fma(mk, c3, part(ax.ca, ax.sa, ax.mf, c0, c1, c4));
    cv[j] = fma(vk, c3, part(sl.vx, sl.vy, sl.vf, c0, c1, c4));
  }
  const double mm = fma(mk, cm[3], part(ax.ca, ax.sa, ax.mf, cm[0], cm[1], cm[4]));
  const double mv = fma(mk, cv[3], part(ax.ca, ax.sa, ax.mf, cv[0], cv[1], cv[4]));
  const double vv = fma(vk, cv[3], part(sl.vx, sl.vy, sl.vf, cv[0], cv[1], cv[4]));
  const double Czk = C[tri(3, 2)], Czf = C[tri(4, 2)], Czt = C[tri(5, 2)];
  const double Ckk = C[tri(3, 3)], Ckf = C[tri(4, 3)], Ckt = C[tri(5, 3)];
  const double e1 = fma(zt, cm[5], cm[2]), f1 = fma(cz, mm, e1);
  const double e2 = fma(kap, cm[3], cm[4]), f2 = fma(cf, mm, e2);
  const double gz = fma(zt, C[tri(5, 5)], Czt);   // (C' without the path terms) z, theta
  const double gf = fma(kap, Ckk, Ckf);           // phi, k
  const double gt = fma(kap, Ckt, C[tri(5, 4)]);  // phi, theta
  C[tri(0, 0)] = vv;
  C[tri(2, 0)] = fma(cz, mv, fma(zt, cv[5], cv[2]));
  C[tri(3, 0)] = cv[3];
  C[tri(4, 0)] = fma(cf, mv, fma(kap, cv[3], cv[4]));
  C[tri(5, 0)] = cv[5];
  C[tri(2, 2)] = fma(cz, add(f1, e1), fma(zt, add(Czt, gz), C[tri(2, 2)]));
  C[tri(3, 2)] = fma(cz, cm[3], fma(zt, Ckt, Czk));
  C[tri(4, 2)] = fma(cz, f2, fma(cf, e1, fma(zt, gt, fma(kap, Czk, Czf))));
  C[tri(5, 2)] = fma(cz, cm[5], gz);
  C[tri(4, 3)] = fma(cf, cm[3], gf);
  C[tri(4, 4)] = fma(cf, add(f2, e2), fma(kap, add(Ckf, gf), C[tri(4, 4)]));
  C[tri(5, 4)] = fma(cf, cm[5], gt);

  const HitFrame hf = hit_frame(hx, hy, hc);
  const double ut = fma(ax.ca, hf.uy, -mul(ax.sa, hf.ux));  // weight of u on t
  const double r0 = fma(hf.ux, sub(hx, p[0]), mul(hf.uy, sub(hy, p[1])));
  // the state's t and r offsets start at 0 on the crossing point
  double f[6] = {0.0, 0.0, p[2], p[3], p[4], p[5]};
  unsigned st = update<0, 2, false>(f, C, ut, hf.V00, hf.V01, hc[5], r0, sub(hz, p[2]));
  p[0] = fma(-ax.sa, f[0], p[0]);
  p[1] = fma(ax.ca, f[0], p[1]);
#pragma unroll
  for (int i = 2; i < 6; ++i) p[i] = f[i];
  p[4] = wrap_phi(p[4]);
  // back to (x, y): only the t row and column carry position variance
  const double tx = -mul(ax.sa, C[tri(0, 0)]), ty = mul(ax.ca, C[tri(0, 0)]);
  C[tri(0, 0)] = -mul(ax.sa, tx);
  C[tri(1, 0)] = mul(ax.ca, tx);
  C[tri(1, 1)] = mul(ax.ca, ty);
#pragma unroll
  for (int j = 2; j < 6; ++j) {
    const double t = C[tri(j, 0)];
    C[tri(j, 0)] = -mul(ax.sa, t);
    C[tri(j, 1)] = mul(ax.ca, t);
  }
  if (!gt0(p[3])) st |= kBadK;
  return st;
}

}  // namespace f64
}  // namespace kf
