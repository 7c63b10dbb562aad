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
//    27), the turning angle from atan2f and one correction (16 instead of 45);
//  * the transport C' = J C J^T through J's factored form J = J_s + u (ds/dp)
//    (89 multiply-adds for a cylinder, 70 for a plane), and the update
//    without the columns and products the general form spends on them.
// Every operation is a correctly rounded double operation, none is done in
// less: the seeds only choose where the double iteration starts.
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

// (double)f by shifts.  Denormals read as zero (the library is built with
// -ftz=true); infinities and NaN stay what they are.
__device__ __forceinline__ double from_float(float f) {
  const int i = __float_as_int(f), e = i & 0x7f800000;
  const int bias = e == 0x7f800000 ? 0x70000000 : 0x38000000;
  const int hi = ((i >> 3) & (int)0x8fffffff) + bias;
  return __hiloint2double(e == 0 ? i & (int)0x80000000 : hi, e == 0 ? 0 : i << 29);
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
// what is not a normal float, take the instruction.
__device__ __forceinline__ float to_float(double x) {
  if (top(x) - 0x38100000u >= 0x0fe00000u) return (float)x;
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

// sqrt(x) = x / sqrt(x): the same with g = x y in front.
__device__ __forceinline__ double sqrt(double x) {
  if (__double2hiint(x) < 0 || !seedable(x)) return sqrt_any(x);
  float s;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(cut_normal(x)));
  const double y = from_normal(s), g = mul(x, y);
  const double e = fma(-g, y, 1.0);
  return fma(mul(g, e), fma(e, 0.375, 0.5), g);
}

// ------------------------------------------------------------- sin and cos
// sin and cos of k pi/128, k = 0..255, evaluated at compile time by Taylor
// series in double-double arithmetic (Knuth's two-sum, Dekker's product) and
// rounded to double.
struct SinCosTable {
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

struct sc {
  double s, c;
};

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
  const double r = fma(k, -9.567553118338697e-19, fma(k, -0.02454369260617026, x));
  const double2 t =
      __ldg(reinterpret_cast<const double2 *>(&kSinCos.v[(int)kf & 255][0]));
  const double z = mul(r, r);
  const double sr = fma(mul(r, z), fma(z, 0x1.1110b41d9fc27p-7, -0x1.5555555542e06p-3), r);
  const double cr = mul(z, fma(z, fma(z, -1.0 / 720.0, 1.0 / 24.0), -0.5));
  return {fma(t.x, cr, fma(t.y, sr, t.x)), fma(t.y, cr, fma(-t.x, sr, t.y))};
}

static __device__ __noinline__ double atan2_any(double y, double x) { return ::atan2(y, x); }

// atan2(y, x) when its sine and cosine are known (y and x over their norm):
// with the float angle h0, sin(h - h0) = sh cos h0 - ch sin h0 is at most
// 1e-6 and is the correction (its cube is below 1e-18 of it).
__device__ __forceinline__ double angle(double y, double x, double sh, double ch) {
  if (top(y) >= 0x46300000u || top(x) >= 0x46300000u) return atan2_any(y, x);  // 2^100, NaN
  const double h0 = from_float(atan2f(cut(y), cut(x)));
  const sc a = sincos(h0);
  return add(h0, fma(sh, a.c, -mul(ch, a.s)));
}

// S(h) = sin(h)/h and dS/dh from sin(h) and cos(h); below |h| = 0.05, where
// cos(h) - S(h) cancels, the Taylor series (the first terms left out are
// below 1e-18 and 3e-17 of the sums).
__device__ __forceinline__ void sinc(double h, double sh, double ch, double &S, double &dS) {
  if (top(h) < 0x3fa99999u) {  // 0.05
    const double z = mul(h, h);
    S = fma(z,
            fma(z, fma(z, fma(z, 1.0 / 362880.0, -1.0 / 5040.0), 1.0 / 120.0), -1.0 / 6.0), 1.0);
    dS = mul(h, fma(z, fma(z, fma(z, 1.0 / 45360.0, -1.0 / 840.0), 1.0 / 30.0), -1.0 / 3.0));
  } else {
    const double ih = rcp(h);
    S = mul(sh, ih);
    dS = mul(sub(ch, S), ih);
  }
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

// ------------------------------------------------------------------- steps

// The Kalman update of both step kinds, on the five components that carry
// variance: index M0 of p and C is the first measured component (with weight
// h0, 1 on a plane), M1 the second, a, b, c the other three.  C holds C', p
// the propagated state, r0, r1 the residual.  The measured rows and columns
// use C'' H^T = K V, which cancels no digits; the rest C' - K (H C').
// Returns kSNotPD and leaves p and C alone if S is not positive definite.
template <int M0, int M1, bool UNIT0>
__device__ __forceinline__ unsigned update(double (&p)[6], double (&C)[21], double h0, double V00,
                                           double V01, double V11, double r0, double r1) {
  constexpr int kRest[3] = {3, 4, 5};
  constexpr int kAll[5] = {M0, M1, 3, 4, 5};
  const double T0 = C[tri(M0, M0)], T1 = C[tri(M1, M0)], U1 = C[tri(M1, M1)];
  const double S00 = UNIT0 ? add(T0, V00) : fma(mul(h0, h0), T0, V00);
  const double S01 = UNIT0 ? add(T1, V01) : fma(h0, T1, V01);
  const double S11 = add(U1, V11);
  const double det = fma(S00, S11, -mul(S01, S01));
  if (!(gt0(S00) && gt0(det))) return kSNotPD;
  const double inv = rcp(det);
  const double Si00 = mul(S11, inv), Si01 = -mul(S01, inv), Si11 = mul(S00, inv);
  const double a00 = UNIT0 ? Si00 : mul(h0, Si00), a01 = UNIT0 ? Si01 : mul(h0, Si01);
  double K0[6], K1[6];
#pragma unroll
  for (int e = 0; e < 5; ++e) {
    const int i = kAll[e];
    const double t = C[tri(i, M0)], u = C[tri(i, M1)];
    K0[i] = fma(t, a00, mul(u, Si01));
    K1[i] = fma(t, a01, mul(u, Si11));
    p[i] = fma(K0[i], r0, fma(K1[i], r1, p[i]));
  }
  // the unmeasured block first: it needs C's measured columns as they were
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    const int i = kRest[e];
    const double k0 = UNIT0 ? K0[i] : mul(h0, K0[i]);
#pragma unroll
    for (int f = 0; f <= e; ++f) {
      const int m = kRest[f];
      C[tri(i, m)] =
          fma(-k0, C[tri(m, M0)], fma(-K1[i], C[tri(m, M1)], C[tri(i, m)]));
    }
  }
  const double ih = UNIT0 ? 1.0 : rcp(h0);
  const double W00 = UNIT0 ? V00 : mul(V00, ih), W01 = UNIT0 ? V01 : mul(V01, ih);
#pragma unroll
  for (int e = 0; e < 5; ++e) {
    const int i = kAll[e];
    C[tri(i, M0)] = fma(K0[i], W00, mul(K1[i], W01));
    if (i != M0) C[tri(i, M1)] = fma(K0[i], V01, mul(K1[i], V11));
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
  const sc th = sincos(p[5]);
  if (!abs_gt(th.c, 0x3f1a36e2eb1c432dull)) return kNoIntersect;  // 1e-4
  const sc ph = sincos(p[4]);
  const double ict = rcp(th.c);
  const double tanth = mul(th.s, ict);
  const double dz = sub(zt, p[2]);
  const double s = mul(dz, tanth);
  const double dw = mul(mul(q, -0.299792458e-2), bz);
  const double w = mul(dw, p[3]);
  const double h = mul(mul(0.5, w), s);
  const sc hh = sincos(h);
  double S, dS;
  sinc(h, hh.s, hh.c, S, dS);
  const double L = mul(s, S);
  const double cm = fma(ph.c, hh.c, -mul(ph.s, hh.s)), sm = fma(ph.c, hh.s, mul(ph.s, hh.c));
  const double c1 = fma(cm, hh.c, -mul(sm, hh.s)), s1 = fma(cm, hh.s, mul(sm, hh.c));
  const double kap = mul(s, dw);
  const double hs2 = mul(mul(0.5, s), kap);
  const double a = mul(hs2, dS), b = mul(hs2, S);
  const double Xk = fma(a, cm, -mul(b, sm)), Yk = fma(a, sm, mul(b, cm));
  const double Xf = -mul(L, sm), Yf = mul(L, cm);
  const double dsz = -tanth, dst = mul(mul(dz, ict), ict);
  p[0] = fma(L, cm, p[0]);
  p[1] = fma(L, sm, p[1]);
  p[2] = zt;
  p[4] = fma(2.0, h, p[4]);

  const double *Z[6] = {&C[3], &C[4], &C[5], &C[8], &C[12], &C[17]};      // row z of C
  const double *T[6] = {&C[15], &C[16], &C[17], &C[18], &C[19], &C[20]};  // row theta
  double c[6];
#pragma unroll
  for (int j = 0; j < 6; ++j) c[j] = fma(dsz, *Z[j], mul(dst, *T[j]));
  const double dd = fma(dsz, c[2], mul(dst, c[5]));
  const double ex = fma(Xf, c[4], fma(Xk, c[3], c[0]));
  const double ey = fma(Yf, c[4], fma(Yk, c[3], c[1]));
  const double ef = fma(kap, c[3], c[4]);
  const double gx = fma(c1, dd, ex), gy = fma(s1, dd, ey), gf = fma(w, dd, ef);
  auto X = [&](int j) { return fma(Xf, C[tri(4, j)], fma(Xk, C[tri(3, j)], C[tri(0, j)])); };
  auto Y = [&](int j) { return fma(Yf, C[tri(4, j)], fma(Yk, C[tri(3, j)], C[tri(1, j)])); };
  auto F = [&](int j) { return fma(kap, C[tri(3, j)], C[tri(4, j)]); };
  const double xk = X(3), xf = X(4), yk = Y(3), yf = Y(4), fk = F(3), ff = F(4);
  const double xx = fma(Xf, xf, fma(Xk, xk, X(0))), xy = fma(Yf, xf, fma(Yk, xk, X(1)));
  const double yy = fma(Yf, yf, fma(Yk, yk, Y(1)));
  const double xt = fma(c1, c[5], X(5)), yt = fma(s1, c[5], Y(5)), ft = fma(w, c[5], F(5));
  C[tri(0, 0)] = fma(c1, gx, fma(c1, ex, xx));
  C[tri(1, 0)] = fma(c1, gy, fma(s1, ex, xy));
  C[tri(1, 1)] = fma(s1, gy, fma(s1, ey, yy));
  C[tri(4, 0)] = fma(c1, gf, fma(w, ex, fma(kap, xk, xf)));
  C[tri(4, 1)] = fma(s1, gf, fma(w, ey, fma(kap, yk, yf)));
  C[tri(4, 4)] = fma(w, gf, fma(w, ef, fma(kap, fk, ff)));
  C[tri(3, 0)] = fma(c1, c[3], xk);
  C[tri(3, 1)] = fma(s1, c[3], yk);
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
// The crossing as in propagate_to_r (kf_device.cuh), with half the curvature
// wh = omega/2 and yh = wh d, so that (cos h, sin h, chord) = (den, yh, d) /
// hypot(den, yh).  In the surface frame n = (ca, sa), t = (-sa, ca) the path
// derivative is ds = -m/(n.u) with m = n.J_s = (ca, sa, ., mk, mf, .), so J's
// rows are
//   t: v = t.J_s - tau m (tau = (t.u)/(n.u)),  z: e_z + zt e_theta + cz m,
//   phi: e_phi + kap e_k + cf m,
// and C' needs only the two products C m^T and C v^T.  The directions come
// from rotating (n.e, t.e), e the chord's direction, by the half angle.
__device__ __forceinline__ unsigned p2r_step(double (&p)[6], double (&C)[21], double q, double bz,
                                             double R, double hx, double hy, double hz,
                                             const double (&hc)[6]) {
  const double x = p[0], y = p[1];
  const double d = fma(R, R, -fma(x, x, mul(y, y)));
  if (!gt0(d)) return kNoIntersect;
  const sc ph = sincos(p[4]);
  const double dw = mul(mul(q, -0.299792458e-2), bz);
  const double w = mul(dw, p[3]), wh = mul(0.5, w);
  const double A = fma(x, ph.c, mul(y, ph.s)), B = fma(y, ph.c, -mul(x, ph.s));
  const double yh = mul(wh, d);
  const double D = fma(A, A, mul(fma(w, B, fma(-wh, yh, 1.0)), d));
  if (!ge0(D)) return kNoIntersect;
  const sc th = sincos(p[5]);
  const double den = add(A, sqrt(D));
  const double inv = rsqrt(fma(den, den, mul(yh, yh)));
  const double ch = mul(den, inv), sh = mul(yh, inv), L = mul(d, inv);
  const double h = angle(yh, den, sh, ch);
  const double s =
      top(w) > 0x3d719799u ? mul(h, rcp(wh)) : mul(d, rcp(den));  // 1e-12; 2 h / omega
  double S, dS;
  sinc(h, sh, ch, S, dS);
  const double cm = fma(ph.c, ch, -mul(ph.s, sh)), sm = fma(ph.c, sh, mul(ph.s, ch));
  const double ist = rcp(th.s), cot = mul(th.c, ist);
  p[0] = fma(L, cm, x);
  p[1] = fma(L, sm, y);
  p[2] = fma(s, cot, p[2]);
  p[4] = fma(2.0, h, p[4]);

  const double iR = rcp(R);
  const double ca = mul(p[0], iR), sa = mul(p[1], iR);
  const double nm = fma(ca, cm, mul(sa, sm)), tm = fma(ca, sm, -mul(sa, cm));
  const double nu = fma(nm, ch, -mul(tm, sh)), tu = fma(tm, ch, mul(nm, sh));
  const double kap = mul(s, dw);
  const double hs2 = mul(mul(0.5, s), kap);
  const double a = mul(hs2, dS), b = mul(hs2, S);
  const double ic = rcp(nu), tau = mul(tu, ic);
  const double cz = -mul(cot, ic), cf = -mul(w, ic);
  const double zt = -mul(mul(s, ist), ist);
  // m and v over the components x, y, k, phi
  const double m[4] = {ca, sa, fma(a, nm, -mul(b, tm)), -mul(L, tm)};
  const double v[4] = {fma(-tau, ca, -sa), fma(-tau, sa, ca),
                       fma(-tau, m[2], fma(a, tm, mul(b, nm))), fma(-tau, m[3], mul(L, nm))};
  double cm_[6], cv[6];  // C m^T, C v^T
#pragma unroll
  for (int j = 0; j < 6; ++j) {
    const double c0 = C[tri(0, j)], c1 = C[tri(1, j)], c3 = C[tri(3, j)], c4 = C[tri(4, j)];
    cm_[j] = fma(m[3], c4, fma(m[2], c3, fma(m[1], c1, mul(m[0], c0))));
    cv[j] = fma(v[3], c4, fma(v[2], c3, fma(v[1], c1, mul(v[0], c0))));
  }
  const double mm = fma(m[3], cm_[4], fma(m[2], cm_[3], fma(m[1], cm_[1], mul(m[0], cm_[0]))));
  const double mv = fma(m[3], cv[4], fma(m[2], cv[3], fma(m[1], cv[1], mul(m[0], cv[0]))));
  const double vv = fma(v[3], cv[4], fma(v[2], cv[3], fma(v[1], cv[1], mul(v[0], cv[0]))));
  const double Czk = C[tri(3, 2)], Czf = C[tri(4, 2)], Czt = C[tri(5, 2)];
  const double Ckk = C[tri(3, 3)], Ckf = C[tri(4, 3)], Ckt = C[tri(5, 3)];
  const double e1 = fma(zt, cm_[5], cm_[2]), f1 = fma(cz, mm, e1);
  const double e2 = fma(kap, cm_[3], cm_[4]), f2 = fma(cf, mm, e2);
  const double gz = fma(zt, C[tri(5, 5)], Czt);           // (C' without the path terms) z, theta
  const double gf = fma(kap, Ckk, Ckf);                   // phi, k
  const double gt = fma(kap, Ckt, C[tri(5, 4)]);          // phi, theta
  C[tri(0, 0)] = vv;
  C[tri(2, 0)] = fma(cz, mv, fma(zt, cv[5], cv[2]));
  C[tri(3, 0)] = cv[3];
  C[tri(4, 0)] = fma(cf, mv, fma(kap, cv[3], cv[4]));
  C[tri(5, 0)] = cv[5];
  C[tri(2, 2)] = fma(cz, add(f1, e1), fma(zt, add(Czt, gz), C[tri(2, 2)]));
  C[tri(3, 2)] = fma(cz, cm_[3], fma(zt, Ckt, Czk));
  C[tri(4, 2)] = fma(cz, f2, fma(cf, e1, fma(zt, gt, fma(kap, Czk, Czf))));
  C[tri(5, 2)] = fma(cz, cm_[5], gz);
  C[tri(4, 3)] = fma(cf, cm_[3], gf);
  C[tri(4, 4)] = fma(cf, add(f2, e2), fma(kap, add(Ckf, gf), C[tri(4, 4)]));
  C[tri(5, 4)] = fma(cf, cm_[5], gt);

  // measurement direction at the hit u = (-hy, hx) / |h|, weight u.t on t
  const double ir = rsqrt(fma(hx, hx, mul(hy, hy)));
  const double ux = -mul(hy, ir), uy = mul(hx, ir);
  const double ut = fma(ca, uy, -mul(sa, ux));
  const double V00 = fma(ux, fma(ux, hc[0], mul(uy, hc[1])),
                         mul(uy, fma(ux, hc[1], mul(uy, hc[2]))));
  const double V01 = fma(ux, hc[3], mul(uy, hc[4]));
  const double r0 = fma(ux, sub(hx, p[0]), mul(uy, sub(hy, p[1])));
  // the state's t and r offsets start at 0 on the crossing point
  double f[6] = {0.0, 0.0, p[2], p[3], p[4], p[5]};
  unsigned st = update<0, 2, false>(f, C, ut, V00, V01, hc[5], r0, sub(hz, p[2]));
  p[0] = fma(-sa, f[0], p[0]);
  p[1] = fma(ca, f[0], p[1]);
#pragma unroll
  for (int i = 2; i < 6; ++i) p[i] = f[i];
  p[4] = wrap_phi(p[4]);
  // back to (x, y): only the t row and column carry position variance
  const double tx = -mul(sa, C[tri(0, 0)]), ty = mul(ca, C[tri(0, 0)]);
  C[tri(0, 0)] = -mul(sa, tx);
  C[tri(1, 0)] = mul(ca, tx);
  C[tri(1, 1)] = mul(ca, ty);
#pragma unroll
  for (int j = 2; j < 6; ++j) {
    const double t = C[tri(j, 0)];
    C[tri(j, 0)] = -mul(sa, t);
    C[tri(j, 1)] = mul(ca, t);
  }
  if (!gt0(p[3])) st |= kBadK;
  return st;
}

}  // namespace f64
}  // namespace kf
