// kf_fp64_group.cuh -- the double-precision step of 32 tracks by four warps.
//
// One thread per track leaves a small batch bound by latency: an FP64 warp
// instruction takes its scheduler's pipe for 64 cycles, so the 359 (p2r) or
// 235 (p2z) of a step are 11 and 7 us on one scheduler while the SM's other
// three pipes are idle, and a 15-layer chain takes 160 us however few tracks
// there are (the redo of 30 marked tracks of a 5,000-track event, say).  Here
// the block's four warps (one per scheduler) run the same 32 tracks, each warp
// other parts of each step, with the state and what the parts exchange in
// shared memory ([slot][32], conflict-free): 6.4 us per p2r and 5.1 per p2z
// layer, a 15-layer chain 91 us.  What bounds it is the step's own chain of
// dependent operations (136 and 98 FP64 instructions in a row at the 76-90
// cycles they take when all four schedulers issue them).  As all four pipes
// work on every track, two and three such blocks on an SM still lead one
// thread per track.  A track's arithmetic is made of the pieces of kf_fp64.cuh
// in the same order, so the results are the same bit for bit.
//
// A split over the lanes of one warp was counted out: the lanes would have to
// run one instruction stream, and what a step does for a row of C' or a
// coordinate of the crossing differs from row to row.
#pragma once

#include "kf_chain.cuh"
#include "kf_device.cuh"
#include "kf_step.cuh"

namespace kf {
namespace f64 {

constexpr int kGroupThreads = kSharedChainThreads;
// Of a block's marked tracks, up to this many run 32 at a time by its four
// warps, more one to a thread: that keeps the schedulers as busy with a seventh
// fewer instructions.
constexpr int kGroupMax = 64;

// Slots of the shared state: the track, C' between transport and update, the
// sines and cosines of the track's angles, and what the warps exchange within
// a step (the two kinds of step in turn).
enum Slot : int {
  kP = 0,
  kC = 6,
  kN = 27,
  kPhS = 48, kPhC, kThS, kThC,
  kKap, kL, kPhi, kAx, kAy, kR0, kR1, kHx, kHy, kV00, kV01, kV11,
  kX,
  // p2r
  kCh = kX, kSh, kIst, kCot, kIwh, kIR, kUx, kUy, kHz, kA, kB, kS, kCa, kSa, kNm, kTm, kMf,
  kTau, kIc, kVx, kVy, kVf, kCm, kCv = kCm + 6, kZt = kCv + 6, kCz, kCf, kZ, kUt, kW00, kW01,
  kSlots,
  // p2z
  kAng = kX, kLen, kHs2, kDsz, kDst, kHhS, kHhC, kSer, kDSer, kFk, kFt, kFf, kDd, kCc
};
static_assert(kCc + 6 <= kSlots, "a plane's slots fit");

struct Shared {
  double v[kSlots][32];
  int ok[32];            // the track reaches the layer's surface
  unsigned status[4][32];
};

// The calling thread's view: its track (lane) and its warp's part in a step.
struct Group {
  Shared &sh;
  int role, lane;
  __device__ __forceinline__ double get(int slot) const { return sh.v[slot][lane]; }
  __device__ __forceinline__ void put(int slot, double x) const { sh.v[slot][lane] = x; }
  __device__ __forceinline__ double c(int i, int j) const { return get(kC + tri(i, j)); }
  __device__ __forceinline__ double n(int i, int j) const { return get(kN + tri(i, j)); }
  __device__ __forceinline__ void put_c(int i, int j, double x) const { put(kC + tri(i, j), x); }
  __device__ __forceinline__ void put_n(int i, int j, double x) const { put(kN + tri(i, j), x); }
};

// Warps 1 to 3 only (warp 0 is on the turning angle).  bar.sync wants the whole
// warp at one instruction, and a lane whose reciprocal has no seed has just been
// in a call of its own: the warp is brought together first.
__device__ __forceinline__ void sync_123() {
  __syncwarp();
  asm volatile("bar.sync 1, 96;" ::: "memory");
}

// The sine and cosine of an angle that a warp has just updated (slots s, s+1).
__device__ __forceinline__ void put_sincos(const Group &g, int s, double x) {
  const sc t = sincos(x);
  g.put(s, t.s);
  g.put(s + 1, t.c);
}

// One p2z step of the block's tracks (p2z_step, kf_fp64.cuh).  Every thread
// calls it; h is read by warp 3 only; more: another step follows (its sines and
// cosines are then made where they cost least, beside the update).  Ends with
// a barrier.
__device__ __forceinline__ unsigned group_p2z(const Group &g, double dw, double zt,
                                              const LayerHit &h, bool more) {
  unsigned st = 0;
  const double w = mul(dw, g.get(kP + 3));
  if (g.role == 0) {
    const PlanePath pa =
        plane_path({g.get(kThS), g.get(kThC)}, sub(zt, g.get(kP + 2)), w);
    const double kap = mul(pa.s, dw);
    g.sh.ok[g.lane] = pa.ok;
    g.put(kAng, pa.h);
    g.put(kLen, pa.s);
    g.put(kKap, kap);
    g.put(kHs2, half_s_kap(pa.s, kap));
    g.put(kDsz, pa.dsz);
    g.put(kDst, pa.dst);
  } else if (g.role == 3) {
    g.put(kHx, from_float(h.hx));
    g.put(kHy, from_float(h.hy));
    g.put(kV00, from_float(h.hc[0]));
    g.put(kV01, from_float(h.hc[1]));
    g.put(kV11, from_float(h.hc[2]));
  }
  __syncthreads();
  const double ha = g.get(kAng), kap = g.get(kKap);
  const bool series = sinc_by_series(ha);
  if (g.role == 0) {
    put_sincos(g, kHhS, ha);
    g.put(kPhi, fma(2.0, ha, g.get(kP + 4)));
  } else if (g.role == 1) {  // S and dS, or what their quotients need
    if (series) {
      const Sinc s = sinc_series(ha);
      g.put(kSer, s.S);
      g.put(kDSer, s.dS);
    } else {
      g.put(kSer, rcp(ha));
    }
  } else if (g.role == 2) {
    const double dsz = g.get(kDsz), dst = g.get(kDst);
    double c[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) g.put(kCc + j, c[j] = fma(dsz, g.c(2, j), mul(dst, g.c(5, j))));
    g.put(kDd, fma(dsz, c[2], mul(dst, c[5])));
  } else {
    const double fk = fma(kap, g.c(3, 3), g.c(4, 3));
    g.put(kFk, fk);
    g.put(kFt, fma(kap, g.c(5, 3), g.c(5, 4)));
    g.put(kFf, fma(kap, fk, fma(kap, g.c(4, 3), g.c(4, 4))));
  }
  __syncthreads();
  {
    const sc hh{g.get(kHhS), g.get(kHhC)};
    Sinc s = sinc_quotient(g.get(kSer), hh.s, hh.c);
    if (series) s = {g.get(kSer), g.get(kDSer)};
    const Bend be = bend(g.get(kLen), g.get(kHs2), s);
    const sc e = turned({g.get(kPhS), g.get(kPhC)}, hh);
    const double c3 = g.get(kCc + 3), c4 = g.get(kCc + 4), c5 = g.get(kCc + 5);
    const double dd = g.get(kDd), ef = fma(kap, c3, c4), gf = fma(w, dd, ef);
    if (g.role == 0) {
      const double x = fma(be.L, e.c, g.get(kP)), y = fma(be.L, e.s, g.get(kP + 1));
      g.put(kAx, x);
      g.put(kAy, y);
      g.put(kR0, sub(g.get(kHx), x));
      g.put(kR1, sub(g.get(kHy), y));
      g.put_n(4, 4, fma(w, gf, fma(w, ef, g.get(kFf))));
      g.put_n(4, 3, fma(w, c3, g.get(kFk)));
      g.put_n(5, 4, fma(w, c5, g.get(kFt)));
    } else {
      const sc f = turned(e, hh);
      const double Xk = fma(be.a, e.c, -mul(be.b, e.s)), Yk = fma(be.a, e.s, mul(be.b, e.c));
      const double Xf = -mul(be.L, e.s), Yf = mul(be.L, e.c);
      auto X = [&](int j) { return row(Xk, Xf, g.c(0, j), g.c(3, j), g.c(4, j)); };
      auto Y = [&](int j) { return row(Yk, Yf, g.c(1, j), g.c(3, j), g.c(4, j)); };
      if (g.role == 1) {
        const double xk = X(3), xf = X(4), ex = row(Xk, Xf, g.get(kCc), c3, c4);
        const double gx = fma(f.c, dd, ex);
        g.put_n(0, 0, fma(f.c, gx, fma(f.c, ex, row(Xk, Xf, X(0), xk, xf))));
        g.put_n(4, 0, fma(f.c, gf, fma(w, ex, fma(kap, xk, xf))));
        g.put_n(3, 0, fma(f.c, c3, xk));
        g.put_n(5, 0, fma(f.c, c5, X(5)));
      } else if (g.role == 2) {
        const double yk = Y(3), yf = Y(4), ey = row(Yk, Yf, g.get(kCc + 1), c3, c4);
        const double gy = fma(f.s, dd, ey);
        g.put_n(1, 1, fma(f.s, gy, fma(f.s, ey, row(Yk, Yf, Y(1), yk, yf))));
        g.put_n(4, 1, fma(f.s, gf, fma(w, ey, fma(kap, yk, yf))));
        g.put_n(3, 1, fma(f.s, c3, yk));
        g.put_n(5, 1, fma(f.s, c5, Y(5)));
      } else {
        const double ex = row(Xk, Xf, g.get(kCc), c3, c4);
        const double ey = row(Yk, Yf, g.get(kCc + 1), c3, c4);
        g.put_n(1, 0, fma(f.c, fma(f.s, dd, ey), fma(f.s, ex, row(Yk, Yf, X(1), X(3), X(4)))));
      }
    }
  }
  __syncthreads();
  if (g.sh.ok[g.lane]) {
    const double V00 = g.get(kV00), V01 = g.get(kV01), V11 = g.get(kV11);
    const double r0 = g.get(kR0), r1 = g.get(kR1);
    const Gain ga = gain<true>(g.n(0, 0), g.n(1, 0), g.n(1, 1), 1.0, V00, V01, V11);
    auto pair = [&](int i) { return gain_of(ga, g.n(i, 0), i == 0 ? g.n(1, 0) : g.n(i, 1)); };
    auto state = [&](const Pair &k, double p) {
      const double v = dot_add(k, r0, r1, p);
      return ga.bad ? p : v;
    };
    auto columns = [&](int i, const Pair &k) {  // the measured columns of row i
      const double v0 = dot(k, V00, V01), v1 = dot(k, V01, V11);
      g.put_c(i, 0, ga.bad ? g.n(i, 0) : v0);
      if (i != 0) g.put_c(i, 1, ga.bad ? g.n(i, 1) : v1);
    };
    auto rest = [&](int i, int m, const Pair &k, double c) {
      const double v = reduced(k, g.n(m, 0), g.n(m, 1), c);
      g.put_c(i, m, ga.bad ? c : v);
    };
    if (g.role == 0) {
      const Pair kx = pair(0), kk = pair(3);
      const double k1 = state(kk, g.get(kP + 3));
      g.put(kP, state(kx, g.get(kAx)));
      g.put(kP + 3, k1);
      columns(0, kx);
      columns(3, kk);
      rest(3, 3, kk, g.c(3, 3));
      if (ga.bad) st |= kSNotPD;
      if (!gt0(k1)) st |= kBadK;
    } else if (g.role == 1) {
      const Pair ky = pair(1), kf = pair(4), kt = pair(5);
      g.put(kP + 1, state(ky, g.get(kAy)));
      columns(1, ky);
      rest(4, 3, kf, g.n(4, 3));
      rest(4, 4, kf, g.n(4, 4));
      rest(5, 5, kt, g.c(5, 5));
    } else if (g.role == 2) {
      const Pair kf = pair(4);
      const double phi = wrap_phi(state(kf, g.get(kPhi)));
      g.put(kP + 4, phi);
      columns(4, kf);
      g.put(kP + 2, zt);
#pragma unroll
      for (int j = 0; j < 6; ++j) g.put_c(2, j, 0.0);
      if (more) put_sincos(g, kPhS, phi);
    } else {
      const Pair kt = pair(5);
      const double th = state(kt, g.get(kP + 5));
      g.put(kP + 5, th);
      columns(5, kt);
      rest(5, 3, kt, g.c(5, 3));
      rest(5, 4, kt, g.n(5, 4));
      if (more) put_sincos(g, kThS, th);
    }
  } else if (g.role == 0) {
    st |= kNoIntersect;
  }
  __syncthreads();
  return st;
}

// One p2r step of the block's tracks (p2r_step, kf_fp64.cuh), likewise.
__device__ __forceinline__ unsigned group_p2r(const Group &g, double dw, double R,
                                              const LayerHit &h, bool more) {
  unsigned st = 0;
  Cross cr;
  const double w = mul(dw, g.get(kP + 3)), wh = mul(0.5, w);
  if (g.role == 0) {
    cr = cross(g.get(kP), g.get(kP + 1), {g.get(kPhS), g.get(kPhC)}, w, wh, R);
    g.sh.ok[g.lane] = cr.ok;
    g.put(kCh, cr.ch);
    g.put(kSh, cr.sh);
    g.put(kL, cr.L);
  } else if (g.role == 1) {
    const double ist = rcp(g.get(kThS));
    g.put(kIst, ist);
    g.put(kCot, mul(g.get(kThC), ist));
    g.put(kIwh, rcp(wh));
  } else if (g.role == 2) {
    g.put(kIR, rcp(R));
  } else {
    double hc[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) hc[e] = from_float(h.hc[e]);
    const double hx = from_float(h.hx), hy = from_float(h.hy);
    const HitFrame hf = hit_frame(hx, hy, hc);
    g.put(kUx, hf.ux);
    g.put(kUy, hf.uy);
    g.put(kV00, hf.V00);
    g.put(kV01, hf.V01);
    g.put(kV11, hc[5]);
    g.put(kHx, hx);
    g.put(kHy, hy);
    g.put(kHz, from_float(h.hz));
  }
  __syncthreads();
  // Warp 0: the turning angle.  Warp 2: the surface frame, and with it the
  // others begin the products C m^T, C v^T (their parts without k, which needs
  // the angle): pm[] three columns each of warps 1 and 3, pv[] two columns each
  // of all three.
  const int j0 = g.role - 1, j1 = g.role + 2, jm = g.role == 1 ? 0 : 3;
  double pm[3] = {0.0, 0.0, 0.0}, pv[2] = {0.0, 0.0};
  if (g.role == 0) {
    const double ha = angle(cr.yh, cr.den, cr.sh, cr.ch), s = arc(cr, ha, w, g.get(kIwh));
    const double kap = mul(s, dw);
    const Bend be = bend(s, half_s_kap(s, kap), sinc(ha, cr.sh, cr.ch));
    g.put(kS, s);
    g.put(kKap, kap);
    g.put(kA, be.a);
    g.put(kB, be.b);
    g.put(kPhi, fma(2.0, ha, g.get(kP + 4)));
  } else {
    Frame fr;
    const double ch = g.get(kCh), sh = g.get(kSh), L = g.get(kL);
    if (g.role == 2) {
      fr = frame(turned({g.get(kPhS), g.get(kPhC)}, {sh, ch}), L, g.get(kP), g.get(kP + 1),
                 g.get(kIR));
      g.put(kAx, fr.x);
      g.put(kAy, fr.y);
      g.put(kCa, fr.ca);
      g.put(kSa, fr.sa);
      g.put(kNm, fr.nm);
      g.put(kTm, fr.tm);
      g.put(kMf, fr.mf);
    }
    sync_123();
    if (g.role == 2) {
      const Slope sl = slope(fr, ch, sh, L);
      g.put(kIc, sl.ic);
      g.put(kTau, sl.tau);
      g.put(kVx, sl.vx);
      g.put(kVy, sl.vy);
      g.put(kVf, sl.vf);
    } else {
      const double ca = g.get(kCa), sa = g.get(kSa), mf = g.get(kMf);
      const double ux = g.get(kUx), uy = g.get(kUy);
#pragma unroll
      for (int j = 0; j < 3; ++j)
        pm[j] = part(ca, sa, mf, g.c(0, jm + j), g.c(1, jm + j), g.c(4, jm + j));
      if (g.role == 1)
        g.put(kR0, fma(ux, sub(g.get(kHx), g.get(kAx)), mul(uy, sub(g.get(kHy), g.get(kAy)))));
      else
        g.put(kUt, fma(ca, uy, -mul(sa, ux)));
    }
    sync_123();
    const double vx = g.get(kVx), vy = g.get(kVy), vf = g.get(kVf);
    pv[0] = part(vx, vy, vf, g.c(0, j0), g.c(1, j0), g.c(4, j0));
    pv[1] = part(vx, vy, vf, g.c(0, j1), g.c(1, j1), g.c(4, j1));
  }
  __syncthreads();
  const double ca = g.get(kCa), sa = g.get(kSa), kap = g.get(kKap);
  const Pair ak = along_k(g.get(kA), g.get(kB), g.get(kNm), g.get(kTm), g.get(kTau));
  const double mk = ak.a, vk = ak.b;
  if (g.role == 0) {
    const double ic = g.get(kIc), cot = g.get(kCot), ist = g.get(kIst), s = g.get(kS);
    g.put(kCz, -mul(cot, ic));
    g.put(kCf, -mul(w, ic));
    g.put(kZt, -mul(mul(s, ist), ist));
    const double z = fma(s, cot, g.get(kP + 2));
    g.put(kZ, z);
    g.put(kR1, sub(g.get(kHz), z));
  } else {
    g.put(kCv + j0, fma(vk, g.c(3, j0), pv[0]));
    g.put(kCv + j1, fma(vk, g.c(3, j1), pv[1]));
    if (g.role == 2) {
      const double ih = rcp(g.get(kUt));
      g.put(kW00, mul(g.get(kV00), ih));
      g.put(kW01, mul(g.get(kV01), ih));
    } else {
#pragma unroll
      for (int j = 0; j < 3; ++j) g.put(kCm + jm + j, fma(mk, g.c(3, jm + j), pm[j]));
    }
  }
  __syncthreads();
  const double zt = g.get(kZt), cz = g.get(kCz), cf = g.get(kCf);
  if (g.role == 0 || g.role == 3) {
    const double cm3 = g.get(kCm + 3), cm4 = g.get(kCm + 4);
    const double mm = fma(mk, cm3, part(ca, sa, g.get(kMf), g.get(kCm), g.get(kCm + 1), cm4));
    const double e1 = fma(zt, g.get(kCm + 5), g.get(kCm + 2));
    if (g.role == 0) {
      const double Czt = g.c(5, 2), f1 = fma(cz, mm, e1), gz = fma(zt, g.c(5, 5), Czt);
      g.put_n(2, 2, fma(cz, add(f1, e1), fma(zt, add(Czt, gz), g.c(2, 2))));
    } else {
      const double Ckf = g.c(4, 3), e2 = fma(kap, cm3, cm4), f2 = fma(cf, mm, e2);
      const double gf = fma(kap, g.c(3, 3), Ckf), gt = fma(kap, g.c(5, 3), g.c(5, 4));
      g.put_n(4, 2, fma(cz, f2, fma(cf, e1, fma(zt, gt, fma(kap, g.c(3, 2), g.c(4, 2))))));
      g.put_n(4, 4, fma(cf, add(f2, e2), fma(kap, add(Ckf, gf), g.c(4, 4))));
    }
  } else {
    const double cv3 = g.get(kCv + 3), cv4 = g.get(kCv + 4), cv5 = g.get(kCv + 5);
    if (g.role == 1) {
      const double mv =
          fma(mk, cv3, part(ca, sa, g.get(kMf), g.get(kCv), g.get(kCv + 1), cv4));
      const double gf = fma(kap, g.c(3, 3), g.c(4, 3)), gt = fma(kap, g.c(5, 3), g.c(5, 4));
      g.put_n(2, 0, fma(cz, mv, fma(zt, cv5, g.get(kCv + 2))));
      g.put_n(4, 0, fma(cf, mv, fma(kap, cv3, cv4)));
      g.put_n(4, 3, fma(cf, g.get(kCm + 3), gf));
      g.put_n(5, 4, fma(cf, g.get(kCm + 5), gt));
    } else {
      g.put_n(0, 0, fma(vk, cv3, part(g.get(kVx), g.get(kVy), g.get(kVf), g.get(kCv),
                                      g.get(kCv + 1), cv4)));
      g.put_n(3, 2, fma(cz, g.get(kCm + 3), fma(zt, g.c(5, 3), g.c(3, 2))));
      g.put_n(5, 2, fma(cz, g.get(kCm + 5), fma(zt, g.c(5, 5), g.c(5, 2))));
      g.put_n(3, 0, cv3);
      g.put_n(5, 0, cv5);
    }
  }
  __syncthreads();
  if (g.sh.ok[g.lane]) {
    const double V00 = g.get(kV00), V01 = g.get(kV01), V11 = g.get(kV11);
    const double r0 = g.get(kR0), r1 = g.get(kR1), ut = g.get(kUt);
    const double W00 = g.get(kW00), W01 = g.get(kW01);
    const Gain ga = gain<false>(g.n(0, 0), g.n(2, 0), g.n(2, 2), ut, V00, V01, V11);
    auto pair = [&](int i) { return gain_of(ga, g.n(i, 0), i == 0 ? g.n(2, 0) : g.n(i, 2)); };
    auto state = [&](const Pair &k, double p) {
      const double v = dot_add(k, r0, r1, p);
      return ga.bad ? p : v;
    };
    // row i's measured columns, the t entry rotated back to (x, y)
    auto columns = [&](int i, const Pair &k) {
      const double v0 = dot(k, W00, W01), v1 = dot(k, V01, V11);
      const double t = ga.bad ? g.n(i, 0) : v0;
      g.put_c(i, 0, -mul(sa, t));
      g.put_c(i, 1, mul(ca, t));
      g.put_c(i, 2, ga.bad ? g.n(i, 2) : v1);
    };
    auto weighted = [&](const Pair &k) { return Pair{mul(ut, k.a), k.b}; };
    auto rest = [&](int i, int m, const Pair &k, double c) {
      const double v = reduced(k, g.n(m, 0), g.n(m, 2), c);
      g.put_c(i, m, ga.bad ? c : v);
    };
    if (g.role == 0) {
      const Pair k = pair(0), kf = pair(4), kw = weighted(kf);
      const double f0 = state(k, 0.0), v = dot(k, W00, W01), tt = ga.bad ? g.n(0, 0) : v;
      g.put(kP, fma(-sa, f0, g.get(kAx)));
      g.put(kP + 1, fma(ca, f0, g.get(kAy)));
      const double tx = -mul(sa, tt), ty = mul(ca, tt);
      g.put_c(0, 0, -mul(sa, tx));
      g.put_c(1, 0, mul(ca, tx));
      g.put_c(1, 1, mul(ca, ty));
      columns(4, kf);
      rest(4, 3, kw, g.n(4, 3));
      rest(4, 4, kw, g.n(4, 4));
      if (ga.bad) st |= kSNotPD;
    } else if (g.role == 1) {
      const Pair kz = pair(2), kk = pair(3);
      const double k1 = state(kk, g.get(kP + 3));
      g.put(kP + 2, state(kz, g.get(kZ)));
      g.put(kP + 3, k1);
      columns(2, kz);
      columns(3, kk);
      rest(3, 3, weighted(kk), g.c(3, 3));
      if (!gt0(k1)) st |= kBadK;
    } else if (g.role == 2) {
      const Pair kt = weighted(pair(5));
      const double phi = wrap_phi(state(pair(4), g.get(kPhi)));
      g.put(kP + 4, phi);
      rest(5, 3, kt, g.c(5, 3));
      rest(5, 4, kt, g.n(5, 4));
      rest(5, 5, kt, g.c(5, 5));
      if (more) put_sincos(g, kPhS, phi);
    } else {
      const Pair kt = pair(5);
      const double th = state(kt, g.get(kP + 5));
      g.put(kP + 5, th);
      columns(5, kt);
      if (more) put_sincos(g, kThS, th);
    }
  } else if (g.role == 0) {
    st |= kNoIntersect;
  }
  __syncthreads();
  return st;
}

// The block's threads of lane `lane` share one track: its inputs, strides and
// where its result goes.
struct GroupTrack {
  const float *state_in, *cov_in;
  float *state_out, *cov_out;
  ChainLoc l6, l21;
};

// After the state is in its slots: the sines and cosines a first step needs.
__device__ __forceinline__ void group_begin(const Group &g) {
  __syncthreads();
  if (g.role == 2) put_sincos(g, kPhS, g.get(kP + 4));
  if (g.role == 3) put_sincos(g, kThS, g.get(kP + 5));
  __syncthreads();
}

__device__ __forceinline__ void group_load(const Group &g, const GroupTrack &t) {
#pragma unroll
  for (int e = 0; e < 27; ++e) {
    if ((e & 3) != g.role) continue;
    const float f = e < 6 ? t.state_in[t.l6.base + e * t.l6.stride]
                          : t.cov_in[t.l21.base + (e - 6) * t.l21.stride];
    g.put(e, from_float(f));
  }
  group_begin(g);
}

// The result as floats, [27][32] in the slots of C' (each warp converts every
// fourth), and its status: the OR of the warps' bits and the finite check.
__device__ __forceinline__ const float *group_result(const Group &g, unsigned &st) {
  float *f = reinterpret_cast<float *>(&g.sh.v[kN][0]);
  g.sh.status[g.role][g.lane] = st;
#pragma unroll
  for (int e = 0; e < 27; ++e)
    if ((e & 3) == g.role) f[e * 32 + g.lane] = to_float(g.get(e));
  __syncthreads();
  float p[6], C[21];
#pragma unroll
  for (int c = 0; c < 6; ++c) p[c] = f[c * 32 + g.lane];
#pragma unroll
  for (int e = 0; e < 21; ++e) C[e] = f[(6 + e) * 32 + g.lane];
  st = g.sh.status[0][g.lane] | g.sh.status[1][g.lane] | g.sh.status[2][g.lane] |
       g.sh.status[3][g.lane] | finite_status(p, C);
  return f;
}

// Store the result (each warp every fourth component, where `store`); the
// status for every thread of the track.  The block may go on to other tracks:
// group_load writes no slot that is read here before its own barrier.
__device__ __forceinline__ unsigned group_store(const Group &g, unsigned st, const GroupTrack &t,
                                                bool store) {
  const float *f = group_result(g, st);
  if (store) {
#pragma unroll
    for (int e = 0; e < 27; ++e) {
      if ((e & 3) != g.role) continue;
      const float v = f[e * 32 + g.lane];
      if (e < 6) __stcs(t.state_out + t.l6.base + e * t.l6.stride, v);
      else __stcs(t.cov_out + t.l21.base + (e - 6) * t.l21.stride, v);
    }
  }
  return st;
}

// The calling thread's track of a list of `count` from place `base` on (32 to
// a block): lanes past the end repeat the last track and store nothing.
__device__ __forceinline__ int64_t group_place(int64_t base, int64_t count, int lane) {
  return base + lane < count ? base + lane : count - 1;
}

// chain_track_fp64 (kf_chain.cuh) for the block's 32 tracks: each lane's
// track through layers 0..L-1, and its result stored (not for a lane that only
// repeats another's track).  Warp 3 reads the hits, the next
// layer's while this one computes.
__device__ __forceinline__ unsigned group_chain(const Group &g, const GroupTrack &t, float qf,
                                                float bz, int L, const int32_t *kinds,
                                                const float *pos, const float *hits,
                                                int64_t hit_stride, const float *hitcovs,
                                                int64_t hc_stride, const ChainLoc &l3,
                                                bool store) {
  const double dw = curvature_rate(from_float(qf), from_float(bz));
  HitCursor cur(hits, hit_stride, hitcovs, hc_stride, l3, t.l6);
  LayerHit next{};
  if (g.role == 3) cur.load(next, kinds[0]);
  group_load(g, t);
  unsigned st = 0;
  for (int l = 0; l < L; ++l) {
    const LayerHit h = next;
    if (g.role == 3 && l + 1 < L) {
      cur.next_layer();
      cur.load(next, kinds[l + 1]);
    }
    const double ps = from_float(pos[l]);
    const bool more = l + 1 < L;
    st |= kinds[l] == kP2z ? group_p2z(g, dw, ps, h, more) : group_p2r(g, dw, ps, h, more);
  }
  return group_store(g, st, t, store);
}

}  // namespace f64
}  // namespace kf
