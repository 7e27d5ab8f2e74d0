// Single-particle transfer maps of Sec. III, one particle per thread.  The
// state is float64 and so is every sum that updates x, px, y, py; what such a
// sum adds as a small correction, and sg's change over an element, is worked
// out in pairs of floats (dfloat.h), because the FP64 pipe is the GB300's
// scarcest unit: every FP64 add, multiply, fma, compare, floor and conversion
// takes one of its two slots per SM clock, 64 clocks of a sub-partition per
// warp instruction.
//
// State: (x, px, y, py, sg, ps) with px = Px/p0, sg = s - c beta0 t.
// Per-particle quantities that depend on ps alone (the chromatic factors of
// PsConst, the thick quadrupoles' matrix entries QuadCoef) are computed once
// per call of a tracked turn and kept per particle (ps changes only in RF
// cavities, after which they are refreshed).
#pragma once

#include "dfloat.h"
#include "sc_internal.cuh"

namespace sc {

// Quadrupole flags: the kind (QF_KIND bits) and, from bit QF_FAM_SHIFT, 1 +
// the index of the quadrupole's family in the per-particle coefficient cache
// (0: the map computes its own coefficients).
enum : int { QF_ZERO = 0, QF_FOCUS_X = 1, QF_FOCUS_Y = 2, QF_KIND = 3, QF_FAM_SHIFT = 4 };

// Largest chromatic phase shift |Delta| = |theta0 (sqrt(1-ps) - 1)| handled by
// the angle-addition series: with terms up to Delta^5 (sin) and Delta^4 (cos),
// the truncation is below 2e-18 for |Delta| <= 2^-8; beyond it the library
// sin/cos/sinh/cosh are used.
constexpr double kMaxDelta = 0.00390625;

// What may go to sg as a float pair, per length of the element.  Float64 rounds
// 1 - (1 + beta0^2 ps)/pz, a drift's slip, by up to 7 2^-53, whatever the slip
// itself; a pair rounds by 2^-46 of its terms some ten (drift) to fourteen
// times (quadrupole) over, at most 3.5 2^-53 where they are below kMaxSlip.  That
// is psigma of 3% at 3 GeV or 0.4% at 400 MeV, and some 0.1 m off axis in a
// quadrupole; beyond, the float64 sums.  The change carried along grows by a
// drift's while it is below kMaxCarry of its length: 2^-46 of it is 2^-53.
// (Against no limits: one turn of 1e6 particles, 128^2, TF32 14.9 -> 15.1 ms, a
// batch 109.5 -> 110.4.  A limit for quadrupoles relative to sg itself made a
// sorted bunch in 32 slices 23% slower: the block that holds sg = 0 took the
// float64 sum in nearly every warp, and the launch waited for it.)
constexpr float kMaxSlip = 0.001953125f;
constexpr float kMaxCarry = 0.0078125f;
// A g0 of the plan (PsConst) that stands for none.
constexpr float kNoSlip = 1e30f;

struct State {
  double x, px, y, py, sg, ps;
};

// (The quadrupole's chromatic factor 1 - ps is formed where a map needs it:
// the cached quadrupole map does not.)
struct PsConst {
  // Drift constants: with the series drift (map_drift) r0 = 1/(1+delta) as d0 (1 + eps), eps what
  // rounding it to d0 left, and g0 = 1 - (1 + beta0^2 ps)/(1+delta), sg's change per unit length
  // on the axis, as an F2 in d1; else (1+delta)^2 = 1 + 2 ps + beta0^2 ps^2 (Eq. BEND2) and
  // 1 + beta0^2 ps.
  double d0, d1;
  float eps;
  double r;  // 1/sqrt(1 - ps)
  F2 qi;     // 1/(4 (1 - ps))
};

__device__ __forceinline__ double opd_sq(double ps, double beta0_sq) {
  return fma(beta0_sq * ps, ps, fma(2.0, ps, 1.0));
}

// 1/sqrt(a) as y (1 + eps): the float reciprocal root refined by one
// third-order step, and half the residual 1 - a y^2; a outside [2^-100, 2^100]
// or not finite: the library call, eps 0.
__device__ __forceinline__ double rsqrt_split(double a, float& eps) {
  if (abs_hi(a) - (923u << 20) < (200u << 20) && a > 0.0) {
    const double f = f32_widen(rsqrtf(f2_split(a).h));  // 2^-22
    const double e = fma(-(a * f), f, 1.0);
    const double y = fma(f * e, fma(0.375, e, 0.5), f);
    const double p = a * y;
    eps = 0.5f * f2_split(fma(-fma(a, y, -p), y, fma(-p, y, 1.0))).h;
    return y;
  }
  eps = 0.f;
  return rsqrt(a);
}

// g0 without cancellation: (1+delta)^2 - (1 + beta0^2 ps)^2 = (1 - beta0^2) ps
// (2 + beta0^2 ps), so with v = that r0^2, g0 = 1 - sqrt(1 - v).  That holds
// for |ps| < 1/2, where (1+delta)^2 and 1 + beta0^2 ps are positive and r0 is
// below 2^27.  Other psigma (not finite ones among them, which a float pair
// cannot hold: f2_split only moves bits) get a g0 that map_drift refuses.
__device__ __noinline__ F2 slip_general(double d, double r0) {
  return f2_split(d * r0 * r0 / (1.0 + sqrt(1.0 - d * r0 * r0)));
}
__device__ __forceinline__ F2 slip(double ps, double beta0_sq, double r0) {
  if (abs_hi(ps) >= 0x3fe00000u) return F2{kNoSlip, 0.f};
  const double d = (1.0 - beta0_sq) * ps * fma(beta0_sq, ps, 2.0);
  const F2 v = f2_mul(f2_split(d), f2_sqr(f2_split(r0)));
  if (fabsf(v.h) < kSlipMaxV) return one_minus_sqrt1m(v);
  return slip_general(d, r0);
}

// r0 = 1/(1+delta) as y (1 + eps).  Where v = (1+delta)^2 - 1 = 2 ps + beta0^2
// ps^2 lies within 2^-7 of 0 (|ps| below 3.9e-3), r0 = 1 + ((1 + v)^(-1/2) - 1)
// with the bracket in float pairs (v to 2^-46 of itself: r0 to 2^-55) takes two
// FP64 instructions where the refined reciprocal root and its residual take
// fourteen (WIDE; float32 fields).  A stand-alone kick/push computes it for
// every particle: one cell of 4e6 particles on 256^2, split TF32, 1621 -> 1418
// us.  With a plan it is computed once per call and after RF cavities, and is
// called there (CALL): inlined, its code made a turn 1% slower that never ran
// it (called: 14.95 -> 14.88 ms).  Float64 fields keep the root: there either
// form spills more in the turn's kernel (18.0 -> 18.3 ms), and the two paths are
// to round alike.
struct InvDelta {
  double y;
  float eps;
};
__device__ __forceinline__ InvDelta inv_delta(double ps, double beta0_sq) {
  const F2 p = f2_split(ps);
  const F2 v = f2_add(f2_mul(f2_sqr(p), f2_split(beta0_sq)), F2{2.f * p.h, 2.f * p.l});
  InvDelta r;
  if (abs_hi(ps) < 0x3fe00000u && fabsf(v.h) < kSlopeMaxU) {
    const F2 c = rsqrt1m_wide(f2_neg(v));
    r.y = 1.0 + f2_to_double(c);
    const F2 rest = f2_add(c, f2_neg(f2_split(r.y - 1.0)));  // (relative to r0, which is 1 to 2^-8)
    r.eps = f_add(rest.h, rest.l);
  } else {
    r.y = rsqrt_split(opd_sq(ps, beta0_sq), r.eps);
  }
  return r;
}
__device__ __noinline__ InvDelta inv_delta_call(double ps, double beta0_sq) { return inv_delta(ps, beta0_sq); }

template <bool SERIES, bool WIDE, bool CALL>
__device__ __forceinline__ void ps_const(PsConst& k, double ps, double beta0_sq, bool quads) {
  k.eps = 0.f;
  if (SERIES) {
    if (WIDE) {
      const InvDelta r0 = CALL ? inv_delta_call(ps, beta0_sq) : inv_delta(ps, beta0_sq);
      k.d0 = r0.y;
      k.eps = r0.eps;
    } else {
      k.d0 = rsqrt_split(opd_sq(ps, beta0_sq), k.eps);
    }
    k.d1 = f2_pack(slip(ps, beta0_sq, k.d0));
  } else {
    k.d0 = opd_sq(ps, beta0_sq);
    k.d1 = fma(beta0_sq, ps, 1.0);
  }
  if (quads) {
    k.r = rsqrt(1.0 - ps);
    const F2 q = f2_sqr(f2_split(k.r));
    k.qi = F2{0.25f * q.h, 0.25f * q.l};
  } else {
    k.r = 0.0;
    k.qi = F2{0.f, 0.f};
  }
}

// What a segment's maps carry along beside the state: the momenta as float
// pairs while they are unchanged, and sg's change so far, added once at the end.
struct Carry {
  F2 px, py;
  bool split;  // px, py hold the state's momenta
  F2 r0, rr;   // r0 and r0^2 (series drift)
  bool has_rr;
  F2 sg;       // change of sg not yet added to the state
  bool has_sg;
};
__device__ __forceinline__ void carry_to_state(State& s, Carry& c) {
  if (c.has_sg) s.sg += f2_to_double(c.sg);
  c.sg = F2{0.f, 0.f};
  c.has_sg = false;
}

// Exact drift (Sec. III-A): with pz = sqrt((1+delta)^2 - px^2 - py^2),
// x += L px/pz, y += L py/pz, sg += L (1 - (1 + beta0^2 ps)/pz).
// Returns sg's change.
__device__ __forceinline__ double drift_general(State& s, double L, double opd2, double opb) {
  const double rpz = rsqrt(fma(-s.py, s.py, fma(-s.px, s.px, opd2)));
  const double Lr = L * rpz;
  s.x = fma(Lr, s.px, s.x);
  s.y = fma(Lr, s.py, s.y);
  return fma(-Lr, opb, L);
}

// The drift in a segment; e.p[0] = L, e.p[1] = L as an F2.
//
// SERIES: 1/pz = r0 (1 - u)^(-1/2) = r0 (1 + w), u = (px^2 + py^2) r0^2, with
// u and w (w is of the size of u, some 1e-7) in float pairs, so that the drift
// takes three FP64 instructions instead of twelve: L/pz = L d0 + (L d0 (w +
// eps)) and the two sums.  w is good to 2^-54, below the rounding of L/pz
// (which is rounded once; the general form rounds 1/pz and its product with L),
// and sg's change L (1 - (1 - g0)(1 + w)) = L (g0 - w + g0 w) to 2^-46 of g0 L, below
// the 2^-53 L the float64 form's cancellation leaves (kMaxSlip).  Momenta or u beyond
// the series (|p| >= 31 mrad), non-finite ones and psigma of a larger g0 or none
// (slip) take the general form; psp: where psigma is when the state does not hold it.
//
// Without SERIES: the general form throughout, sg's change carried as an F2 where
// it is as small.
template <bool SERIES>
__device__ __forceinline__ void map_drift(State& s, const DevElem& e, const PsConst& k, Carry& c, const double* psp,
                                          double beta0_sq) {
  if (SERIES) {
    if (!c.split) {
      c.px = f2_split(s.px);
      c.py = f2_split(s.py);
      c.split = true;
    }
    if (!c.has_rr) {
      c.r0 = f2_split(k.d0);
      c.rr = f2_sqr(c.r0);
      c.has_rr = true;
    }
    const F2 u = f2_mul(f2_add(f2_sqr(c.px), f2_sqr(c.py)), c.rr);
    const uint32_t m = max(abs_hi(s.px), abs_hi(s.py));
    const F2 g0 = f2_unpack(k.d1);
    if (m < 0x3fe00000u && u.h < kDriftMaxU && fabsf(g0.h) < kMaxSlip) {
      const F2 w = rsqrt1m_series(u), L = f2_unpack(e.p[1]);
      const F2 we{w.h, f_add(w.l, k.eps)};  // d0 (1 + w + eps) = r0 (1 + w) to 2^-64
      const double Lr = fma(e.p[0], k.d0, f2_to_double(f2_mul(f2_mul(L, c.r0), we)));
      s.x = fma(Lr, s.px, s.x);
      s.y = fma(Lr, s.py, s.y);
      const F2 q = f2_add(f2_add(g0, f2_neg(w)), f2_mul(g0, w));
      if (fabsf(c.sg.h) > kMaxCarry * L.h) carry_to_state(s, c);
      c.sg = f2_add(c.sg, f2_mul(q, L));
      c.has_sg = true;
    } else {
      const double ps = psp ? *psp : s.ps;
      s.sg += drift_general(s, e.p[0], opd_sq(ps, beta0_sq), fma(beta0_sq, ps, 1.0));
    }
  } else {
    const double d = drift_general(s, e.p[0], k.d0, k.d1);
    const double L = e.p[0];
    if (abs_hi(d) < kHi2p50 && abs_hi(d) + (9u << 20) < abs_hi(L)) {  // 2^-9 L (kMaxSlip)
      if (fabsf(c.sg.h) > kMaxCarry * f2_unpack(e.p[1]).h) carry_to_state(s, c);
      c.sg = f2_add(c.sg, f2_split(d));
      c.has_sg = true;
    } else {
      s.sg += d;
    }
  }
}

// Thick quadrupole (Sec. III-B) for H_approx with K1 = k1:
//   w = sqrt(|k1| (1-ps)), a = sqrt((1-ps)/|k1|) = s1/sqk, bq = sqrt(|k1|/(1-ps)) = sqk r
//   focusing plane:   u = u0 cos wL + a pu0 sin wL,  pu = pu0 cos wL - bq u0 sin wL
//   defocusing plane: u = u0 cosh wL + a pu0 sinh wL, pu = pu0 cosh wL + bq u0 sinh wL
// wL = theta0 s1 = theta0 + Delta, theta0 = sqk L; cos/sin/cosh/sinh of
// theta0 come from the host, those of the small Delta from their Taylor
// series, combined by the addition theorems.
// sg: d sg/ds = ps/gamma0^2 - (px^2+py^2)/2.  Each plane conserves
// h_u = ((1-ps) pu^2 + k_u u^2)/2 (k_x = k1, k_y = -k1) and
// d(u pu)/ds = (1-ps) pu^2 - k_u u^2, so
//   int_0^L pu^2 ds = (h_u L + [u pu]_0^L / 2) / (1-ps),
// which gives sg += ps L/gamma0^2 - (L S2 + D) / (4 (1-ps)) with
// S2 = (1-ps)(px0^2+py0^2) + k1 (x0^2 - y0^2), D = [x px + y py]_0^L, i.e.
//   sg += ps L/gamma0^2 - (L/4)(px0^2+py0^2) - (L k1 (x0^2-y0^2) + D) / (4 (1-ps)),
// in float pairs (quad_slip: some 1e-6 of a metre, good to 2^-42 of itself; kMaxSlip).
// e.p = {L/4, L/gamma0^2, cos theta0, sin theta0, cosh theta0, sinh theta0, sqk, 1/sqk, L k1,
//        then L/4, L/gamma0^2 and L k1 as F2}
// (theta0 = sqk L = sqk (4 e.p[0]), the host's product bit for bit), e.flags =
// QF_* (plus the family bits); a zero-gradient quadrupole (QF_ZERO) has e.p[0] = L.
//
// The entries of the two planes' 2x2 matrices depend on ps alone (QuadCoef:
// u = cu u0 + sua pu0, pu = cu pu0 + sub u0), so a turn's tracking keeps them
// per particle and quadrupole family (computed where psc is, read by the map).
struct QuadCoef {
  double cx, sxa, sxb, cy, sya, syb;
};

__device__ __forceinline__ QuadCoef quad_coef(const DevElem& e, double ps, double r) {
  const double s1 = (1.0 - ps) * r;  // sqrt(1 - ps)
  const double th0 = e.p[6] * (4.0 * e.p[0]);
  const double delta = fma(th0, s1, -th0);
  double c, sn, ch, sh;
  if (fabs(delta) <= kMaxDelta) {
    const double d2 = delta * delta;
    const double sd = fma(delta, fma(d2, 1.0 / 120.0, -1.0 / 6.0) * d2, delta);   // sin(delta)
    const double cm = fma(d2, 1.0 / 24.0, -0.5) * d2;                             // cos(delta) - 1
    const double shd = fma(delta, fma(d2, 1.0 / 120.0, 1.0 / 6.0) * d2, delta);   // sinh(delta)
    const double chm = fma(d2, 1.0 / 24.0, 0.5) * d2;                             // cosh(delta) - 1
    const double c0 = e.p[2], s0 = e.p[3], ch0 = e.p[4], sh0 = e.p[5];
    c = fma(-s0, sd, fma(c0, cm, c0));
    sn = fma(c0, sd, fma(s0, cm, s0));
    ch = fma(sh0, shd, fma(ch0, chm, ch0));
    sh = fma(ch0, shd, fma(sh0, chm, sh0));
  } else {
    const double th = th0 * s1;
    sincos(th, &sn, &c);
    ch = cosh(th);
    sh = sinh(th);
  }
  const double a = s1 * e.p[7];
  const double bq = e.p[6] * r;
  // focusing plane on trig (c, sn), defocusing on hyperbolic (ch, sh)
  if ((e.flags & QF_KIND) == QF_FOCUS_X) return QuadCoef{c, a * sn, -bq * sn, ch, a * sh, bq * sh};
  return QuadCoef{ch, a * sh, bq * sh, c, a * sn, -bq * sn};
}

// sg's change in float64, for states quad_slip's floats cannot hold or are too short for.
__device__ __forceinline__ void quad_slip_slow(State& s, const DevElem& e, double x0, double px0, double y0, double py0) {
  const double xy = fma(x0, x0, -y0 * y0);
  const double pp = fma(px0, px0, py0 * py0);
  // L k1 (x0^2 - y0^2) + D, D = x px + y py - x0 px0 - y0 py0
  const double u = fma(e.p[8], xy, fma(-y0, py0, fma(-x0, px0, fma(s.x, s.px, s.y * s.py))));
  s.sg = fma(-u, 0.25 / (1.0 - s.ps), fma(-e.p[0], pp, fma(s.ps, e.p[1], s.sg)));
}

__device__ __forceinline__ void quad_apply(State& s, const DevElem& e, const QuadCoef& q, const PsConst& k, Carry& c) {
  const double x0 = s.x, px0 = s.px, y0 = s.y, py0 = s.py;
  s.x = fma(q.cx, x0, q.sxa * px0);
  s.px = fma(q.cx, px0, q.sxb * x0);
  s.y = fma(q.cy, y0, q.sya * py0);
  s.py = fma(q.cy, py0, q.syb * y0);
  const F2 p0 = c.split ? c.px : f2_split(px0), q0 = c.split ? c.py : f2_split(py0);
  c.px = f2_split(s.px);
  c.py = f2_split(s.py);
  c.split = true;
  const F2 a0 = f2_split(x0), b0 = f2_split(y0), a1 = f2_split(s.x), b1 = f2_split(s.y), ps = f2_split(s.ps);
  const F2 L4 = f2_unpack(e.p[9]), Lg = f2_unpack(e.p[10]), K = f2_unpack(e.p[11]);
  const float size = quad_slip_size(a0, p0, b0, q0, a1, c.px, b1, c.py, ps, k.qi, L4, Lg, K);
  const F2 d = quad_slip(a0, p0, b0, q0, a1, c.px, b1, c.py, ps, k.qi, L4, Lg, K);
  const uint32_t m = max(max(max(abs_hi(x0), abs_hi(px0)), max(abs_hi(y0), abs_hi(py0))),
                         max(max(abs_hi(s.x), abs_hi(s.px)), max(max(abs_hi(s.y), abs_hi(s.py)), abs_hi(s.ps))));
  if (m < kHi2p50 && size < 4.f * kMaxSlip * L4.h) {  // (L4 = L/4)
    c.sg = f2_add(c.sg, d);
    c.has_sg = true;
  } else {
    quad_slip_slow(s, e, x0, px0, y0, py0);
  }
}

__device__ __forceinline__ void map_quad(State& s, const DevElem& e, const PsConst& k, double inv_gamma0_sq,
                                         Carry& c) {
  if ((e.flags & QF_KIND) == QF_ZERO) {  // flow of H0: straight line with the chromatic factor
    const double L = e.p[0];
    const double f = (1.0 - s.ps) * L;
    const double pp = fma(s.px, s.px, s.py * s.py);
    s.x = fma(f, s.px, s.x);
    s.y = fma(f, s.py, s.y);
    s.sg = fma(-0.5 * L, pp, fma(s.ps, L * inv_gamma0_sq, s.sg));
    return;
  }
  quad_apply(s, e, quad_coef(e, s.ps, k.r), k, c);
}

// The map with the particle's cached coefficients: qc points at its entry of
// the family's six arrays of n (cx, sxa, sxb, cy, sya, syb).
__device__ __forceinline__ void map_quad_cached(State& s, const DevElem& e, const double* __restrict__ qc, size_t n,
                                                const PsConst& k, Carry& c) {
  const QuadCoef q{qc[0], qc[n], qc[2 * n], qc[3 * n], qc[4 * n], qc[5 * n]};
  quad_apply(s, e, q, k, c);
}

// Flow of H0 = (px^2+py^2)/2 (1-ps) + ps^2/(2 gamma0^2) over l.
__device__ __forceinline__ void h0_flow(State& s, const PsConst& k, double l, double inv_gamma0_sq) {
  const double f = (1.0 - s.ps) * l;
  const double pp = fma(s.px, s.px, s.py * s.py);
  s.x = fma(f, s.px, s.x);
  s.y = fma(f, s.py, s.y);
  s.sg = fma(-0.5 * l, pp, fma(s.ps, l * inv_gamma0_sq, s.sg));
}

// Sextupole (Sec. III-C).  Thin: the V step of Eq. Sym2 as one kick,
// px -= k2l/2 (x^2 - y^2), py += k2l x y; e.p = {k2l/2, k2l}.  Thick
// (e.flags = 1): Eq. Sym2, H0 flows of a L, c L, a L around two kicks of
// integrated strength k2l/2; e.p = {k2l/4, k2l/2, a L, c L}.
__device__ __forceinline__ void sext_kick(State& s, double half, double full) {
  s.px = fma(-half, (s.x - s.y) * (s.x + s.y), s.px);
  s.py = fma(full * s.x, s.y, s.py);
}

// (Thick elements and the exact dipole are not inlined: their registers stay
// out of the hot kernels' allocation.)
__device__ __noinline__ void map_sext_thick(State& s, const DevElem& e, const PsConst& k, double inv_gamma0_sq) {
  h0_flow(s, k, e.p[2], inv_gamma0_sq);
  sext_kick(s, e.p[0], e.p[1]);
  h0_flow(s, k, e.p[3], inv_gamma0_sq);
  sext_kick(s, e.p[0], e.p[1]);
  h0_flow(s, k, e.p[2], inv_gamma0_sq);
}

__device__ __forceinline__ void map_sext(State& s, const DevElem& e, const PsConst& k, double inv_gamma0_sq) {
  if (e.flags != 1)
    sext_kick(s, e.p[0], e.p[1]);
  else
    map_sext_thick(s, e, k, inv_gamma0_sq);
}

// Exact sector dipole (Sec. III-A, uniform field without H_approx): the
// particle's circle in the bending plane carried to the exit face.  With
// P^2 = (1+delta)^2 - py^2, pz0 = sqrt(P^2 - px0^2), C = cos(angle), S = sin(angle):
//   px = px0 C + (pz0 - 1 - x0/rho) S,  pz = sqrt(P^2 - px^2),
//   x = (x0 + rho (1 - pz0)) C + rho px0 S + rho (pz - 1),
//   alpha = angle + asin(px0/P) - asin(px/P),
//   y += py rho alpha,  sg += L - (1 + beta0^2 ps) rho alpha.
// e.p = {L, angle, C, S, rho, 1/rho}; zero angle (e.flags = 1): the exact drift.
__device__ __noinline__ void map_exact_bend(State& s, const DevElem& e, double beta0_sq) {
  if (e.flags == 1) {
    s.sg += drift_general(s, e.p[0], opd_sq(s.ps, beta0_sq), fma(beta0_sq, s.ps, 1.0));
    return;
  }
  const double L = e.p[0], angle = e.p[1], C = e.p[2], S = e.p[3], rho = e.p[4], h = e.p[5];
  const double x0 = s.x, px0 = s.px;
  const double P2 = fma(-s.py, s.py, opd_sq(s.ps, beta0_sq));
  const double pz0 = sqrt(fma(-px0, px0, P2));
  const double px = fma(px0, C, (pz0 - 1.0 - x0 * h) * S);
  const double pz = sqrt(fma(-px, px, P2));
  const double rP = rsqrt(P2);
  const double alpha = angle + (asin(px0 * rP) - asin(px * rP));
  s.x = fma(x0 + rho * (1.0 - pz0), C, fma(rho * px0, S, rho * (pz - 1.0)));
  s.px = px;
  s.y = fma(s.py * rho, alpha, s.y);
  s.sg += fma(-fma(beta0_sq, s.ps, 1.0) * rho, alpha, L);
}

// Linear sector dipole from H_approx with curvature h (Sec. III, Eq. H plus
// the bending field's h^2 x^2 / 2):
//   x = C x0 + (S/h) px0 + ((1-C)/h) ps,  px = -hS x0 + C px0 + S ps,
//   y += L py, sg += ps L/gamma0^2 - (S x0 + ((1-C)/h) px0 + (L - S/h) ps).
// e.p = {L, C, S, S/h, (1-C)/h, h S, L - S/h}; angle 0: e.flags = 1 (H0 flow).
__device__ __forceinline__ void map_bend(State& s, const DevElem& e, const PsConst& k, double inv_gamma0_sq) {
  const double L = e.p[0];
  if (e.flags == 1) {
    const double f = (1.0 - s.ps) * L;
    const double pp = fma(s.px, s.px, s.py * s.py);
    s.x = fma(f, s.px, s.x);
    s.y = fma(f, s.py, s.y);
    s.sg = fma(-0.5 * L, pp, fma(s.ps, L * inv_gamma0_sq, s.sg));
    return;
  }
  const double C = e.p[1], S = e.p[2], Soh = e.p[3], Cm = e.p[4], hS = e.p[5], LS = e.p[6];
  const double x0 = s.x, px0 = s.px, ps = s.ps;
  s.x = fma(C, x0, fma(Soh, px0, Cm * ps));
  s.px = fma(-hS, x0, fma(C, px0, S * ps));
  s.y = fma(L, s.py, s.y);
  s.sg = fma(ps, L * inv_gamma0_sq, s.sg) - fma(S, x0, fma(Cm, px0, LS * ps));
}

// Thin RF cavity: ps += V/(beta0^2 E0) sin(lag - 2 pi h sg / C).
// e.p = {V/(beta0^2 E0), 2 pi h / C, lag}.
__device__ __forceinline__ void map_rf(State& s, const DevElem& e) {
  s.ps = fma(e.p[0], sin(fma(-e.p[1], s.sg, e.p[2])), s.ps);
}

// Push through n_elem elements with the ps-dependent quantities k (valid on
// entry).  quads: refresh k's square roots after an RF cavity.  Returns true
// when an RF cavity changed ps (k then holds the new values).  qc: the
// particle's entry in the quadrupole coefficient cache (arrays of n), valid
// until an RF cavity; NULL: none.  psp: where the particle's psigma is when
// the state does not hold it (segments of drifts and thin sextupoles), else
// NULL.  XE: the segment may hold thick sextupoles or exact dipoles (their
// code is compiled only into the kernels that need it, keeping the common
// kernels' registers).  SERIES: which drift (and which d0, d1 of k); WIDE: see
// ps_const.
template <bool XE, bool SERIES, bool WIDE>
__device__ __forceinline__ bool push_elements(State& s, PsConst& k, const DevElem* __restrict__ el, int n_elem,
                                              double beta0_sq, double inv_gamma0_sq, bool quads,
                                              const double* __restrict__ qc, size_t n, const double* psp) {
  bool changed = false;
  Carry c;
  c.split = c.has_rr = c.has_sg = false;
  c.px = c.py = c.r0 = c.rr = c.sg = F2{0.f, 0.f};
#pragma unroll 1
  for (int i = 0; i < n_elem; ++i) {
    const DevElem& e = el[i];
    switch (e.type) {
      case SC_DRIFT: map_drift<SERIES>(s, e, k, c, psp, beta0_sq); break;
      case SC_QUAD: {
        const int fam = e.flags >> QF_FAM_SHIFT;
        if (qc && fam && !changed)
          map_quad_cached(s, e, qc + (size_t)(fam - 1) * 6 * n, n, k, c);
        else
          map_quad(s, e, k, inv_gamma0_sq, c);
        break;
      }
      case SC_SEXT:
        if (XE)
          map_sext(s, e, k, inv_gamma0_sq);
        else
          sext_kick(s, e.p[0], e.p[1]);
        c.split = false;
        break;
      case SC_BEND:
        map_bend(s, e, k, inv_gamma0_sq);
        c.split = false;
        break;
      case SC_EXACT_BEND:
        if (XE) map_exact_bend(s, e, beta0_sq);
        c.split = false;
        break;
      case SC_RF:
        carry_to_state(s, c);  // the cavity reads sg
        c.has_rr = false;
        map_rf(s, e);
        ps_const<SERIES, WIDE, true>(k, s.ps, beta0_sq, quads);
        changed = true;
        break;
      default: break;
    }
  }
  if (c.has_sg) s.sg += f2_to_double(c.sg);
  return changed;
}

}  // namespace sc
