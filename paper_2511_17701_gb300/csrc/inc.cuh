// inc.cuh -- the FP64 pusher's increment form (plain log-r grid): the pieces that the particle
// kernel (push_inc.cuh) and the adjoint (adjoint.cu) are made of, for pairs of floats (DF) and,
// where a derivative is taken, for pairs with two derivatives (D2F).
//
// GB300 executes 2 FP64 operations per clock and SM against 128 FP32 ones, and the FP64
// routine (push64) needs ~560 of them per particle. But everything a step computes for the
// momentum ends in an increment that is mostly a small part of u: u^{n+1} = u^n + du. An
// increment of at most 2^-5 of |u|, computed in pairs of floats (dfloat.cuh, relative error
// ~2^-48), leaves an error of 2^-53 in u, below what the FP64 routine's own rounding leaves
// (3e-16 of |u| rms). So the metric and its derivatives at x^n, the tetrads, the field
// interpolation, both Boris half steps and the geodesic substep are evaluated in float pairs, as
// increments, and u^n + du is formed in FP64 by one addition per component. The coordinate
// substep is not small against the offset it changes: its result is, as in push64, one FP64
// evaluation of the map at the predictor's point.
//
// A half step or a geodesic substep that changes the momentum by more than INC_MAX of it (strong
// fields, cold particles, the rows on the axes) is taken in FP64, the rest as above. A particle
// that the bounds behind this do not cover (an iteration that the predictor does not resolve,
// values outside the range of FP32) is left to push64, untouched.
//
// Measured: a step of the 2048^2 workload (134 M particles) 173.6 -> 70.5 ms, of the 512^2 one
// (16.8 M) 21.0 -> 9.8 ms. One push against 80-bit arithmetic, 20,000 particles with |u| = 1, the
// iterations run to rounding: rms errors of |u| 1.1e-16 on 64^2, 5.8e-17 on 512^2 (push64:
// 3.6e-16 on both), of the offsets 2.6e-17 to 3.6e-17 (2.8e-17 to 4.3e-17).
#pragma once
#include "dual_df.cuh"
#include "refine.cuh"

namespace {

// The largest |increment| / |u| of a Boris half step or the geodesic substep that pairs take: 2^-5
// of a relative error of about 2^-48 is 2^-53 of u. Measured, |u| = 0.1 on 64^2 in a field that
// kicks most particles by about that: 3.9e-16 of |u| rms, 2.3e-15 at most (the FP64 routine with
// its iterations run to rounding: 3.7e-16, 1.2e-15); |u| = 1e-3:
// 5.3e-16 and 5.7e-15 (5.4e-16, 6.2e-15).
// Massless particles, whose FP64 push rounds less (no half steps: 6.9e-17), take half of it.
constexpr float INC_MAX = 0x1p-5f;
// below this, squared, the pairs' own floor of 2^-149 would show in an increment that is not
// exactly zero
constexpr float INC_UU = 0x1p-100f;
// whether an increment of square dd is within sqrt(times2) INC_MAX of a momentum of square uu
__device__ __forceinline__ bool inc_within(float times2, float dd, float uu) {
  return dd <= times2 * (INC_MAX * INC_MAX) * uu && uu >= INC_UU;
}
constexpr float INC_E = 0.055f;      // largest |offset of xi| of the radial series
constexpr float INC_D = 0.035f;      // largest |offset of theta| of the angular series
constexpr int INC_ROWS = 64;          // rows from either axis with theta as map_theta rounds it
constexpr float INC_R = 1024.0f;     // largest r: the metric's smallest products, ~ r^-6 dxi^-2, keep
                                     // their low parts in FP32's range

__device__ __forceinline__ DF df2(const float2 v) { return DF(v.x, v.y); }

// The grid's constants in pairs that the increment form reads
struct IncC {
  DF a, M, dxi, dth, ig2, dt, a2;
};
__device__ __forceinline__ IncC inc_c(const GridP &g) {
  return {DF(g.d_a[0], g.d_a[1]),     DF(g.d_M[0], g.d_M[1]),   DF(g.d_dxi[0], g.d_dxi[1]),
          DF(g.d_dth[0], g.d_dth[1]), DF(g.d_ig2[0], g.d_ig2[1]), DF(g.d_dt[0], g.d_dt[1]),
          DF(g.d_a2[0], g.d_a2[1])};
}

// r, sin(theta), cos(theta) in pairs at x1 = i + o1, x2 = j + o2 from the tables of the
// nearest cell corner (rows' corner j + c2, d: theta's offset from it). The series' leading
// terms are pairs, their tails (below 2^-24 of the result's last bit but one) plain floats.
// Returns whether the offsets are in range.
__device__ __forceinline__ bool inc_point_d(const IncC &k, const PushTables &tb, int i, int j,
                                            DF o1, DF o2, int c2, DF d, DF &r, DF &s, DF &c) {
  const int c1 = o1.hi >= 0.5f;
  const DF q1 = fast_two_sum(__fsub_rn(o1.hi, (float)c1), o1.lo);
  const DF e = q1 * k.dxi;
  const float ef = e.hi;
  // exp(e) = 1 + e + e^2/2 + e^3/6 + e^4 (1/24 + ...)
  float t = fmaf(1.0f / 40320.0f, ef, 1.0f / 5040.0f);
  t = fmaf(t, ef, 1.0f / 720.0f);
  t = fmaf(t, ef, 1.0f / 120.0f);
  DF x = dfc(1.0 / 24.0) + DF(t * ef);
  x = fma_(x, e, dfc(1.0 / 6.0));
  x = fma_(x, e, DF(0.5f));
  x = fma_(x, e, DF(1.0f));
  x = fma_(x, e, DF(1.0f));
  r = df2(__ldg(tb.r_df + i + c1 + G_)) * x;
  const DF q = d * d;
  const float qf = q.hi;
  t = fmaf(1.0f / 362880.0f, qf, -1.0f / 5040.0f);
  t = fmaf(t, qf, 1.0f / 120.0f);
  const DF se = fma_((dfc(-1.0 / 6.0) + DF(t * qf)) * q, d, d);  // sin(d)
  t = fmaf(1.0f / 40320.0f, qf, -1.0f / 720.0f);
  t = fmaf(t, qf, 1.0f / 24.0f);
  const DF ce = fma_(DF(-0.5f) + DF(t * qf), q, DF(1.0f));  // cos(d)
  const DF s0 = df2(__ldg(tb.s_df + j + c2 + G_)), c0 = df2(__ldg(tb.c_df + j + c2 + G_));
  s = fma_(s0, ce, c0 * se);
  c = fma_(c0, ce, -(s0 * se));
  return fabsf(ef) <= INC_E && fabsf(d.hi) <= INC_D && o1.hi >= 0.0f && o1.hi <= 1.0f &&
         o2.hi >= 0.0f && o2.hi <= 1.0f && r.hi <= INC_R;
}

__device__ __forceinline__ bool inc_point(const IncC &k, const PushTables &tb, int i, int j, DF o1,
                                          DF o2, DF &r, DF &s, DF &c) {
  const int c2 = o2.hi >= 0.5f;
  const DF q2 = fast_two_sum(__fsub_rn(o2.hi, (float)c2), o2.lo);
  return inc_point_d(k, tb, i, j, o1, o2, c2, q2 * k.dth, r, s, c);
}
// At x^n = (i + dx1, j + dx2): in the rows near the axes theta is formed as map_theta forms it
// (x2 dtheta, rounded) and its offset from the corner's exact. Next to theta = pi that rounding
// is a relative 2e-16 / (pi - theta) of sin(theta), which the momentum's increments, of order u
// there, would show at ~1e-12 if it were formed in another way.
__device__ __forceinline__ bool inc_point_n(const GridP &g, const IncC &k, const PushTables &tb,
                                            int i, int j, double dx2, DF o1, DF o2, DF &r, DF &s,
                                            DF &c) {
  const int c2 = o2.hi >= 0.5f;
  DF d;
  if (j < INC_ROWS || j >= g.n_th - INC_ROWS) {
    d = df_of(__dmul_rn(__dadd_rn((double)j, dx2), g.dth) - __ldg(tb.th64 + j + c2 + G_));
  } else {
    d = fast_two_sum(__fsub_rn(o2.hi, (float)c2), o2.lo) * k.dth;
  }
  return inc_point_d(k, tb, i, j, o1, o2, c2, d, r, s, c);
}

// Metric, its derivatives and the tetrad coefficients at x^n in pairs: the quantities of
// local_full, written so that each takes few operations (one reciprocal, three reciprocal
// square roots: of Sigma, Sigma + 2 M r and A).
template <typename R>
__device__ __forceinline__ void inc_local(const IncC &k, R r, R s, R c, Local<R> &L) {
  const R s2 = s * s, r2 = r * r, f = k.dxi * r, sc = s * c;
  const R Sig = fma_(k.a2, c * c, r2);
  const R Mr = k.M * r, M2r = df_scale(Mr, 2.0f);
  const R S2 = Sig + M2r;
  const R Rr = r2 + k.a2, Del = Rr - M2r, as2 = k.a2 * s2;
  const R A = fma_(Rr, Rr, -(as2 * Del));
  const R P = Sig * S2, Pf = P * f;
  const R iQ = df_rcp(Pf * s2);
  const R iu = iQ * s2, is2 = iQ * Pf;
  const R iP = iu * f, fi = iu * P;
  const R iSig = iP * S2, iS2 = iP * Sig;
  const R rSig = df_rsqrt(Sig), rS2 = df_rsqrt(S2), rA = df_rsqrt(A);
  const R qSig = Sig * rSig, qS2 = S2 * rS2;
  Geo<R> &o = L.G;
  const R fi2 = fi * fi, AP = A * iP;
  o.opz = S2 * iSig;
  o.H11 = AP * fi2;
  o.H13 = k.a * iSig * fi;
  o.H22 = iSig * k.ig2;
  o.H33 = iSig * is2;
  o.beta1 = M2r * iS2 * fi;
  L.alpha = qSig * rS2;
  const R dxS = df_scale(r * f, 2.0f), a2sc = k.a2 * sc * k.dth, deS = df_scale(a2sc, -2.0f);
  const R qS = dxS * iSig, qe = deS * iSig, Mf = k.M * f;
  const R ipf = iP * fi2;
  // d(A)/dx1 = 2 f (2 r R - a^2 s^2 (r - M)), d(P)/dx1 = dxS S2 + Sigma (dxS + 2 M f)
  const R dxA = df_scale(f * fma_(df_scale(r, 2.0f), Rr, -(as2 * (r - k.M))), 2.0f);
  const R dxP = fma_(dxS, S2, Sig * (dxS + df_scale(Mf, 2.0f)));
  L.d1H11 = fma_(ipf, dxA - AP * dxP, -(df_scale(k.dxi, 2.0f) * o.H11));
  L.d2H11 = ipf * deS * (Del - AP * (S2 + Sig));
  L.d1H22 = -(qS * o.H22);
  L.d2H22 = -(qe * o.H22);
  L.d1H33 = -(qS * o.H33);
  L.d2H33 = -((qe + df_scale(sc * is2 * k.dth, 2.0f)) * o.H33);
  L.d1H13 = -((qS + k.dxi) * o.H13);
  L.d2H13 = -(qe * o.H13);
  const R fsr = fma_(f, Sig, -(r * dxS)), rde = Mr * deS;
  const R ia = iP * L.alpha;
  L.d1alpha = -(k.M * fsr * ia);
  L.d2alpha = rde * ia;
  const R w = df_scale(fi * iS2 * iS2, 2.0f);
  L.d1beta1 = fma_(w * k.M, fsr, -(k.dxi * o.beta1));
  L.d2beta1 = -(w * rde);
  L.rH11 = f * qSig * qS2 * rA;
  L.sH11 = fi * (rSig * rS2) * (A * rA);
  L.rh22 = rSig * (k.ig2 * k.dth);
  L.sh22 = qSig * k.dth;
  const R sA = s * rSig;
  L.rh33 = qSig * rA * (s * is2);
  L.sh33 = sA * (A * rA);
  const R faS = f * k.a * S2;
  L.k13 = -(faS * sA * rA);
  L.m13 = -(faS * (rA * rA));
}

// The geodesic substep as a map of the increment d = t - u: the same equation as GeoMap,
// d -> G(u + d) - u. R: DF or float (the predictor, from the pairs' high parts).
template <typename R>
struct GeoInc {
  R u0, u1, c0, c1, e1, e2, f1, f2, D1a, D1b, D2a, D2b, hdt;
  R H11, H22, d1H11, d1H22, d2H11, d2H22;
};
__device__ __forceinline__ float half_(float a) { return 0.5f * a; }
__device__ __forceinline__ DF half_(DF a) { return df_scale(a, 0.5f); }
__device__ __forceinline__ float twice_(float a) { return 2.0f * a; }
__device__ __forceinline__ DF twice_(DF a) { return df_scale(a, 2.0f); }
template <typename R, typename D>
__device__ __forceinline__ void geo_inc_apply(const GeoInc<R> &m, D d0, D d1, R &n0, R &n1) {
  const R b0 = m.u0 + half_(d0), b1 = m.u1 + half_(d1);
  const R b1s = b1 * b1;
  const R q = fma_(b0, fma_(m.H11, b0, m.c1), fma_(m.H22, b1s, m.c0));  // gamma_bar^2
  const R ig = rsqrt_(q);
  const R gb = q * ig, ha = m.hdt * ig;
  const R k1 = fma_(b0, fma_(m.d1H11, b0, m.e2), fma_(m.d1H22, b1s, m.e1));
  const R k2 = fma_(b0, fma_(m.d2H11, b0, m.f2), fma_(m.d2H22, b1s, m.f1));
  n0 = fma_(b0, m.D1b, -fma_(gb, m.D1a, ha * k1));
  n1 = fma_(b0, m.D2b, -fma_(gb, m.D2a, ha * k2));
}
// A = d(map)/d(increment) (GeoMap::jacobian in b = u + d/2); the map depends on u_1, u_2 and d
// through b alone, so its derivative with respect to u_1, u_2 is 2 A
template <typename R>
__device__ __forceinline__ void geo_inc_jacobian(const GeoInc<R> &m, R d0, R d1, R J[2][2]) {
  const R b0 = m.u0 + half_(d0), b1 = m.u1 + half_(d1), b1s = b1 * b1;
  const R h11b = m.H11 * b0, h22b = m.H22 * b1;
  const R q = fma_(b0, h11b + m.c1, fma_(h22b, b1, m.c0));
  const R ig = rsqrt_(q), ha = m.hdt * ig;
  const R k1 = fma_(b0, fma_(m.d1H11, b0, m.e2), fma_(m.d1H22, b1s, m.e1));
  const R k2 = fma_(b0, fma_(m.d2H11, b0, m.f2), fma_(m.d2H22, b1s, m.f1));
  const R q0 = h11b + half_(m.c1);                   // half of dq/db
  const R hh = -(ha * ig * ig);                      // d(ha) = hh (q0 db0 + h22b db1)
  const R g0 = ig * q0, g1 = ig * h22b, a0 = hh * q0, a1 = hh * h22b;
  J[0][0] = half_(m.D1b - fma_(g0, m.D1a, fma_(a0, k1, ha * (twice_(m.d1H11 * b0) + m.e2))));
  J[0][1] = -half_(fma_(g1, m.D1a, fma_(a1, k1, ha * twice_(m.d1H22 * b1))));
  J[1][0] = half_(m.D2b - fma_(g0, m.D2a, fma_(a0, k2, ha * (twice_(m.d2H11 * b0) + m.f2))));
  J[1][1] = -half_(fma_(g1, m.D2a, fma_(a1, k2, ha * twice_(m.d2H22 * b1))));
}
// the map's derivative by u_3 (through c0, c1, e1, e2, f1, f2 of geo_inc_setup)
__device__ __forceinline__ void geo_inc_d3(const Local<DF> &L, const GeoInc<DF> &m, DF u3, DF d0,
                                           DF d1, DF d[2]) {
  const DF b0 = m.u0 + half_(d0), b1 = m.u1 + half_(d1), b1s = b1 * b1;
  const DF q = fma_(b0, fma_(m.H11, b0, m.c1), fma_(m.H22, b1s, m.c0));
  const DF ig = rsqrt_(q), ha = m.hdt * ig;
  const DF k1 = fma_(b0, fma_(m.d1H11, b0, m.e2), fma_(m.d1H22, b1s, m.e1));
  const DF k2 = fma_(b0, fma_(m.d2H11, b0, m.f2), fma_(m.d2H22, b1s, m.f1));
  const DF dq = fma_(L.G.H33, u3, L.G.H13 * b0);        // half of dq/du_3
  const DF dg = ig * dq, dh = -(ha * ig * ig * dq);      // of gamma_bar, ha
  const DF g1 = twice_(fma_(L.d1H33, u3, L.d1H13 * b0));
  const DF g2 = twice_(fma_(L.d2H33, u3, L.d2H13 * b0));
  d[0] = -fma_(dg, m.D1a, fma_(dh, k1, ha * g1));
  d[1] = -fma_(dg, m.D2a, fma_(dh, k2, ha * g2));
}
// whether the method's n_iter iterations come within a tenth of tol of the fixed point
// (method_converges on FP32 values)
__device__ __forceinline__ bool inc_converges(float d1, const float J[2][2], int n_iter, float tol,
                                              float scale) {
  const float rho = spectral_radius(J);
  if (!(rho < 0.25f)) return false;
  return !(rho > 0.0f) ||
         d1 * exp2f((float)n_iter * log2f(rho)) <= 0.1f * tol * fmaxf(1.0f, scale);
}

// the map's coefficients for metric values of type M and a momentum of type R
template <typename M, typename R>
__device__ __forceinline__ void geo_inc_setup(const IncC &k, const Local<M> &L, const R u[3],
                                              float m2, GeoInc<R> &m) {
  const R uu = u[2] * u[2], u2x2 = df_scale(u[2], 2.0f);
  const Geo<M> &o = L.G;
  m.u0 = u[0];
  m.u1 = u[1];
  m.c0 = fma_(o.H33, uu, R(m2));
  m.c1 = o.H13 * u2x2;
  m.e1 = L.d1H33 * uu;
  m.e2 = L.d1H13 * u2x2;
  m.f1 = L.d2H33 * uu;
  m.f2 = L.d2H13 * u2x2;
  m.D1a = R(k.dt * L.d1alpha);
  m.D1b = R(k.dt * L.d1beta1);
  m.D2a = R(k.dt * L.d2alpha);
  m.D2b = R(k.dt * L.d2beta1);
  m.hdt = R(df_scale(k.dt * L.alpha, 0.5f));
  m.H11 = R(o.H11);
  m.H22 = R(o.H22);
  m.d1H11 = R(L.d1H11);
  m.d1H22 = R(L.d1H22);
  m.d2H11 = R(L.d2H11);
  m.d2H22 = R(L.d2H22);
}

// The fixed point (n0, n1) of the map. The FP32 map gives the increment to FP32 rounding, one
// evaluation in pairs there and one Newton step with the FP32 Jacobian J, d + (I - J)^{-1} r =
// G + M J r with r = G - d and M = (I - J)^{-1}, leave an error of |J| 2^-24 |r|, far below the
// pairs' rounding of d. n_iter, tol: the method's iterations and what they have to come within
// (inc_converges), else the method's iterations themselves are run, in pairs (LITERAL). h33:
// h^33 u_3^2. Returns GEO_SMALL; GEO_LARGE where the increment is beyond the bound, and the point
// (n0, n1), within the pairs' rounding of the fixed point, that FP64 evaluations have to start
// from, with the contraction rho there; GEO_NONE: not resolved.
enum { GEO_NONE = 0, GEO_SMALL, GEO_LARGE };
template <bool LITERAL>
__device__ __forceinline__ int geo_inc_solve(const GeoInc<DF> &m, float h33, int n_iter, float tol,
                                             float times2, DF &n0, DF &n1, float &rho) {
  const GeoInc<float> mf = {m.u0.hi,  m.u1.hi,  m.c0.hi,  m.c1.hi,  m.e1.hi,    m.e2.hi,   m.f1.hi,
                            m.f2.hi,  m.D1a.hi, m.D1b.hi, m.D2a.hi, m.D2b.hi,   m.hdt.hi,  m.H11.hi,
                            m.H22.hi, m.d1H11.hi, m.d1H22.hi, m.d2H11.hi, m.d2H22.hi};
  float p0 = 0.0f, p1 = 0.0f, first = 0.0f;
  for (int it = 0; it < n_iter; ++it) {
    float q0, q1;
    geo_inc_apply(mf, p0, p1, q0, q1);
    const float d = fmaxf(fabsf(q0 - p0), fabsf(q1 - p1));
    if (it == 0) first = d;
    p0 = q0;
    p1 = q1;
    if (d <= 0x1p-20f * fmaxf(fabsf(q0), fabsf(q1))) break;
  }
  geo_inc_apply(m, DF(p0), DF(p1), n0, n1);
  float J[2][2];
  geo_inc_jacobian(mf, p0, p1, J);
  const float r0 = (n0 - DF(p0)).hi, r1 = (n1 - DF(p1)).hi;
  const float w0 = fmaf(J[0][0], r0, J[0][1] * r1), w1 = fmaf(J[1][0], r0, J[1][1] * r1);
  const float a = 1.0f - J[0][0], d = 1.0f - J[1][1];
  const float idet = __fdividef(1.0f, fmaf(a, d, -J[0][1] * J[1][0]));
  n0 = n0 + DF(idet * fmaf(d, w0, J[0][1] * w1));
  n1 = n1 + DF(idet * fmaf(J[1][0], w0, a * w1));
  const float us = fmaxf(fabsf(m.u0.hi), fabsf(m.u1.hi));
  // (a NaN anywhere makes one of the comparisons false)
  const float ds = fmaxf(fabsf(n0.hi), fabsf(n1.hi));
  bool fixed = true;
  rho = spectral_radius(J);
  if (!(fabsf(r0) + fabsf(r1) <= fmaf(0x1p-16f, ds, 0x1p-40f) &&
        inc_converges(first, J, n_iter, tol, us))) {
    // (an iteration that does not contract amplifies the pairs' rounding as well as FP64's)
    if (!LITERAL || !(rho < 0.5f)) return GEO_NONE;
    n0 = n1 = DF(0.0f);
    fixed = false;
#pragma unroll 1
    for (int it = 0; it < n_iter && !fixed; ++it) {
      const DF l0 = n0, l1 = n1;
      geo_inc_apply(m, l0, l1, n0, n1);
      fixed = n0.hi == l0.hi && n0.lo == l0.lo && n1.hi == l1.hi && n1.lo == l1.lo;
    }
  }
  // the increment and the momentum as lengths in the tetrad frame, squared (h^13 aside)
  const float dd = fmaf(mf.H11 * n0.hi, n0.hi, mf.H22 * n1.hi * n1.hi);
  const float uu = fmaf(mf.u0, fmaf(mf.H11, mf.u0, mf.c1), fmaf(mf.H22 * mf.u1, mf.u1, h33));
  const bool none = n0.hi == 0.0f && n1.hi == 0.0f;
  if (none || inc_within(times2, dd, uu)) return GEO_SMALL;
  return fixed && dd < 0x1p60f ? GEO_LARGE : GEO_NONE;
}

// One Boris half step's increment of the covariant u, added to du (u = u^n + du in pairs):
// u' - u = 2 e D + s (p x t) in the tetrad frame (boris), with eD = e D, eB = e B given. h, x:
// the momentum and its increment in that frame. M: the metric's type, R: the vectors'.
template <typename M, typename R>
__device__ __forceinline__ void inc_boris_core(const Local<M> &L, const R eD[3], const R eB[3],
                                               const R u[3], R du[3], R h[3], R x[3]) {
  h[0] = L.sH11 * fma_(-L.m13, u[2], u[0]);
  h[1] = L.rh22 * u[1];
  h[2] = L.rh33 * u[2];
  const R m0 = h[0] + eD[0], m1 = h[1] + eD[1], m2 = h[2] + eD[2];
  const R ig = df_rsqrt(fma_(m0, m0, fma_(m1, m1, fma_(m2, m2, R(1.0f)))));
  const R t0 = eB[0] * ig, t1 = eB[1] * ig, t2 = eB[2] * ig;
  const R sf = df_scale(df_rcp(fma_(t0, t0, fma_(t1, t1, fma_(t2, t2, R(1.0f))))), 2.0f);
  const R p0 = fma_(m1, t2, fma_(-m2, t1, m0));
  const R p1 = fma_(m2, t0, fma_(-m0, t2, m1));
  const R p2 = fma_(m0, t1, fma_(-m1, t0, m2));
  x[0] = fma_(sf, fma_(p1, t2, -(p2 * t1)), df_scale(eD[0], 2.0f));
  x[1] = fma_(sf, fma_(p2, t0, -(p0 * t2)), df_scale(eD[1], 2.0f));
  x[2] = fma_(sf, fma_(p0, t1, -(p1 * t0)), df_scale(eD[2], 2.0f));
  du[0] = du[0] + fma_(L.rH11, x[0], L.k13 * x[2]);
  du[1] = fma_(L.sh22, x[1], du[1]);
  du[2] = fma_(L.sh33, x[2], du[2]);
}
// False: the increment is beyond the bound (inc_within).
__device__ __forceinline__ bool inc_boris(const Local<DF> &L, const DF eD[3], const DF eB[3],
                                          const DF u[3], float times2, DF du[3]) {
  DF h[3], x[3];
  inc_boris_core(L, eD, eB, u, du, h, x);
  const float xx = fmaf(x[0].hi, x[0].hi, fmaf(x[1].hi, x[1].hi, x[2].hi * x[2].hi));
  const float hh = fmaf(h[0].hi, h[0].hi, fmaf(h[1].hi, h[1].hi, h[2].hi * h[2].hi));
  const bool none = fabsf(x[0].hi) + fabsf(x[1].hi) + fabsf(x[2].hi) == 0.0f;
  return (none || inc_within(times2, xx, hh)) && hh < 0x1p60f;
}

// bilinear interpolation in pairs at the cell-relative offsets (o1, o2) of cell (i1, i2) for
// a component offset by h1/2, h2/2 (w: the weights of both kinds per direction, c: their cells)
struct IncLerp {
  int i[2], j[2];
  DF w1[2], w2[2];
};
__device__ __forceinline__ void inc_lerp(int i1, int i2, DF o1, DF o2, IncLerp &l) {
  l.i[0] = i1;
  l.j[0] = i2;
  l.w1[0] = o1;
  l.w2[0] = o2;
  const bool b1 = o1.hi < 0.5f, b2 = o2.hi < 0.5f;
  l.i[1] = i1 - (b1 ? 1 : 0);
  l.j[1] = i2 - (b2 ? 1 : 0);
  l.w1[1] = o1 + DF(b1 ? 0.5f : -0.5f);
  l.w2[1] = o2 + DF(b2 ? 0.5f : -0.5f);
}
__device__ __forceinline__ DF inc_interp(const double *__restrict__ pl, int NX, const IncLerp &l,
                                         int h1, int h2) {
  const double *p = pl + (int64_t)(l.j[h2] + G_) * NX + (l.i[h1] + G_);
  const DF p00 = df_of(__ldg(p)), p10 = df_of(__ldg(p + 1));
  const DF p01 = df_of(__ldg(p + NX)), p11 = df_of(__ldg(p + NX + 1));
  const DF a = fma_(l.w1[h1], p10 - p00, p00), b = fma_(l.w1[h1], p11 - p01, p01);
  return fma_(l.w2[h2], b - a, a);
}

// The coordinate map of Eq. (discretized-geodesic-x) at a point, from r, sin, cos there:
// with w0 = u_1 / f (f = dr/dx1), k = h-tilde^22 u_2 = u_2 / dtheta^2 and
//   I = A w0 / S2 + a u_3,  X = w0 (I + a u_3) + k u_2 + u_3^2 / sin^2,
//   G = (S2 (m2 Sigma + X))^(-1/2)  [= alpha / (gamma Sigma)],   S2 = Sigma + 2 M r,
// V^1 = (G I - 2 M r / S2) / f, V^2 = G k, dphi/dt = G (a w0 + u_3 / sin^2): the metric's
// products regrouped so that no 1/Sigma is needed (one reciprocal, of S2 f sin^2).
template <typename R>
struct Vel {
  R v1, v2, v3;
};
__device__ __forceinline__ Vel<DF> inc_velocity(const IncC &k, DF r, DF s, DF c, const DF u[3],
                                                float m2) {
  const DF s2 = s * s, r2 = r * r, f = k.dxi * r;
  const DF Sig = fma_(k.a2, c * c, r2), M2r = df_scale(k.M * r, 2.0f), S2 = Sig + M2r;
  const DF Rr = r2 + k.a2, A = fma_(Rr, Rr, -(k.a2 * s2 * (Rr - M2r)));
  const DF fs = f * s2, iQ = df_rcp(S2 * fs), iS2 = iQ * fs;
  const DF fi = iQ * S2 * s2, w0 = u[0] * fi, au = k.a * u[2];
  const DF I = fma_(A * iS2, w0, au), kk = k.ig2 * u[1];
  const DF z = u[2] * (iQ * S2 * f);
  const DF X = fma_(w0, I + au, fma_(kk, u[1], u[2] * z));
  const DF Gf = df_rsqrt(S2 * (m2 != 0.0f ? Sig + X : X));
  return {fi * fma_(Gf, I, -(M2r * iS2)), Gf * kk, Gf * fma_(k.a, w0, z)};
}

// r, sin(theta), cos(theta) in FP64 at offsets (o1, o2) of cell (i1, i2): r from the nearest
// corner's table, theta formed from x2 = i2 + o2 as map_theta forms it and its offset from the
// corner's theta exact (as local_rsc)
__device__ __forceinline__ void inc_point64(const GridP &g, const PushTables &tb, int i1, int i2,
                                            double o1, double o2, double x2, double &ex, double &s,
                                            double &c) {
  const int c1 = gt_pos(o1, 0.5), c2 = gt_pos(o2, 0.5);
  const double e = (o1 - (c1 ? 1.0 : 0.0)) * g.dxi;
  if (abs_le(e, (double)INC_E)) {
    double p = 1.0 / 40320.0;
    p = fma(p, e, 1.0 / 5040.0);
    p = fma(p, e, 1.0 / 720.0);
    p = fma(p, e, 1.0 / 120.0);
    p = fma(p, e, 1.0 / 24.0);
    p = fma(p, e, 1.0 / 6.0);
    p = fma(p, e, 0.5);
    p = fma(p, e, 1.0);
    ex = __ldg(tb.r64 + i1 + c1 + G_) * fma(p, e, 1.0);
  } else {
    ex = map_e(g, (double)i1 + o1);
  }
  const double th = __dmul_rn(x2, g.dth);
  const double d = th - __ldg(tb.th64 + i2 + c2 + G_);
  if (abs_le(d, (double)INC_D)) {
    const double q = d * d;
    double sp = fma(-1.0 / 5040.0, q, 1.0 / 120.0);
    sp = fma(sp, q, -1.0 / 6.0);
    const double se = fma(sp * q, d, d);
    double cp = fma(1.0 / 40320.0, q, -1.0 / 720.0);
    cp = fma(cp, q, 1.0 / 24.0);
    cp = fma(cp, q, -0.5);
    const double ce = fma(cp, q, 1.0);
    const double s0 = __ldg(tb.s64 + i2 + c2 + G_), c0 = __ldg(tb.c64 + i2 + c2 + G_);
    s = fma(s0, ce, c0 * se);
    c = fma(c0, ce, -s0 * se);
  } else {
    sincos(th, &s, &c);
  }
}

// The tetrad and the fields in it (times e = qm alpha dt/4) at x^n in FP64: for the half steps in
// strong fields, and the adjoint's derivative by the amplitude
struct Strong {
  double rH11, sH11, rh22, sh22, rh33, sh33, k13, m13, eB[3], eD[3];
  float top;  // the largest of the planes' values there
};
__device__ __forceinline__ void strong_frame(const GridP &g, double *const B[3],
                                             double *const D[3], const PushTables &tb, int i1,
                                             int i2, double dx1, double dx2, double qm,
                                             Strong &w) {
  double r, s, c;
  inc_point64(g, tb, i1, i2, dx1, dx2, __dadd_rn((double)i2, dx2), r, s, c);
  const double s2 = s * s, r2 = r * r, f = g.dxi * r;
  const double Sig = fma(g.a2, c * c, r2), M2r = g.M2 * r, S2 = Sig + M2r;
  const double Rr = r2 + g.a2, A = fma(Rr, Rr, -(g.a2 * s2 * (Rr - M2r)));
  const double rSig = rsqrt(Sig), rS2 = rsqrt(S2), rA = rsqrt(A);
  const double ifs = rcp_nr(f * s), qSig = Sig * rSig, qA = A * rA;
  w.rH11 = f * qSig * (S2 * rS2) * rA;
  w.sH11 = ifs * s * (rSig * rS2) * qA;
  w.rh22 = rSig * (g.ig2 * g.dth);
  w.sh22 = qSig * g.dth;
  w.rh33 = qSig * rA * (ifs * f);
  w.sh33 = s * rSig * qA;
  const double faS = f * g.a * S2;
  w.k13 = -(faS * (s * rSig) * rA);
  w.m13 = -(faS * (rA * rA));
  const double e = 0.25 * qm * (qSig * rS2) * g.dt;  // half of qm alpha dt/2
  const bool l1 = lt_pos(dx1, 0.5) || dx1 == 0.0, l2 = lt_pos(dx2, 0.5) || dx2 == 0.0;
  const double w1[2] = {dx1, l1 ? dx1 + 0.5 : dx1 - 0.5}, w2[2] = {dx2, l2 ? dx2 + 0.5 : dx2 - 0.5};
  double V[6];
  w.top = 0.0f;
#pragma unroll 1
  for (int q = 0; q < 6; ++q) {  // one copy of the code
    const int h1 = q == 1 || q == 2 || q == 3, h2 = q == 0 || q == 2 || q == 4;
    const double *pl = q < 3 ? B[q] : D[q - 3];
    const double *p = pl + sidx(g, i1 - (h1 && l1 ? 1 : 0), i2 - (h2 && l2 ? 1 : 0));
    const double p00 = __ldg(p), p10 = __ldg(p + 1), p01 = __ldg(p + g.NX), p11 = __ldg(p + g.NX + 1);
    const double a1 = h1 ? w1[1] : w1[0], a2 = h2 ? w2[1] : w2[0];
    const double x = fma(a1, p10 - p00, p00), y = fma(a1, p11 - p01, p01);
    V[q] = fma(a2, y - x, x);
    w.top = fmaxf(w.top, fabsf(f32_trunc(V[q])));
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const double *v = V + 3 * q;
    double *o = q ? w.eD : w.eB;
    o[0] = e * (v[0] * w.rH11);
    o[1] = e * (w.sh22 * v[1]);
    o[2] = e * fma(w.k13, v[0], w.sh33 * v[2]);
  }
}
// The geodesic substep in FP64 from the increment (d0, d1) that the pairs found, where it is large
// against u (cold particles, and next to the axes, where the metric changes by order one over a
// step): evaluations of the FP64 map until the pairs' error in it, below 2^-46 of the increment,
// has contracted (by rho each) to FP64's rounding.
__device__ __forceinline__ void strong_geodesic(const GridP &g, const PushTables &tb, int i1,
                                                int i2, double dx1, double dx2, double m2,
                                                DF d0, DF d1, float rho, double u[3]) {
  Pt<double> p;
  inc_point64(g, tb, i1, i2, dx1, dx2, __dadd_rn((double)i2, dx2), p.r, p.s, p.c);
  p.f = g.dxi * p.r;
  p.gg = g.dth;
  p.igg = g.ig2;
  p.gp = 0.0;
  Local<double> L;
  local_full<false>(g, p, L, false);
  const GeoMap<double> m(g, L, u, m2);
  double t0 = u[0] + df_to_double(d0), t1 = u[1] + df_to_double(d1);
#pragma unroll 1
  for (float left = 1.0f; left > 0x1p-9f; left *= rho) {
    double n0, n1;
    m.apply(t0, t1, n0, n1);
    t0 = n0;
    t1 = n1;
  }
  u[0] = t0;
  u[1] = t1;
}

// The FP64 evaluation of the map t -> dx + dt V((x^n + t)/2) that the result comes from, in
// inc_velocity's grouping: ~80 FP64 operations.
__device__ __forceinline__ void inc_coord64(const GridP &g, const PushTables &tb, int i1, int i2,
                                            double dx1, double dx2, const double u[3], double m2,
                                            double t1, double t2, double &n1, double &n2,
                                            double &v3) {
  double ex, s, c;
  const double o2 = 0.5 * __dadd_rn(dx2, t2);
  inc_point64(g, tb, i1, i2, 0.5 * __dadd_rn(dx1, t1), o2, __dadd_rn((double)i2, o2), ex, s, c);
  const double s2 = s * s, r2 = ex * ex, f = g.dxi * ex;
  const double Sig = fma(g.a2, c * c, r2), M2r = g.M2 * ex, S2 = Sig + M2r;
  const double Rr = r2 + g.a2, A = fma(Rr, Rr, -(g.a2 * s2 * (Rr - M2r)));
  const double fs = f * s2, iQ = rcp_nr(S2 * fs), iS2 = iQ * fs, T = iQ * S2;
  const double fi = T * s2, w0 = u[0] * fi, au = g.a * u[2];
  const double I = fma(A * iS2, w0, au), kk = g.ig2 * u[1];
  const double z = u[2] * (T * f);
  const double X = fma(w0, I + au, fma(kk, u[1], u[2] * z));
  const double Gf = rsqrt(S2 * fma(m2, Sig, X));
  n1 = fma(g.dt * fi, fma(Gf, I, -(M2r * iS2)), dx1);
  n2 = fma(g.dt * Gf, kk, dx2);
  v3 = Gf * fma(g.a, w0, z);
}

// The coordinate substep (n_iter, tol: the method's iterations and what they have to come
// within; FINE: the FP64 evaluations stop once what is left, the contraction times the last
// update, is below 2^-55, else once the update is within tol): as coord_refined (FP32 predictor,
// one step in pairs, FP64 evaluations until the stop rule holds), the FP32 and pair maps in
// inc_velocity's grouping.
template <bool FINE>
__device__ __forceinline__ bool inc_coord(const GridP &g, const IncC &k, const PushTables &tb,
                                          int n_iter, float tol, int i1, int i2, double dx1, double dx2, DF o1, DF o2,
                                          const double u[3], const DF ud[3], double m2, float m2f,
                                          double &t1, double &t2, double &v3) {
  const float uf[3] = {ud[0].hi, ud[1].hi, ud[2].hi};
  const float a1 = o1.hi, a2 = o2.hi, dt = g.f_dt;
  const float au = g.f_a * uf[2], kk = g.f_ig2 * uf[1], ku = kk * uf[1];
  float p1 = a1, p2 = a2, first = 0.0f, d_prev = 0.0f;
  for (int it = 0; it < n_iter; ++it) {
    Pt<float> pf;
    rsc32<false>(g, tb, i1, i2, 0.5f * (a1 + p1), 0.5f * (a2 + p2), pf);
    const float s2 = pf.s * pf.s, r2 = pf.r * pf.r, M2r = g.f_M2 * pf.r;
    const float Sig = fmaf(g.f_a2, pf.c * pf.c, r2), S2 = Sig + M2r, Rr = r2 + g.f_a2;
    const float A = fmaf(Rr, Rr, -(g.f_a2 * s2 * (Rr - M2r)));
    const float fs = pf.f * s2, iQ = __fdividef(1.0f, S2 * fs), iS2 = iQ * fs, T = iQ * S2;
    const float fi = T * s2, w0 = uf[0] * fi, I = fmaf(A * iS2, w0, au), z = uf[2] * (T * pf.f);
    const float X = fmaf(w0, I + au, fmaf(uf[2], z, ku));
    const float Gf = rsqrtf(S2 * fmaf(m2f, Sig, X));
    const float n1 = fmaf(dt * fi, fmaf(Gf, I, -(M2r * iS2)), a1), n2 = fmaf(dt * Gf, kk, a2);
    const float d = fmaxf(fabsf(n1 - p1), fabsf(n2 - p2));
    if (it == 0) first = d;
    const bool fixed = (n1 == p1 && n2 == p2) || settled32_rate(d, d_prev);
    d_prev = d;
    p1 = n1;
    p2 = n2;
    if (fixed) break;
  }
  if (!(p1 > -1.0f && p1 < 2.0f && p2 > -1.0f && p2 < 2.0f)) return false;
  float J[2][2];
  {
    Pt<float> pf;
    rsc32<false>(g, tb, i1, i2, 0.5f * (a1 + p1), 0.5f * (a2 + p2), pf);
    Local<float> Lf;
    local_full<false>(g, pf, Lf);
    coord_jacobian(g, Lf, uf, m2f, J);
  }
  double s1, s2;
  {
    const DF h1 = df_scale(o1 + DF(p1), 0.5f), h2 = df_scale(o2 + DF(p2), 0.5f);
    DF r, s, c;
    // (the midpoint lies within half a cell of the cell: the nearest corner's offset is at
    // most half a cell there too)
    inc_point(k, tb, i1, i2, h1, h2, r, s, c);
    const Vel<DF> v = inc_velocity(k, r, s, c, ud, m2f);
    DF s1d, s2d;
    newton_df(J, DF(p1), DF(p2), fma_(k.dt, v.v1, o1), fma_(k.dt, v.v2, o2), s1d, s2d);
    s1 = df_to_double(s1d);
    s2 = df_to_double(s2d);
  }
  if (!(finite64(s1) && finite64(s2))) return false;
  const float stop = FINE ? fminf(0x1p-43f, 0x1p-55f / fmaxf(spectral_radius(J), 0x1p-30f)) : tol;
  bool conv = false;
  for (int it = 1; it < n_iter && !conv; ++it) {
    inc_coord64(g, tb, i1, i2, dx1, dx2, u, m2, s1, s2, t1, t2, v3);
    conv = converged(t1, s1, stop) && converged(t2, s2, stop);
    s1 = t1;
    s2 = t2;
  }
  const float scale = fmaxf(fabsf(f32_trunc(t1)), fabsf(f32_trunc(t2)));
  return conv && scale < 2.0f && inc_converges(first, J, n_iter, tol, scale);
}

// The coordinate substep in the two cell rows next to an axis, where the map (~1/sin^2(theta))
// has more than one fixed point within reach: the method's iterations from x^n in pairs, then
// FP64 evaluations from the point they settle at, until what is left is below 2^-55. False:
// they do not settle within n_iter, or come near the small-angle clamp.
__device__ __forceinline__ bool inc_coord_axis(const GridP &g, const IncC &k, const PushTables &tb,
                                               int i1, int i2, double dx1, double dx2, DF o1,
                                               DF o2, const double u[3], const DF ud[3], double m2,
                                               float m2f, double &t1, double &t2, double &v3) {
  DF p1 = o1, p2 = o2;
  float d = 0.0f, d_prev = 1.0f;
  bool settled = false;
#pragma unroll 1
  for (int it = 0; it < g.n_iter && !settled; ++it) {
    DF r, s, c;
    inc_point(k, tb, i1, i2, df_scale(o1 + p1, 0.5f), df_scale(o2 + p2, 0.5f), r, s, c);
    if (!(s.hi > 2.0f * g.d_ss[0])) return false;
    const Vel<DF> v = inc_velocity(k, r, s, c, ud, m2f);
    const DF n1 = fma_(k.dt, v.v1, o1), n2 = fma_(k.dt, v.v2, o2);
    if (it > 0) d_prev = d;
    d = fmaxf(fabsf((n1 - p1).hi), fabsf((n2 - p2).hi));
    p1 = n1;
    p2 = n2;
    settled = d <= 0x1p-44f;
    if (!(fabsf(p1.hi - 0.5f) < 1.5f && fabsf(p2.hi - 0.5f) < 1.5f)) return false;
  }
  const float rate = fminf(fmaxf(d / d_prev, 0x1p-12f), 1.0f);  // the contraction, or above it
  if (!settled || rate > 0.25f) return false;
  double s1 = df_to_double(p1), s2 = df_to_double(p2);
  const float stop = 0x1p-55f / rate;
  bool conv = false;
#pragma unroll 1
  for (int it = 0; it < g.n_iter && !conv; ++it) {
    inc_coord64(g, tb, i1, i2, dx1, dx2, u, m2, s1, s2, t1, t2, v3);
    conv = converged(t1, s1, stop) && converged(t2, s2, stop);
    s1 = t1;
    s2 = t2;
  }
  return conv && fabsf(f32_trunc(t1)) < 2.0f && fabsf(f32_trunc(t2)) < 2.0f;
}

// floor of a pair
__device__ __forceinline__ int inc_floor(DF a) {
  const float f = floorf(a.hi);
  return (int)f - (f == a.hi && a.lo < 0.0f ? 1 : 0);
}

}  // namespace
