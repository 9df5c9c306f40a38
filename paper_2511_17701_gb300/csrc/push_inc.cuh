// push_inc.cuh -- one particle of the FP64 path in the increment form (inc.cuh), included by
// particles.cu.
#pragma once
#include "inc.cuh"

namespace {

// An FP32 estimate of whether a Boris half step stays below INC_MAX for a momentum of order 1
// (fields of one node, no interpolation): where it does not, both half steps are taken in FP64
// at once, without trying the pairs first.
__device__ __forceinline__ bool inc_small(const GridP &g, const FieldPtrsT<double> &F,
                                          const PushTables &tb, int i1, int i2, float f_qm) {
  const float r = __ldg(tb.r + i1 + G_), s = __ldg(tb.s + i2 + G_), c = __ldg(tb.c + i2 + G_);
  const float Sig = fmaf(g.f_a2, c * c, r * r), S2 = fmaf(g.f_M2, r, Sig);
  const float Rr = fmaf(r, r, g.f_a2), iSig = __fdividef(1.0f, Sig);
  const float f = g.f_dxi * r;
  const float h11 = f * f * S2 * iSig, h22 = g.f_dth * g.f_dth * Sig, h33 = Rr * Rr * s * s * iSig;
  const float alpha = rsqrtf(S2 * iSig);
  const int64_t n = sidx(g, i1, i2);
  const float b0 = f32_trunc(__ldg(F.Bn[0] + n)), b1 = f32_trunc(__ldg(F.Bn[1] + n)),
              b2 = f32_trunc(__ldg(F.Bn[2] + n)), d0 = f32_trunc(__ldg(F.D[0] + n)),
              d1 = f32_trunc(__ldg(F.D[1] + n)), d2 = f32_trunc(__ldg(F.D[2] + n));
  const float BB = fmaf(h11 * b0, b0, fmaf(h22 * b1, b1, h33 * b2 * b2));
  const float DD = fmaf(h11 * d0, d0, fmaf(h22 * d1, d1, h33 * d2 * d2));
  const float e = 0.5f * f_qm * alpha * g.f_dt;  // twice the half step's coefficient
  return e * e * (BB + DD) <= INC_MAX * INC_MAX;
}

// A Boris half step in FP64, for strong fields
// (u + hat_cov(x) with the half step's change x in that frame, not hat_cov(cov_hat(u) + x): the two
// maps' roundings then enter with the change, not with u)
__device__ __forceinline__ void strong_boris(const Strong &w, double u[3]) {
  const double m0 = fma(w.sH11, fma(-w.m13, u[2], u[0]), w.eD[0]);
  const double m1 = fma(w.rh22, u[1], w.eD[1]), m2 = fma(w.rh33, u[2], w.eD[2]);
  const double ig = rsqrt(fma(m0, m0, fma(m1, m1, fma(m2, m2, 1.0))));
  const double t0 = w.eB[0] * ig, t1 = w.eB[1] * ig, t2 = w.eB[2] * ig;
  const double sf = 2.0 * rcp_nr(fma(t0, t0, fma(t1, t1, fma(t2, t2, 1.0))));
  const double p0 = fma(m1, t2, fma(-m2, t1, m0)), p1 = fma(m2, t0, fma(-m0, t2, m1));
  const double p2 = fma(m0, t1, fma(-m1, t0, m2));
  const double x0 = fma(sf, fma(p1, t2, -(p2 * t1)), 2.0 * w.eD[0]);
  const double x1 = fma(sf, fma(p2, t0, -(p0 * t2)), 2.0 * w.eD[1]);
  const double x2 = fma(sf, fma(p0, t1, -(p1 * t0)), 2.0 * w.eD[2]);
  u[0] = u[0] + fma(x0, w.rH11, w.k13 * x2);
  u[1] = fma(w.sh22, x1, u[1]);
  u[2] = fma(w.sh33, x2, u[2]);
}

// floor of t in (-2, 2), on the integer pipe
__device__ __forceinline__ int inc_cell(double t) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(t);
  const unsigned long long a = b & 0x7fffffffffffffffull, one = 0x3ff0000000000000ull;
  if (a == b) return a >= one ? 1 : 0;
  return a == 0 ? 0 : (a > one ? -2 : -1);
}

// q = qc w of one particle. The unit of charge is the caller's, so q may lie anywhere in FP64's
// range, far outside that of a pair: the deposit in pairs takes q's fraction, in [1, 2), and the
// power of two goes back onto each contribution, exactly, on the integer pipe (add_scaled).
// Whether q's exponent leaves room for that (and q is finite); zero does.
__device__ __forceinline__ bool inc_charge(double q) {
  const unsigned h = (unsigned)__double2hiint(q) & 0x7fffffffu, ex = h >> 20;
  return (ex >= 1023u - 860u && ex <= 1023u + 900u) || (h | (unsigned)__double2loint(q)) == 0u;
}
// adds v 2^e, e in the upper word's exponent field; |v| is 0 or in [2^-126, 2^100]
__device__ __forceinline__ void add_scaled(double *p, DF v, int e) {
  const double x = df_to_double(v);
  const int h = __double2hiint(x);
  atomicAdd(p, (h << 1) == 0 ? x : __hiloint2double(h + e, __double2loint(x)));
}

// deposit64 in pairs, relative to the start cell: the end points a, b are the positions as
// deposit64 rounds them (absolute coordinates). From row or column 16 on they are multiples of
// 2^-48, which a pair holds exactly; before that they have up to 53 bits, so the lengths of the
// move's two parts, which the fluxes are proportional to, are differences formed in FP64 (with
// differences of pairs the flux of a move of 3e-3 cells in the first cells was off by up to 1e-12
// of itself). The rest of deposit64's ~70 FP64 operations is in pairs: their 2^-47 is at or below
// the rounding's share of a move. (i, j): the start cell, (c1, c2): the end cell relative to it.
__device__ __forceinline__ void inc_parts(double a, double b, int c, DF &first, DF &second) {
  if (c == 0) {
    first = second = df_scale(df_of(b - a), 0.5f);
  } else {
    const double r = c > 0 ? 1.0 : (double)(c + 1);
    first = df_of(r - a);
    second = df_of(b - r);
  }
}
__device__ __forceinline__ void inc_deposit(const GridP &g, const FieldPtrsT<double> &F,
                                            double charge, DF idt, int i, int j, double xa1,
                                            double xa2, int c1, int c2, double xb1, double xb2,
                                            DF v3) {
  const int qh = __double2hiint(charge);
  const bool some = (qh << 1) != 0;
  const int e = some ? (qh & 0x7ff00000) - 0x3ff00000 : 0;  // q = 2^e times its fraction
  const DF q = df_of(__hiloint2double(some ? qh - e : qh, __double2loint(charge)));
  const int NX = g.NX;
  const DF qi = q * idt;
  const DF a1 = df_of(xa1), a2 = df_of(xa2), b1 = df_of(xb1), b2 = df_of(xb2);
  DF p1, l1, p2, l2;  // the parts' lengths in the start cell, in the end cell
  inc_parts(xa1, xb1, c1, p1, l1);
  inc_parts(xa2, xb2, c2, p2, l2);
  const DF m1 = df_scale(a1 + b1, 0.5f), m2 = df_scale(a2 + b2, 0.5f);
  // the relay point: the midpoint clamped to the two cells' common range
  const DF r1 = c1 == 0 ? m1 : DF(c1 > 0 ? 1.0f : (float)(c1 + 1));
  const DF r2 = c2 == 0 ? m2 : DF(c2 > 0 ? 1.0f : (float)(c2 + 1));
  const int64_t ka = sidx(g, i, j), kb = sidx(g, i + c1, j + c2);
  double *J1 = F.J[0], *J2 = F.J[1], *J3 = F.J[2];
  {
    const DF F1 = qi * p1, F2 = qi * p2;
    const DF t = F1 * df_scale(a2 + r2, 0.5f), s = F2 * df_scale(a1 + r1, 0.5f);
    add_scaled(J1 + ka, F1 - t, e);
    add_scaled(J1 + ka + NX, t, e);
    add_scaled(J2 + ka, F2 - s, e);
    add_scaled(J2 + ka + 1, s, e);
  }
  {
    const DF F1 = qi * l1, F2 = qi * l2;
    const DF t = F1 * (df_scale(r2 + b2, 0.5f) + DF(-(float)c2));
    const DF s = F2 * (df_scale(r1 + b1, 0.5f) + DF(-(float)c1));
    add_scaled(J1 + kb, F1 - t, e);
    add_scaled(J1 + kb + NX, t, e);
    add_scaled(J2 + kb, F2 - s, e);
    add_scaled(J2 + kb + 1, s, e);
  }
  const int n1 = inc_floor(m1), n2 = inc_floor(m2);
  const DF w1 = m1 + DF(-(float)n1), w2 = m2 + DF(-(float)n2);
  const int64_t k = sidx(g, i + n1, j + n2);
  const DF qv = q * v3, x = qv * w1, y = qv - x;
  const DF xt = x * w2, yt = y * w2;
  add_scaled(J3 + k, y - yt, e);
  add_scaled(J3 + k + 1, x - xt, e);
  add_scaled(J3 + k + NX, yt, e);
  add_scaled(J3 + k + NX + 1, xt, e);
}

// A massless particle's momentum has no scale: the step's equations keep their form under u -> c u.
// The pairs take it in a unit, the power of two that brings its largest component to [1, 2)
// (exactly). False: beyond 2^+-480, where FP64's squares end too.
__device__ __forceinline__ bool photon_unit(double u[3], double &unit) {
  int top = 0;
#pragma unroll
  for (int q = 0; q < 3; ++q) top = max(top, __double2hiint(u[q]) & 0x7ff00000);
  if (top < ((1023 - 480) << 20) || top > ((1023 + 480) << 20)) return false;
  unit = __hiloint2double(top, 0);
  const double down = __hiloint2double((2046 << 20) - top, 0);
#pragma unroll
  for (int q = 0; q < 3; ++q) u[q] *= down;
  return true;
}

// One particle in the increment form; false: nothing stored, push64 has to take it. Loops that
// the compiler would unroll stay loops: the code is straight-line and long, and warps waited
// for its instructions (17% of their time with every copy unrolled).
template <bool DEPOSIT>
__device__ __forceinline__ bool push_inc(const GridP &g, const FieldPtrsT<double> &F,
                                         const PushTables &tb, const SpeciesDevT<double> &s,
                                         int64_t kp, unsigned long long *diag) {
  const int i1 = s.i1[kp], i2 = s.i2[kp];
  if (!(i2 >= 0 && i2 < g.n_th && i1 >= 0 && i1 < g.n_r)) return false;
  if (DEPOSIT && !inc_charge(s.qc * s.w[kp])) return false;
  const bool em = s.m2 != 0.0, axis = i2 < 2 || i2 >= g.n_th - 2;
  const double dx1 = s.dx1[kp], dx2 = s.dx2[kp];
  const DF o1 = df_of(dx1), o2 = df_of(dx2);
  // Next to theta = pi an absolute position x2 ~ n_theta has a last place of up to n_theta 2^-52
  // cells, and dphi/dt, ~ 1/d^2 at a distance of d cells, follows a position rounded the other way
  // by twice that over d. Within n_theta 2^-10 cells of the axis (an angle of pi / 1024), where it
  // is above 2^-41 = 4.5e-13 of dphi/dt, push64's own sequence of roundings is kept.
  const float pole = (float)g.n_th * 0x1p-10f;
  if (axis && (float)(g.n_th - i2) - o2.hi < pole) return false;
  const IncC k = inc_c(g);
  double un[3] = {s.u1[kp], s.u2[kp], s.u3[kp]}, unit = 1.0;
  if (!em && !photon_unit(un, unit)) return false;
  DF ud[3] = {df_of(un[0]), df_of(un[1]), df_of(un[2])};
  {
    const DF u[3] = {ud[0], ud[1], ud[2]};
    DF du[3] = {DF(0.0f), DF(0.0f), DF(0.0f)};
    Local<DF> L;
    {
      DF r, sn, cs;
      if (!inc_point_n(g, k, tb, i1, i2, dx2, o1, o2, r, sn, cs) || !(sn.hi > 2.0f * g.d_ss[0])) return false;
      inc_local(k, r, sn, cs, L);
    }
    DF eD[3], eB[3];
    Strong w;
    // (far outside this range of q/m the force's factors, not the force, leave FP32's range). The
    // two forms round differently, so each particle decides for itself: a vote of the warp would
    // make its bits depend on the particles beside it.
    const float qm = fabsf(s.f_qm);
    bool weak = !em || (((qm >= 0x1p-60f && qm <= 0x1p30f) || s.qm == 0.0) &&
                        inc_small(g, F, tb, i1, i2, s.f_qm));
    if (em && weak) {
      IncLerp l;
      inc_lerp(i1, i2, o1, o2, l);
      const DF e = df_scale(df_of(s.qm) * L.alpha * k.dt, 0.25f);  // half of qm alpha dt/2
      DF V[6];
#pragma unroll 1
      for (int q = 0; q < 6; ++q) {
        const int h1 = q == 1 || q == 2 || q == 3, h2 = q == 0 || q == 2 || q == 4;
        V[q] = inc_interp(q < 3 ? F.Bn[q] : F.D[q - 3], g.NX, l, h1, h2);
      }
      vec_hat(L, V, eB);
      vec_hat(L, V + 3, eD);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        eB[q] = e * eB[q];
        eD[q] = e * eD[q];
      }
      weak = inc_boris(L, eD, eB, u, 1.0f, du);
    }
    if (!weak) {
      strong_frame(g, F.Bn, F.D, tb, i1, i2, dx1, dx2, s.qm, w);
      strong_boris(w, un);
#pragma unroll
      for (int q = 0; q < 3; ++q) ud[q] = df_of(un[q]);
      du[0] = du[1] = du[2] = DF(0.0f);
    } else {
#pragma unroll
      for (int q = 0; q < 3; ++q) ud[q] = u[q] + du[q];
    }
    {
      GeoInc<DF> m;
      geo_inc_setup(k, L, ud, em ? 1.0f : 0.0f, m);
      DF d0, d1;
      float rho;
      // in the axis rows the result is the method's to rounding, as push64's is there
      const int found = geo_inc_solve<true>(m, L.G.H33.hi * ud[2].hi * ud[2].hi, g.n_iter,
                                            axis ? 0x1p-54f : g.f_iter_tol,
                                            em ? 1.0f : 0.25f, d0, d1, rho);
      if (found == GEO_NONE) return false;
      if (found == GEO_LARGE) {
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          un[q] += df_to_double(du[q]);
          du[q] = DF(0.0f);
        }
        strong_geodesic(g, tb, i1, i2, dx1, dx2, s.m2, d0, d1, rho, un);
      } else {
        du[0] = du[0] + d0;
        du[1] = du[1] + d1;
      }
    }
    if (em && weak) {  // (twice the bound, so that a particle next to it need not start over)
#pragma unroll
      for (int q = 0; q < 3; ++q) ud[q] = df_of(un[q]) + du[q];
      if (!inc_boris(L, eD, eB, ud, 4.0f, du)) return false;
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) un[q] += df_to_double(du[q]);
    if (!weak) strong_boris(w, un);
#pragma unroll
    for (int q = 0; q < 3; ++q) ud[q] = df_of(un[q]);
  }
  double t1, t2, v3;
  const float m2f = em ? 1.0f : 0.0f;
  if (axis) {
    if (!inc_coord_axis(g, k, tb, i1, i2, dx1, dx2, o1, o2, un, ud, s.m2, m2f, t1, t2, v3))
      return false;
  } else if (!inc_coord<false>(g, k, tb, g.n_iter, g.f_iter_tol, i1, i2, dx1, dx2, o1, o2, un, ud,
                               s.m2, m2f, t1, t2, v3)) {
    return false;
  }
  if (!(finite64(un[0]) && finite64(un[1]) && finite64(un[2]))) return false;
  const int c1 = inc_cell(t1);
  int c2 = inc_cell(t2);
  const int j1 = i1 + c1;
  int j2 = i2 + c2;
  const double e1 = t1 - (double)c1;
  double e2 = t2 - (double)c2;
  bool reflected = false;
  if (j2 < 0 || j2 >= g.n_th) {  // reflection off an axis (Sec. 3.3.3)
    j2 = j2 < 0 ? 0 : g.n_th - 1;
    e2 = 1.0 - e2;
    c2 = j2 - i2;
    un[1] = -un[1];
    // the midpoint of x^n and the reflected x^{n+1}, below, has to be clear of the small-angle clamp
    const double b2 = (double)c2 + e2;
    const float mid = 0.5f * (f32_trunc(dx2) + f32_trunc(b2)) + (float)(j2 == 0 ? i2 : i2 + 1 - g.n_th);
    if (!axis || fabsf(mid - (j2 == 0 ? 0.0f : 1.0f)) * g.f_dth < 2.0f * g.d_ss[0]) return false;
    reflected = true;
  }
  if (axis) {
    // (ends next to theta = pi: see above)
    if ((float)(g.n_th - j2) - f32_trunc(e2) < pole) return false;
    // dphi/dt varies by order one over the distance to the axis, which next to theta = pi makes
    // it sensitive to how the midpoint is rounded: as push64 rounds it, from the absolute positions
    const double p1 = i1, p2 = i2;
    const double m1 = 0.5 * __dadd_rn(__dadd_rn(p1, dx1), __dadd_rn((double)j1, e1));
    const double m2 = 0.5 * __dadd_rn(__dadd_rn(p2, dx2), __dadd_rn((double)j2, e2));
    Pt<double> p;
    inc_point64(g, tb, i1, i2, m1 - p1, m2 - p2, m2, p.r, p.s, p.c);
    p.f = g.dxi * p.r;
    p.gg = g.dth;
    p.igg = g.ig2;
    p.gp = 0.0;
    double v1, v2;
    velocity64<false>(g, p, un, s.m2, v1, v2, v3);
  }
  if (!em) {
#pragma unroll
    for (int q = 0; q < 3; ++q) un[q] *= unit;
  }
  if (reflected) count(diag, DG_REFLECT);
  s.i1[kp] = j1; s.i2[kp] = j2; s.dx1[kp] = e1; s.dx2[kp] = e2;
  s.u1[kp] = un[0]; s.u2[kp] = un[1]; s.u3[kp] = un[2];
  if (j1 < 0) { s.tag[kp] = 2; count(diag, DG_LEFT_INNER); }
  else if (j1 >= g.n_r) { s.tag[kp] = 2; count(diag, DG_LEFT_OUTER); }
  s.phi[kp] = s.phi[kp] + g.dt * v3;
  if (DEPOSIT) {
    const double p1 = i1, p2 = i2;
    inc_deposit(g, F, s.qc * s.w[kp], df_of(g.idt), i1, i2,
                __dadd_rn(__dadd_rn(p1, dx1), -p1), __dadd_rn(__dadd_rn(p2, dx2), -p2), c1, c2,
                __dadd_rn(__dadd_rn((double)j1, e1), -p1), __dadd_rn(__dadd_rn((double)j2, e2), -p2),
                df_of(v3));
  }
  return true;
}

}  // namespace
