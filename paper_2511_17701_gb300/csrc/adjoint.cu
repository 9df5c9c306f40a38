// adjoint.cu -- adjoint of the GR pusher over frozen fields (Sec. 3.1 of arXiv:2511.17701):
// gradients of the final test-particle state (x1, x2, phi, u_1, u_2, u_3) with respect to the
// initial state and the field amplitude (the Wald field is linear in B0), for massive charged
// test particles.
//
// Forward: every particle is pushed n_steps steps in the em-plane fields times
// scale = B0 / (the amplitude the planes hold), both implicit substeps iterated to an exact
// repeat (at most n_iter times), with the state stored every `every` steps (checkpoints).
// Backward (reverse sweep, one thread per particle): for each checkpoint segment, last to
// first, the segment's states are recomputed into scratch memory, then the steps are
// traversed backwards with lambda <- J^T lambda, where J is the 6 x 7 Jacobian of one step
// (inputs: the state and the scale). J comes from forward-mode dual numbers through the same
// templates the pusher uses (pusher.cuh): one pass seeding x1, x2 (the metric differentiated
// too) and one seeding u_1, u_2, u_3 and the scale (metric values only; it depends on x
// alone). At the two implicit substeps the implicit-function theorem replaces
// differentiation through the iterations: at the fixed point t* = G(t*, p),
// dt* = (I - dG/dt)^{-1} (dG/dp) dp. The Jacobians of a segment are formed while its states
// are recomputed and kept in scratch memory for the reverse sweep.
//
// Both passes run a step in the increment form of inc.cuh where it applies: the state's
// increment and the derivatives by x1, x2, which are small against the state and 1, in pairs of
// floats, added in FP64; those by u_1, u_2, u_3 and the scale in FP64. The general FP64 form
// (step_values, step_jacobian) takes the rest.
#include "dual.cuh"
#include "grpic_internal.cuh"
#include "inc.cuh"
#include "pusher.cuh"

namespace {

constexpr int TPB_ADJ = 64;
using D2 = Dual<2>;
using D4 = Dual<4>;

// the point at absolute code coordinates on the plain log-r grid (the adjoint's entry points
// reject quasi-spherical grids): r, sin(theta), cos(theta) with theta clamped to
// [small_angle, pi - small_angle] for the metric (Sec. 3.3.2), with zero derivative there,
// and the map's factors f = dxi r, gg = dtheta
template <typename R>
__device__ __forceinline__ void rsc_abs(const GridP &g, const R &x1, const R &x2, Pt<R> &p) {
  const R e = g.r_min * exp_(x1 * g.dxi);
  p.r = e;
  p.f = g.dxi * e;
  p.gg = R(g.dth);
  p.igg = R(g.ig2);
  p.gp = R(0.0);
  R &s = p.s, &c = p.c;
  const R th = x2 * g.dth;
  const double tv = val(th);
  if (tv < g.small_angle || tv > GRPIC_PI - g.small_angle) {
    double sv, cv;
    sincos(tv < g.small_angle ? g.small_angle : GRPIC_PI - g.small_angle, &sv, &cv);
    s = R(sv);
    c = R(cv);
  } else {
    sincos_(th, s, c);
  }
}

// bilinear interpolation at absolute code coordinates for a Yee offset (s1, s2)
template <typename R>
__device__ __forceinline__ R interp_abs(const double *__restrict__ pl, int NX, const R &x1,
                                        const R &x2, double s1, double s2) {
  const R y1 = x1 - s1, y2 = x2 - s2;
  const double f1 = floor(val(y1)), f2 = floor(val(y2));
  const int i0 = (int)f1, j0 = (int)f2;
  const R w1 = y1 - f1, w2 = y2 - f2;
  const double *p = pl + (int64_t)(j0 + G_) * NX + (i0 + G_);
  const double p00 = __ldg(p), p10 = __ldg(p + 1), p01 = __ldg(p + NX), p11 = __ldg(p + NX + 1);
  return (1.0 - w1) * (1.0 - w2) * p00 + w1 * (1.0 - w2) * p10 + (1.0 - w1) * w2 * p01 +
         w1 * w2 * p11;
}

// metric with derivatives, tetrad-frame fields (at unit amplitude and at `scale`) and the
// Boris coefficient at x^n
template <typename R>
struct Frame {
  Local<R> L;
  R Bh1[3], Dh1[3];  // unit amplitude
  R Bh[3], Dh[3], hq;
};
template <typename R>
__device__ __forceinline__ void frame_at(const GridP &g, const FieldPtrsT<double> &F,
                                         const R x[2], const R &scale, double qm, Frame<R> &fr) {
  R Bv[3], Dv[3];
  Bv[0] = interp_abs(F.B[0], g.NX, x[0], x[1], 0.0, 0.5);
  Bv[1] = interp_abs(F.B[1], g.NX, x[0], x[1], 0.5, 0.0);
  Bv[2] = interp_abs(F.B[2], g.NX, x[0], x[1], 0.5, 0.5);
  Dv[0] = interp_abs(F.D[0], g.NX, x[0], x[1], 0.5, 0.0);
  Dv[1] = interp_abs(F.D[1], g.NX, x[0], x[1], 0.0, 0.5);
  Dv[2] = interp_abs(F.D[2], g.NX, x[0], x[1], 0.0, 0.0);
  Pt<R> p;
  rsc_abs(g, x[0], x[1], p);
  local_full(g, p, fr.L);
  vec_hat(fr.L, Bv, fr.Bh1);
  vec_hat(fr.L, Dv, fr.Dh1);
  for (int i = 0; i < 3; ++i) {
    fr.Bh[i] = scale * fr.Bh1[i];
    fr.Dh[i] = scale * fr.Dh1[i];
  }
  fr.hq = qm * fr.L.alpha * 0.5 * g.dt;
}

// one EM half step: to the tetrad frame, Boris over dt/2, back (steps 3-5 and 7-9)
template <typename M, typename R>
__device__ __forceinline__ void em_half(const Local<M> &L, const R Dh[3], const R Bh[3],
                                        const R &hq, const R uin[3], R uout[3]) {
  R uh[3];
  cov_hat(L, uin, uh);
  boris(uh, Dh, Bh, hq);
  hat_cov(L, uh, uout);
}

// coordinate velocity dx^i/dt of Eq. (discretized-geodesic-x) from the metric at the point
template <typename M, typename R>
__device__ __forceinline__ void velocity(const Geo<M> &o, const R u[3], R &v1, R &v2) {
  const R q = fma_(o.H11 * u[0], u[0], fma_(o.H22 * u[1], u[1],
              fma_(o.H33 * u[2], u[2], fma_(o.H13, (R)2 * u[0] * u[2], (R)1))));
  const R ag = rsqrt_(o.opz * q);  // alpha / gamma
  v1 = fma_(ag, fma_(o.H11, u[0], o.H13 * u[2]), R(-o.beta1));
  v2 = ag * o.H22 * u[1];
}
template <typename R>
__device__ __forceinline__ void geo_abs(const GridP &g, const R &x1, const R &x2, Geo<R> &o) {
  Pt<R> p;
  rsc_abs(g, x1, x2, p);
  geo_from_rsc(g, p, o);
}

// dphi/dt of Eq. (discretized-geodesic-x-phi) at a point
template <typename R>
__device__ __forceinline__ R phi_rate(const GridP &g, const R &x1, const R &x2, const R u[3]) {
  Geo<R> o;
  geo_abs(g, x1, x2, o);
  const R q = fma_(o.H11 * u[0], u[0], fma_(o.H22 * u[1], u[1],
              fma_(o.H33 * u[2], u[2], fma_(o.H13, (R)2 * u[0] * u[2], (R)1))));
  return rsqrt_(o.opz * q) * fma_(o.H13, u[0], o.H33 * u[2]);
}

// The values of one step from state st = (x1, x2, phi, u1, u2, u3).
struct StepVals {
  double u1[3];  // after the first EM half step
  double t[2];   // converged geodesic iterate (u_1, u_2)
  double un[3];  // u^{n+1}
  double xn[2];  // converged x^{n+1}
  double phin;   // phi^{n+1}
  bool ok;       // finite and inside 0 <= x1 < n_r, 0 <= x2 <= n_th
};

__device__ __noinline__ void step_values(const GridP &g, const FieldPtrsT<double> &F,
                                            const double st[6], double scale, double qm,
                                            int n_iter, StepVals &sv, Frame<double> &fr) {
  const double x[2] = {st[0], st[1]}, u[3] = {st[3], st[4], st[5]};
  frame_at(g, F, x, scale, qm, fr);
  em_half(fr.L, fr.Dh, fr.Bh, fr.hq, u, sv.u1);
  const GeoMap<double> gm(g, fr.L, sv.u1, 1.0);
  double t0 = sv.u1[0], t1 = sv.u1[1];
  for (int it = 0; it < n_iter; ++it) {
    double n0, n1;
    gm.apply(t0, t1, n0, n1);
    const bool fixed = n0 == t0 && n1 == t1;
    t0 = n0;
    t1 = n1;
    if (fixed) break;
  }
  sv.t[0] = t0;
  sv.t[1] = t1;
  const double u2[3] = {t0, t1, sv.u1[2]};
  em_half(fr.L, fr.Dh, fr.Bh, fr.hq, u2, sv.un);
  double a0 = x[0], a1 = x[1];  // the first iterate is x^n
  for (int it = 0; it < n_iter; ++it) {
    Geo<double> o;
    geo_abs(g, 0.5 * (x[0] + a0), 0.5 * (x[1] + a1), o);
    double v1, v2;
    velocity(o, sv.un, v1, v2);
    const double n0 = fma(g.dt, v1, x[0]), n1 = fma(g.dt, v2, x[1]);
    const bool fixed = n0 == a0 && n1 == a1;
    a0 = n0;
    a1 = n1;
    if (fixed) break;
  }
  sv.xn[0] = a0;
  sv.xn[1] = a1;
  sv.ok = isfinite(a0) && isfinite(a1) && isfinite(sv.un[0]) && isfinite(sv.un[1]) &&
          isfinite(sv.un[2]) && a0 >= 0.0 && a0 < g.n_r && a1 >= 0.0 && a1 <= g.n_th;
  sv.phin = sv.ok ? fma(g.dt, phi_rate(g, 0.5 * (x[0] + a0), 0.5 * (x[1] + a1), sv.un), st[2])
                  : st[2];
}

__device__ __forceinline__ bool inside(const GridP &g, const double st[6]) {
  bool ok = st[0] >= 0.0 && st[0] < g.n_r && st[1] >= 0.0 && st[1] <= g.n_th;
  for (int q = 2; q < 6; ++q) ok = ok && isfinite(st[q]);
  return ok;
}

// inverse of a 2 x 2 matrix I - A
__device__ __forceinline__ void inv_i_minus(const double A[2][2], double M[2][2]) {
  const double a = 1.0 - A[0][0], b = -A[0][1], c = -A[1][0], d = 1.0 - A[1][1];
  const double id = 1.0 / (a * d - b * c);
  M[0][0] = d * id;
  M[0][1] = -b * id;
  M[1][0] = -c * id;
  M[1][1] = a * id;
}

// The step's Jacobian at st: J[r][c] = d(output r)/d(input c), outputs x1, x2, phi, u1, u2,
// u3 after the step, inputs x1, x2, u1, u2, u3, scale (the phi column is the unit vector).
constexpr int JC = 6;  // stored input columns
__device__ __noinline__ void step_jacobian(const GridP &g, const FieldPtrsT<double> &F, const double st[6],
                              double scale, double qm, const StepVals &sv,
                              const Frame<double> &fr, double J[6][JC]) {
  // the implicit-function theorem's matrices: (I - dG/dt)^{-1} of the geodesic map at its fixed
  // point and (I - dt/2 dV/dx_bar)^{-1} at the final coordinate midpoint
  double Mt[2][2], Mx[2][2];
  {
    const GeoMap<double> gv(g, fr.L, sv.u1, 1.0);
    GeoMap<D2> gd;
#define WIDEN(m) gd.m = D2(gv.m);
    WIDEN(u0) WIDEN(u1) WIDEN(hu0) WIDEN(hu1) WIDEN(c0) WIDEN(c1) WIDEN(e1) WIDEN(e2)
    WIDEN(f1) WIDEN(f2) WIDEN(D1a) WIDEN(D1b) WIDEN(D2a) WIDEN(D2b) WIDEN(hdt)
    WIDEN(H11) WIDEN(H22) WIDEN(d1H11) WIDEN(d1H22) WIDEN(d2H11) WIDEN(d2H22)
#undef WIDEN
    D2 t0(sv.t[0]), t1(sv.t[1]), n0, n1;
    t0.d[0] = 1.0;
    t1.d[1] = 1.0;
    gd.apply(t0, t1, n0, n1);
    const double A[2][2] = {{n0.d[0], n0.d[1]}, {n1.d[0], n1.d[1]}};
    inv_i_minus(A, Mt);
    D2 xb1(0.5 * (st[0] + sv.xn[0])), xb2(0.5 * (st[1] + sv.xn[1]));
    xb1.d[0] = 1.0;
    xb2.d[1] = 1.0;
    Geo<D2> ob;
    geo_abs(g, xb1, xb2, ob);
    const D2 un[3] = {D2(sv.un[0]), D2(sv.un[1]), D2(sv.un[2])};
    D2 v1, v2;
    velocity(ob, un, v1, v2);
    const double h = 0.5 * g.dt;
    const double B[2][2] = {{h * v1.d[0], h * v1.d[1]}, {h * v2.d[0], h * v2.d[1]}};
    inv_i_minus(B, Mx);
  }
  // pass A: x1, x2 seeded; the metric, fields and tetrads differentiated
  {
    D2 X[2] = {D2(st[0]), D2(st[1])};
    X[0].d[0] = 1.0;
    X[1].d[1] = 1.0;
    const D2 U[3] = {D2(st[3]), D2(st[4]), D2(st[5])};
    Frame<D2> fd;
    frame_at(g, F, X, D2(scale), qm, fd);
    D2 U1[3], U2[3], U3[3];
    em_half(fd.L, fd.Dh, fd.Bh, fd.hq, U, U1);
    const GeoMap<D2> gm(g, fd.L, U1, D2(1.0));
    D2 n0, n1;
    gm.apply(D2(sv.t[0]), D2(sv.t[1]), n0, n1);
    U2[0] = D2(sv.t[0]);
    U2[1] = D2(sv.t[1]);
    U2[2] = U1[2];
    for (int k = 0; k < 2; ++k) {
      U2[0].d[k] = Mt[0][0] * n0.d[k] + Mt[0][1] * n1.d[k];
      U2[1].d[k] = Mt[1][0] * n0.d[k] + Mt[1][1] * n1.d[k];
    }
    em_half(fd.L, fd.Dh, fd.Bh, fd.hq, U2, U3);
    Geo<D2> ob;
    geo_abs(g, 0.5 * (X[0] + sv.xn[0]), 0.5 * (X[1] + sv.xn[1]), ob);
    D2 v1, v2;
    velocity(ob, U3, v1, v2);
    D2 XN[2] = {D2(sv.xn[0]), D2(sv.xn[1])};
    for (int k = 0; k < 2; ++k) {
      const double r0 = X[0].d[k] + g.dt * v1.d[k], r1 = X[1].d[k] + g.dt * v2.d[k];
      XN[0].d[k] = Mx[0][0] * r0 + Mx[0][1] * r1;
      XN[1].d[k] = Mx[1][0] * r0 + Mx[1][1] * r1;
    }
    const D2 v3 = phi_rate(g, 0.5 * (X[0] + XN[0]), 0.5 * (X[1] + XN[1]), U3);
    for (int k = 0; k < 2; ++k) {
      J[0][k] = XN[0].d[k];
      J[1][k] = XN[1].d[k];
      J[2][k] = g.dt * v3.d[k];
      J[3][k] = U3[0].d[k];
      J[4][k] = U3[1].d[k];
      J[5][k] = U3[2].d[k];
    }
  }
  // pass B: u_1, u_2, u_3 and the scale seeded; the metric at x^n and at the final
  // coordinate midpoint is fixed (values), the fields are linear in the scale
  {
    D4 U[3] = {D4(st[3]), D4(st[4]), D4(st[5])};
    for (int i = 0; i < 3; ++i) U[i].d[i] = 1.0;
    D4 Bh[3], Dh[3];
    for (int i = 0; i < 3; ++i) {
      Bh[i] = D4(fr.Bh[i]);
      Bh[i].d[3] = fr.Bh1[i];
      Dh[i] = D4(fr.Dh[i]);
      Dh[i].d[3] = fr.Dh1[i];
    }
    const D4 hq(fr.hq);
    D4 U1[3], U2[3], U3[3];
    em_half(fr.L, Dh, Bh, hq, U, U1);
    const GeoMap<D4> gm(g, fr.L, U1, D4(1.0));
    D4 n0, n1;
    gm.apply(D4(sv.t[0]), D4(sv.t[1]), n0, n1);
    U2[0] = D4(sv.t[0]);
    U2[1] = D4(sv.t[1]);
    U2[2] = U1[2];
    for (int k = 0; k < 4; ++k) {
      U2[0].d[k] = Mt[0][0] * n0.d[k] + Mt[0][1] * n1.d[k];
      U2[1].d[k] = Mt[1][0] * n0.d[k] + Mt[1][1] * n1.d[k];
    }
    em_half(fr.L, Dh, Bh, hq, U2, U3);
    Geo<double> ob;
    geo_abs(g, 0.5 * (st[0] + sv.xn[0]), 0.5 * (st[1] + sv.xn[1]), ob);
    D4 v1, v2;
    velocity(ob, U3, v1, v2);
    D4 XN[2] = {D4(sv.xn[0]), D4(sv.xn[1])};
    for (int k = 0; k < 4; ++k) {
      const double r0 = g.dt * v1.d[k], r1 = g.dt * v2.d[k];
      XN[0].d[k] = Mx[0][0] * r0 + Mx[0][1] * r1;
      XN[1].d[k] = Mx[1][0] * r0 + Mx[1][1] * r1;
    }
    const D4 v3 = phi_rate(g, 0.5 * (st[0] + XN[0]), 0.5 * (st[1] + XN[1]), U3);
    for (int k = 0; k < 4; ++k) {
      J[0][2 + k] = XN[0].d[k];
      J[1][2 + k] = XN[1].d[k];
      J[2][2 + k] = g.dt * v3.d[k];
      J[3][2 + k] = U3[0].d[k];
      J[4][2 + k] = U3[1].d[k];
      J[5][2 + k] = U3[2].d[k];
    }
  }
}

// ---------------------------------------------------------------------------------
// A step in the increment form. GB300's FP64 pipe bounded both passes (~1800 FP64 operations
// per particle-step forward, ~5500 backward, most of them exp and sincos per iterate and the
// metric's derivatives in duals); here FP64 is left with the half steps (250 operations with the
// fields and tetrads), one or two evaluations of the coordinate map, the additions to the state
// and, backward, the derivatives along the momentum and the scale (~600). 65,536 orbits on
// 512^2, 100 steps forward and back: 107 -> 39 ms (28 ms with the half steps and all derivatives
// in pairs, whose errors were larger: see ADJ_MAX and the scratch layout below). The backward
// kernel waits for instructions, FP64 results and its pair arithmetic at 8 warps per SM (255
// registers, spills).
// ---------------------------------------------------------------------------------
constexpr int INC_MIN_ITER = 16;   // iteration counts below are taken literally (general form)
constexpr float INC_ADJ_TOL = 1e-16f;
// Half steps and geodesic maps up to this (the turn and the kick of a half step; the map's
// contraction): beyond, the derivatives by x1, x2 in pairs, whose errors are about 1e-14 of the
// entries, leave more than the general form's rounding (200^2, 20 steps, half steps that turn the
// momentum by 0.04: the gradient by x1 off by 3.1e-15 of its rms, the general form's by 8.8e-16;
// at 0.005 7.0e-16 and 9.9e-16).
constexpr float ADJ_MAX = 0x1p-7f;

// A Boris half step from u in FP64 (inc_boris_core) and what its derivatives need of it: m = h + e
// D, t = e B / gamma, p = m + m x t, c = p x t, sf = 2 / (1 + t^2)
struct HalfStep {
  double m[3], t[3], p[3], c[3], ig, sf;
};
__device__ __forceinline__ void cross64(const double a[3], const double b[3], double o[3]) {
  o[0] = fma(a[1], b[2], -(a[2] * b[1]));
  o[1] = fma(a[2], b[0], -(a[0] * b[2]));
  o[2] = fma(a[0], b[1], -(a[1] * b[0]));
}
__device__ __forceinline__ void adj_half64(const Strong &w, double scale, double u[3],
                                           HalfStep &h) {
  h.m[0] = fma(scale, w.eD[0], w.sH11 * fma(-w.m13, u[2], u[0]));
  h.m[1] = fma(scale, w.eD[1], w.rh22 * u[1]);
  h.m[2] = fma(scale, w.eD[2], w.rh33 * u[2]);
  h.ig = rsqrt(fma(h.m[0], h.m[0], fma(h.m[1], h.m[1], fma(h.m[2], h.m[2], 1.0))));
  double x[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) h.t[q] = scale * w.eB[q] * h.ig;
  h.sf = 2.0 * rcp_nr(fma(h.t[0], h.t[0], fma(h.t[1], h.t[1], fma(h.t[2], h.t[2], 1.0))));
  cross64(h.m, h.t, x);
#pragma unroll
  for (int q = 0; q < 3; ++q) h.p[q] = h.m[q] + x[q];
  cross64(h.p, h.t, h.c);
#pragma unroll
  for (int q = 0; q < 3; ++q) x[q] = fma(h.sf, h.c[q], 2.0 * scale * w.eD[q]);
  u[0] += fma(x[0], w.rH11, w.k13 * x[2]);
  u[1] = fma(w.sh22, x[1], u[1]);
  u[2] = fma(w.sh33, x[2], u[2]);
}

struct AdjStep {
  int i1, i2;
  DF o1, o2;            // x^n in its cell
  DF r, s, c;           // there
  Local<DF> L;
  Strong w;             // tetrad and fields (unit amplitude) at x^n
  HalfStep h[2];
  DF u[3], u1[3], dg[2], u2[3], un[3];  // u^n, after the first EM half step, the geodesic
                        // substep's increment, after it, u^{n+1}
  double u64[3], x64[2], v3, mid[2];    // u^{n+1}, x^{n+1}, dphi/dt; the midpoint's offsets
};

// The values of a step, the half steps in FP64; false: not covered by the increment form.
__device__ __forceinline__ bool adj_inc_step(const GridP &g, const FieldPtrsT<double> &F,
                                             const PushTables &tb, const IncC &k,
                                             const double st[6], double scale, double qm,
                                             int n_iter, AdjStep &a) {
  const double f1 = floor(st[0]), f2 = floor(st[1]);
  a.i1 = (int)f1;
  a.i2 = (int)f2;
  if (!(a.i1 >= 0 && a.i1 < g.n_r && a.i2 >= 2 && a.i2 < g.n_th - 2)) return false;
  const double dx1 = st[0] - f1, dx2 = st[1] - f2;
  a.o1 = df_of(dx1);
  a.o2 = df_of(dx2);
  if (!inc_point_n(g, k, tb, a.i1, a.i2, dx2, a.o1, a.o2, a.r, a.s, a.c)) return false;
  inc_local(k, a.r, a.s, a.c, a.L);
  strong_frame(g, F.B, F.D, tb, a.i1, a.i2, dx1, dx2, qm, a.w);
  // the derivatives take the planes' own values in pairs, which have to be clear of the range
  // where a pair loses its low half (2^-74)
  if (!(a.w.top == 0.0f || (a.w.top >= 0x1p-30f && a.w.top <= 0x1p40f))) return false;
  double u[3] = {st[3], st[4], st[5]};
  float turn = 0.0f, kick = 0.0f, mm = 1.0f;
#pragma unroll
  for (int q = 0; q < 3; ++q) a.u[q] = df_of(u[q]);
  adj_half64(a.w, scale, u, a.h[0]);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float t = f32_trunc(a.h[0].t[q]), d = f32_trunc(scale * a.w.eD[q]);
    const float m = f32_trunc(a.h[0].m[q]);
    turn = fmaf(t, t, turn);
    kick = fmaf(d, d, kick);
    mm = fmaf(m, m, mm);
    a.u1[q] = df_of(u[q]);
  }
  // (a NaN anywhere makes one of the comparisons false)
  if (!(4.0f * turn <= ADJ_MAX * ADJ_MAX && 4.0f * kick <= ADJ_MAX * ADJ_MAX * mm && mm < 0x1p60f))
    return false;
  GeoInc<DF> m;
  geo_inc_setup(k, a.L, a.u1, 1.0f, m);
  float rho;
  const int found = geo_inc_solve<false>(m, a.L.G.H33.hi * a.u1[2].hi * a.u1[2].hi, n_iter,
                                         INC_ADJ_TOL, 0.0625f, a.dg[0], a.dg[1], rho);
  if (found == GEO_NONE || !(rho <= ADJ_MAX)) return false;
  if (found == GEO_LARGE) {
    strong_geodesic(g, tb, a.i1, a.i2, dx1, dx2, 1.0, a.dg[0], a.dg[1], rho, u);
  } else {
    u[0] += df_to_double(a.dg[0]);
    u[1] += df_to_double(a.dg[1]);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) a.u2[q] = df_of(u[q]);
  adj_half64(a.w, scale, u, a.h[1]);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    a.u64[q] = u[q];
    a.un[q] = df_of(u[q]);
  }
  double t1, t2;
  if (!inc_coord<true>(g, k, tb, n_iter, INC_ADJ_TOL, a.i1, a.i2, dx1, dx2, a.o1, a.o2, a.u64,
                       a.un, 1.0, 1.0f, t1, t2, a.v3))
    return false;
  a.mid[0] = 0.5 * (dx1 + t1);
  a.mid[1] = 0.5 * (dx2 + t2);
  a.x64[0] = f1 + t1;
  a.x64[1] = f2 + t2;
  return finite64(a.u64[0]) && finite64(a.u64[1]) && finite64(a.u64[2]);
}

// a field component at x^n with its derivatives along x1, x2
__device__ __forceinline__ D2F adj_interp_d(const double *__restrict__ pl, int NX, const IncLerp &l,
                                            int h1, int h2) {
  const double *p = pl + (int64_t)(l.j[h2] + G_) * NX + (l.i[h1] + G_);
  const DF p00 = df_of(__ldg(p)), p10 = df_of(__ldg(p + 1));
  const DF p01 = df_of(__ldg(p + NX)), p11 = df_of(__ldg(p + NX + 1));
  const DF x0 = p10 - p00, x1 = p11 - p01, y0 = p01 - p00;
  const DF xy = x1 - x0, a = fma_(l.w1[h1], x0, p00), b = fma_(l.w1[h1], x1, p01);
  return D2F(fma_(l.w2[h2], b - a, a), fma_(l.w2[h2], xy, x0), fma_(l.w1[h1], xy, y0));
}

// The momentum's derivative along x1, x2: du' of u^{n+1} - u^n for metric values L and fields with
// their derivatives. K: the geodesic substep's (I - A)^{-1}.
__device__ __forceinline__ void adj_momentum_d(const IncC &k, const Local<D2F> &L, const D2F eD[3],
                                               const D2F eB[3], const AdjStep &a,
                                               const DF K[2][2], D2F du[3]) {
  D2F h[3], x[3], v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    v[q] = D2F(a.u[q]);
    du[q] = D2F(0.0f);
  }
#pragma unroll 1
  for (int half = 0;; ++half) {
    inc_boris_core(L, eD, eB, v, du, h, x);
    if (half) return;
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = D2F(a.u1[q], du[q].d0, du[q].d1);
    GeoInc<D2F> m;
    geo_inc_setup(k, L, v, 1.0f, m);
    D2F n0, n1;
    geo_inc_apply(m, a.dg[0], a.dg[1], n0, n1);
    // implicit-function theorem at the fixed point
    du[0].d0 = du[0].d0 + fma_(K[0][0], n0.d0, K[0][1] * n1.d0);
    du[0].d1 = du[0].d1 + fma_(K[0][0], n0.d1, K[0][1] * n1.d1);
    du[1].d0 = du[1].d0 + fma_(K[1][0], n0.d0, K[1][1] * n1.d0);
    du[1].d1 = du[1].d1 + fma_(K[1][0], n0.d1, K[1][1] * n1.d1);
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] = D2F(a.u2[q], du[q].d0, du[q].d1);
  }
}

// (I - A)^{-1}
__device__ __forceinline__ void adj_inv(const DF A[2][2], DF K[2][2]) {
  const DF p = DF(1.0f) - A[0][0], q = DF(1.0f) - A[1][1];
  const DF id = df_rcp(fma_(p, q, -(A[0][1] * A[1][0])));
  K[0][0] = q * id;
  K[0][1] = A[0][1] * id;
  K[1][0] = A[1][0] * id;
  K[1][1] = p * id;
}

// A step's derivatives in scratch memory: entry (row, column) of rows x1, x2, phi, u1, u2, u3
// and columns x1, x2, u1, u2, u3, scale at w[(row * JC + column) n], either J - 1, as pairs (lo,
// hi) in the first two columns and as doubles in the others, or J as doubles; which one is the
// lowest bit of entry (phi, scale), a double in both: clear for J - 1, set for J. (An entry that
// is near 1 would not do: half an ulp of it, always upwards, is in every step's product.)
//
// Why two types: of J - 1 the first two columns are small (1e-3 where J has a 1), so pairs leave
// less of J than FP64 does. The others hold entries that are the whole of J (dt dV/du, the
// rotation between u_1, u_2 and u_3, the fields for the scale), of which pairs kept 2^-47, a part
// of it (the grid's constants, the fields) the same in every step: on 200^2, 30 steps, |u| up to
// 0.5, the gradients' rms errors against 80-bit arithmetic were 2.7e-15 (u1), 1.8e-15 (u2), 3.4e-15
// (scale) where FP64 throughout has 1.5e-15, 1.3e-15, 1.1e-15; now 4.5e-16, 5.4e-16, 4.4e-16.
__device__ __forceinline__ constexpr bool adj_is64(int c) { return c >= 2; }
constexpr int ADJ_FORM = 2 * JC + 5;  // that entry
__device__ __forceinline__ double adj_form(double x, bool general) {
  const long long b = __double_as_longlong(x);
  return __longlong_as_double(general ? b | 1ll : b & ~1ll);
}

// dV_j / du_k of the coordinate velocities at the midpoint in FP64 (adj_inc_jacobian's Vu)
__device__ __forceinline__ void adj_vu64(const GridP &g, const PushTables &tb, const AdjStep &a,
                                         double V[3][3]) {
  double r, s, c;
  inc_point64(g, tb, a.i1, a.i2, a.mid[0], a.mid[1], __dadd_rn((double)a.i2, a.mid[1]), r, s, c);
  const double *u = a.u64;
  const double s2 = s * s, r2 = r * r, f = g.dxi * r;
  const double Sig = fma(g.a2, c * c, r2), M2r = g.M2 * r, S2 = Sig + M2r;
  const double Rr = r2 + g.a2, A = fma(Rr, Rr, -(g.a2 * s2 * (Rr - M2r)));
  const double fs = f * s2, iQ = rcp_nr(S2 * fs), T = iQ * S2, fi = T * s2, AS = A * (iQ * fs);
  const double w0 = u[0] * fi, au = g.a * u[2], I = fma(AS, w0, au), kk = g.ig2 * u[1];
  const double is2 = T * f, z = u[2] * is2, X = fma(w0, I + au, fma(kk, u[1], u[2] * z));
  const double G = rsqrt(S2 * (Sig + X)), iN = G * G * S2, P0 = fi * I, P2 = fma(g.a, w0, z);
  const double q0 = P0 * iN, q1 = kk * iN, q2 = P2 * iN;
  V[0][0] = G * fma(fi * fi, AS, -(q0 * P0));
  V[1][1] = G * fma(-q1, kk, g.ig2);
  V[2][2] = G * fma(-q2, P2, is2);
  V[0][1] = V[1][0] = -(G * (q0 * kk));
  V[0][2] = V[2][0] = G * fma(g.a, fi, -(q0 * P2));
  V[1][2] = V[2][1] = -(G * (q1 * P2));
}
// A half step's derivative: of the increment, added to dw, along a direction that changes u by du
// and the scale by ds
__device__ __forceinline__ void adj_half64_d(const Strong &w, const HalfStep &h,
                                             const double du[3], double ds, double dw[3]) {
  double md[3] = {w.sH11 * fma(-w.m13, du[2], du[0]), w.rh22 * du[1], w.rh33 * du[2]};
  double td[3], pd[3], x[3], y[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) md[q] = fma(ds, w.eD[q], md[q]);
  const double a = -(h.ig * h.ig) * fma(h.m[0], md[0], fma(h.m[1], md[1], h.m[2] * md[2]));
  const double b = h.ig * ds;  // t' = t a + e B b
#pragma unroll
  for (int q = 0; q < 3; ++q) td[q] = fma(h.t[q], a, w.eB[q] * b);
  const double sd = -(h.sf * h.sf) * fma(h.t[0], td[0], fma(h.t[1], td[1], h.t[2] * td[2]));
  cross64(md, h.t, x);
  cross64(h.m, td, y);
#pragma unroll
  for (int q = 0; q < 3; ++q) pd[q] = md[q] + (x[q] + y[q]);
  cross64(pd, h.t, x);
  cross64(h.p, td, y);
#pragma unroll
  for (int q = 0; q < 3; ++q) x[q] = fma(sd, h.c[q], fma(h.sf, x[q] + y[q], 2.0 * ds * w.eD[q]));
  dw[0] += fma(x[0], w.rH11, w.k13 * x[2]);
  dw[1] = fma(w.sh22, x[1], dw[1]);
  dw[2] = fma(w.sh33, x[2], dw[2]);
}

__device__ __forceinline__ void adj_inc_jacobian(const GridP &g, const FieldPtrsT<double> &F,
                                                 const PushTables &tb, const IncC &k, DF scale,
                                                 DF qm, const AdjStep &a, double *wd, int64_t n) {
  float2 *w = reinterpret_cast<float2 *>(wd);
  const DF zero(0.0f);
  // the coordinate map's velocity (inc_velocity's grouping) at the midpoint: its derivatives
  // along x (Vx) and along u (Vu, FP64): with P_j = half of dX/du_j, V_j + beta_j = G P_j and
  // dV_j/du_k = G (c_jk - P_j P_k / N), N = m2 Sigma + X
  DF Vx[3][2], N[2][2];
  {
    DF r, s, c;
    inc_point(k, tb, a.i1, a.i2, df_of(a.mid[0]), df_of(a.mid[1]), r, s, c);
    const D2F R(r, k.dxi * r, zero), S(s, zero, c * k.dth), C(c, zero, -(s * k.dth));
    const D2F s2 = S * S, r2 = R * R, f = k.dxi * R;
    const D2F Sig = fma_(k.a2, C * C, r2), M2r = df_scale(k.M * R, 2.0f), S2 = Sig + M2r;
    const D2F Rr = r2 + k.a2, A = fma_(Rr, Rr, -(k.a2 * s2 * (Rr - M2r)));
    const D2F fs = f * s2, iQ = df_rcp(S2 * fs), iS2 = iQ * fs, T = iQ * S2;
    const D2F fi = T * s2, w0 = a.un[0] * fi, AS = A * iS2, is2 = T * f;
    const DF au = k.a * a.un[2], kk = k.ig2 * a.un[1];
    const D2F I = fma_(AS, w0, D2F(au)), z = a.un[2] * is2;
    const D2F X = fma_(w0, I + au, fma_(a.un[2], z, D2F(kk * a.un[1])));
    const D2F G = df_rsqrt(S2 * (Sig + X));
    const D2F P0 = fi * I, P2 = fma_(k.a, w0, z);
    const D2F V0 = fma_(G, P0, -(M2r * iS2 * fi)), V1 = G * kk, V2 = G * P2;
    Vx[0][0] = V0.d0; Vx[0][1] = V0.d1;
    Vx[1][0] = V1.d0; Vx[1][1] = V1.d1;
    Vx[2][0] = V2.d0; Vx[2][1] = V2.d1;
    const DF h = df_scale(k.dt, 0.5f);
    const DF B[2][2] = {{h * Vx[0][0], h * Vx[0][1]}, {h * Vx[1][0], h * Vx[1][1]}};
    // N = (I - B)^{-1} - I = (I - B)^{-1} B
    DF Mx[2][2];
    adj_inv(B, Mx);
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int p = 0; p < 2; ++p) N[q][p] = fma_(Mx[q][0], B[0][p], Mx[q][1] * B[1][p]);
  }
  double Vu[3][3];
  adj_vu64(g, tb, a, Vu);
  // the geodesic substep: (I - A)^{-1}, and its change along u_1, u_2, u_3 (P)
  DF K[2][2];
  double P[2][3];
  {
    GeoInc<DF> m;
    geo_inc_setup(k, a.L, a.u1, 1.0f, m);
    DF A[2][2], d3[2];
    geo_inc_jacobian(m, a.dg[0], a.dg[1], A);
    geo_inc_d3(a.L, m, a.u1[2], a.dg[0], a.dg[1], d3);
    adj_inv(A, K);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
      for (int p = 0; p < 2; ++p)
        P[q][p] = df_to_double(df_scale(fma_(K[q][0], A[0][p], K[q][1] * A[1][p]), 2.0f));
      P[q][2] = df_to_double(fma_(K[q][0], d3[0], K[q][1] * d3[1]));
    }
  }
  {  // x1, x2: metric, tetrads and fields move; pairs
    Local<D2F> L;
    D2F eB[3], eD[3];
    const D2F R(a.r, k.dxi * a.r, zero), S(a.s, zero, a.c * k.dth), C(a.c, zero, -(a.s * k.dth));
    inc_local(k, R, S, C, L);
    IncLerp l;
    inc_lerp(a.i1, a.i2, a.o1, a.o2, l);
    D2F V[6];
#pragma unroll 1
    for (int q = 0; q < 6; ++q) {
      const int h1 = q == 1 || q == 2 || q == 3, h2 = q == 0 || q == 2 || q == 4;
      V[q] = adj_interp_d(q < 3 ? F.B[q] : F.D[q - 3], g.NX, l, h1, h2);
    }
    vec_hat(L, V, eB);
    vec_hat(L, V + 3, eD);
    const D2F e = df_scale(scale * qm * k.dt, 0.25f) * L.alpha;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      eB[q] = e * eB[q];
      eD[q] = e * eD[q];
    }
    D2F du[3];
    adj_momentum_d(k, L, eD, eB, a, K, du);
    const DF u64[3] = {df_of(Vu[0][0]), df_of(Vu[1][1]), df_of(Vu[2][2])};
    const DF x01 = df_of(Vu[0][1]), x02 = df_of(Vu[0][2]), x12 = df_of(Vu[1][2]);
#pragma unroll 1
    for (int col = 0; col < 2; ++col) {
      DF w3[3], x[3], f[3];
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        w3[q] = col ? du[q].d1 : du[q].d0;
        x[q] = col ? Vx[q][1] : Vx[q][0];
      }
      f[0] = fma_(u64[0], w3[0], fma_(x01, w3[1], fma_(x02, w3[2], x[0])));
      f[1] = fma_(x01, w3[0], fma_(u64[1], w3[1], fma_(x12, w3[2], x[1])));
      f[2] = fma_(x02, w3[0], fma_(x12, w3[1], fma_(u64[2], w3[2], x[2])));
      const DF y0 = k.dt * (f[0] + fma_(N[0][0], f[0], N[0][1] * f[1]));
      const DF y1 = k.dt * (f[1] + fma_(N[1][0], f[0], N[1][1] * f[1]));
      // dphi/dt moves with the midpoint, x + y/2
      const DF ph = k.dt * (f[2] + df_scale(fma_(Vx[2][0], y0, Vx[2][1] * y1), 0.5f));
      const DF o[6] = {y0, y1, ph, w3[0], w3[1], w3[2]};
#pragma unroll
      for (int q = 0; q < 6; ++q)
        w[(int64_t)(q * JC + col) * n] = make_float2(o[q].lo, o[q].hi);
    }
  }
  // u_1, u_2, u_3 and the scale: the metric's values alone, in FP64
  double Nx[2][2], Vp[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    Nx[q][0] = df_to_double(N[q][0]);
    Nx[q][1] = df_to_double(N[q][1]);
    Vp[q] = 0.5 * df_to_double(Vx[2][q]);
  }
#pragma unroll 1
  for (int col = 2; col < JC; ++col) {
    const double s[3] = {col == 2 ? 1.0 : 0.0, col == 3 ? 1.0 : 0.0, col == 4 ? 1.0 : 0.0};
    const double ds = col == 5 ? 1.0 : 0.0;
    double dw[3] = {0.0, 0.0, 0.0}, d[3];
    adj_half64_d(a.w, a.h[0], s, ds, dw);
#pragma unroll
    for (int q = 0; q < 3; ++q) d[q] = s[q] + dw[q];
    dw[0] += fma(P[0][0], d[0], fma(P[0][1], d[1], P[0][2] * d[2]));
    dw[1] += fma(P[1][0], d[0], fma(P[1][1], d[1], P[1][2] * d[2]));
#pragma unroll
    for (int q = 0; q < 2; ++q) d[q] = s[q] + dw[q];
    adj_half64_d(a.w, a.h[1], d, ds, dw);
    double f[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) d[q] = s[q] + dw[q];
#pragma unroll
    for (int q = 0; q < 3; ++q) f[q] = fma(Vu[q][0], d[0], fma(Vu[q][1], d[1], Vu[q][2] * d[2]));
    const double y0 = g.dt * (f[0] + fma(Nx[0][0], f[0], Nx[0][1] * f[1]));
    const double y1 = g.dt * (f[1] + fma(Nx[1][0], f[0], Nx[1][1] * f[1]));
    const double ph = g.dt * (f[2] + fma(Vp[0], y0, Vp[1] * y1));
    const double o[6] = {y0, y1, col == 5 ? adj_form(ph, false) : ph, dw[0], dw[1], dw[2]};
#pragma unroll
    for (int q = 0; q < 6; ++q) wd[(int64_t)(q * JC + col) * n] = o[q];
  }
}

// One step forward from st in either form; false: the particle left the domain
template <bool INC>
__device__ __forceinline__ bool adj_advance(const GridP &g, const FieldPtrsT<double> &F,
                                            const PushTables &tb, const IncC &k, double scale,
                                            DF scale_df, double qm, DF qm_df, int n_iter,
                                            double st[6], double *w, int64_t n) {
  if (INC) {
    AdjStep a;
    if (adj_inc_step(g, F, tb, k, st, scale, qm, n_iter, a)) {
      const bool ok = a.x64[0] >= 0.0 && a.x64[0] < g.n_r && a.x64[1] >= 0.0 && a.x64[1] <= g.n_th;
      if (!ok) return false;
      if (w) adj_inc_jacobian(g, F, tb, k, scale_df, qm_df, a, w, n);
      st[0] = a.x64[0];
      st[1] = a.x64[1];
      st[2] = fma(g.dt, a.v3, st[2]);
      st[3] = a.u64[0];
      st[4] = a.u64[1];
      st[5] = a.u64[2];
      return true;
    }
  }
  StepVals sv;
  Frame<double> fr;
  step_values(g, F, st, scale, qm, n_iter, sv, fr);
  if (!sv.ok) return false;
  if (w) {
    double J[6][JC];
    step_jacobian(g, F, st, scale, qm, sv, fr, J);
    for (int r = 0; r < 6; ++r)
      for (int c = 0; c < JC; ++c) w[(int64_t)(r * JC + c) * n] = J[r][c];
    w[(int64_t)ADJ_FORM * n] = adj_form(J[2][5], true);
  }
  st[0] = sv.xn[0]; st[1] = sv.xn[1]; st[2] = sv.phin;
  st[3] = sv.un[0]; st[4] = sv.un[1]; st[5] = sv.un[2];
  return true;
}

template <bool INC>
__global__ void __launch_bounds__(TPB_ADJ) k_adj_forward(
    const __grid_constant__ GridP g, const __grid_constant__ FieldPtrsT<double> F,
    const __grid_constant__ PushTables tb, int64_t n, double qm, double scale, int n_steps,
    int every, int n_iter, const double *__restrict__ st0, double *__restrict__ out,
    double *__restrict__ ckpt) {
  const IncC kc = inc_c(g);
  const DF sd = df_of(scale), qd = df_of(qm);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    double st[6];
    for (int q = 0; q < 6; ++q) st[q] = st0[q * n + k];
    bool bad = !inside(g, st);
    for (int step = 0; step < n_steps; ++step) {
      if (step % every == 0) {
        double *c = ckpt + (int64_t)(step / every) * 6 * n;
        for (int q = 0; q < 6; ++q) c[q * n + k] = bad ? NAN : st[q];
      }
      if (bad) continue;
      bad = !adj_advance<INC>(g, F, tb, kc, scale, sd, qm, qd, n_iter, st, nullptr, n);
    }
    for (int q = 0; q < 6; ++q) out[q * n + k] = bad ? NAN : st[q];
  }
}

// lambda <- J^T lambda and the scale's derivative. With J - 1 in pairs: lambda += (J - 1)^T
// lambda, the pairs' products in pairs on lambda scaled by the power of two that brings its
// largest entry near 1 (any magnitude keeps its bits), the others and the sums in FP64.
__device__ __forceinline__ void adj_reverse(const double *w, int64_t n, double lam[6],
                                            double &gs) {
  // inputs x1, x2, u1, u2, u3 are state rows 0, 1, 3, 4, 5; phi passes through
  const int row[5] = {0, 1, 3, 4, 5};
  if (__double_as_longlong(w[(int64_t)ADJ_FORM * n]) & 1ll) {
    double nl[JC] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int r = 0; r < 6; ++r)
#pragma unroll
      for (int c = 0; c < JC; ++c) nl[c] = fma(w[(int64_t)(r * JC + c) * n], lam[r], nl[c]);
#pragma unroll
    for (int c = 0; c < 5; ++c) lam[row[c]] = nl[c];
    gs += nl[5];
    return;
  }
  unsigned top = 0;
#pragma unroll
  for (int q = 0; q < 6; ++q)
    top = max(top, ((unsigned)__double2hiint(lam[q]) >> 20) & 0x7ffu);
  const unsigned tc = min(max(top, 1u), 2045u);
  const double down = __hiloint2double((int)((2046u - tc) << 20), 0);  // 2^(1023 - tc)
  const double up = __hiloint2double((int)(tc << 20), 0);              // 2^(tc - 1023)
  DF l[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) l[q] = df_of(lam[q] * down);
  DF nl[2] = {DF(0.0f), DF(0.0f)};
  double nd[JC] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int r = 0; r < 6; ++r)
#pragma unroll
    for (int c = 0; c < JC; ++c) {
      const double *e = w + (int64_t)(r * JC + c) * n;
      if (adj_is64(c)) {
        nd[c] = fma(*e, lam[r], nd[c]);
      } else {
        const float2 v = *reinterpret_cast<const float2 *>(e);
        nl[c] = fma_(DF(v.y, v.x), l[r], nl[c]);
      }
    }
  const bool lost = top == 0x7ffu;  // infinities and NaN stay such
#pragma unroll
  for (int c = 0; c < 2; ++c) nd[c] = df_to_double(nl[c]) * up;
#pragma unroll
  for (int c = 0; c < 5; ++c) lam[row[c]] += lost ? NAN : nd[c];
  gs += lost ? NAN : nd[5];
}

// The step's code is larger than the instruction caches: warps that wander through it apart from
// one another fetch it once each, and most of their time went to waiting for instructions (7.0 of
// 10.9 cycles between issues, with all derivatives in pairs). The barrier before each step
// keeps a block's warps together, so that a fetch serves all of them; every thread reaches it,
// particles or none. Together with one copy of the Jacobian's code for all columns that gave 39.6
// -> 31.0 ms for 65,536 orbits, 100 steps forward and back, events around repeated passes; 1 x
// 256, 2 x 256 and 4 x 128 threads per SM measured 1 to 8% slower. Barriers inside the step as well
// took twice as long (what a step keeps across them goes to local memory).
#ifndef GRPIC_ADJ_BWD_TPB
#define GRPIC_ADJ_BWD_TPB 128
#endif
#ifndef GRPIC_ADJ_BWD_BLOCKS
#define GRPIC_ADJ_BWD_BLOCKS 2
#endif
constexpr int TPB_BWD = GRPIC_ADJ_BWD_TPB;
template <bool INC>
__global__ void __launch_bounds__(TPB_BWD, GRPIC_ADJ_BWD_BLOCKS) k_adj_backward(
    const __grid_constant__ GridP g, const __grid_constant__ FieldPtrsT<double> F,
    const __grid_constant__ PushTables tb, int64_t n, double qm, double scale, double gfac,
    int n_steps, int every, int n_iter, const double *__restrict__ ckpt,
    const double *__restrict__ gout, double *__restrict__ gin, double *__restrict__ gscale,
    double *__restrict__ scratch) {
  const IncC kc = inc_c(g);
  const DF sd = df_of(scale), qd = df_of(qm);
  const int n_seg = (n_steps + every - 1) / every;
  for (int64_t k0 = blockIdx.x * (int64_t)blockDim.x; k0 < n; k0 += (int64_t)gridDim.x * blockDim.x) {
    const bool have = k0 + threadIdx.x < n;
    const int64_t k = have ? k0 + threadIdx.x : n - 1;
    double lam[6];
    bool zero = true;
    for (int q = 0; q < 6; ++q) {
      lam[q] = gout[q * n + k];
      zero = zero && lam[q] == 0.0;
    }
    double gs = 0.0;
    bool bad = !have;
    for (int seg = n_seg - 1; seg >= 0; --seg) {
      const int s0 = seg * every, len = min(n_steps, s0 + every) - s0;
      double st[6];
      const double *c = ckpt + (int64_t)seg * 6 * n;
      for (int q = 0; q < 6; ++q) st[q] = c[q * n + k];
      bad = bad || !inside(g, st);
      // recompute the segment from its checkpoint, keeping each step's Jacobian
      double *w = scratch + k;
      for (int j = 0; j < len; ++j) {
        __syncthreads();
        if (!bad)
          bad = !adj_advance<INC>(g, F, tb, kc, scale, sd, qm, qd, n_iter, st,
                                  w + (int64_t)j * 6 * JC * n, n);
      }
      // reverse sweep: lambda_n = J_n^T lambda_{n+1}
      for (int j = len - 1; j >= 0 && !bad; --j) adj_reverse(w + (int64_t)j * 6 * JC * n, n, lam, gs);
    }
    if (!have) continue;
    // a particle that reached a boundary has no gradient: zero where its cotangent was zero
    // (it does not enter the loss), NaN otherwise
    const double fill = zero ? 0.0 : NAN;
    for (int q = 0; q < 6; ++q) gin[q * n + k] = bad ? fill : lam[q];
    gscale[k] = bad ? fill : gs * gfac;
  }
}

// out[0] = sum of x[0..n): one block, fixed order (deterministic)
__global__ void __launch_bounds__(1024) k_sum(const double *__restrict__ x, int64_t n,
                                              double *__restrict__ out) {
  __shared__ double red[1024];
  double a = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) a += x[i];
  red[threadIdx.x] = a;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = red[0];
}

int adj_blocks(int64_t n, int tpb) {
  int64_t b = (n + tpb - 1) / tpb;
  const int64_t cap = N_SM * 32;
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

// Whether the increment form may take steps: rows away from the axes clear of the
// small-angle clamp, an iteration limit that is one (the general form takes a small one
// literally), and a charge-to-mass ratio, an amplitude and a time step whose products with
// values of order 1 stay far inside a pair's range (2^-126, 2^128).
static bool adj_inc_applies(const GridP &g, int n_iter, double qm, double scale) {
  const auto in_range = [](double x) {
    return x == 0.0 || (fabs(x) >= 0x1p-40 && fabs(x) <= 0x1p30);
  };
  return n_iter >= INC_MIN_ITER && g.small_angle < g.dth && in_range(qm) && in_range(scale) &&
         g.dt >= 0x1p-40 && g.dt <= 0x1p30;
}

cudaError_t launch_adjoint_forward(const GridP &g, const FieldPtrsT<double> &F,
                                   const PushTables &tb, int64_t n, double qm, double scale,
                                   int n_steps, int every, int n_iter, const double *st0,
                                   double *out, double *ckpt, cudaStream_t st) {
  if (n <= 0) return cudaGetLastError();
  const auto kernel = adj_inc_applies(g, n_iter, qm, scale) ? k_adj_forward<true> : k_adj_forward<false>;
  kernel<<<adj_blocks(n, TPB_ADJ), TPB_ADJ, 0, st>>>(g, F, tb, n, qm, scale, n_steps, every,
                                                     n_iter, st0, out, ckpt);
  COUNT_LAUNCH(1);
  return cudaGetLastError();
}

cudaError_t launch_adjoint_backward(const GridP &g, const FieldPtrsT<double> &F,
                                    const PushTables &tb, int64_t n, double qm, double scale,
                                    double gfac, int n_steps, int every, int n_iter,
                                    const double *ckpt, const double *gout, double *gin,
                                    double *gscale_pp, double *gscale_sum, double *scratch,
                                    cudaStream_t st) {
  if (n <= 0) return cudaMemsetAsync(gscale_sum, 0, sizeof(double), st);
  const auto kernel = adj_inc_applies(g, n_iter, qm, scale) ? k_adj_backward<true> : k_adj_backward<false>;
  kernel<<<adj_blocks(n, TPB_BWD), TPB_BWD, 0, st>>>(g, F, tb, n, qm, scale, gfac, n_steps, every,
                                                     n_iter, ckpt, gout, gin, gscale_pp, scratch);
  k_sum<<<1, 1024, 0, st>>>(gscale_pp, n, gscale_sum);
  COUNT_LAUNCH(2);
  return cudaGetLastError();
}
