// refine.cuh -- pieces of the implicit substeps' solvers that the particle kernels and the
// adjoint share: tests of doubles on the integer pipe, stop rules, Newton steps.
#pragma once
#include "pusher.cuh"

namespace {

// x is neither infinite nor NaN
__device__ __forceinline__ bool finite64(double x) {
  return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}
// |x| <= c and |x| < c for a constant c >= 0 (x NaN: false): the ordering of non-negative
// doubles is the ordering of their bit patterns
__device__ __forceinline__ bool abs_le(double x, double c) {
  return ((unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull) <=
         (unsigned long long)__double_as_longlong(c);
}
__device__ __forceinline__ bool abs_lt(double x, double c) {
  return ((unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull) <
         (unsigned long long)__double_as_longlong(c);
}
// x < c and x > c for a constant c > 0 (x NaN: false): as signed integers, negative doubles
// order below every positive one and positive doubles order as their bit patterns
__device__ __forceinline__ bool lt_pos(double x, double c) {
  return __double_as_longlong(x) < __double_as_longlong(c) && finite64(x);
}
__device__ __forceinline__ bool gt_pos(double x, double c) {
  return __double_as_longlong(x) > __double_as_longlong(c) && finite64(x);
}

// Stop rule of the FP32 implicit iterations: the update within ITER_TOL32 max(1, |value|),
// two FP32 ulps at 1. The remaining error, rho / (1 - rho) of that update (rho the
// contraction), is then below the rounding of the stored values.
constexpr float ITER_TOL32 = 0x1p-22f;
__device__ __forceinline__ bool settled32(float n0, float t0, float n1, float t1) {
  return fabsf(n0 - t0) <= ITER_TOL32 * fmaxf(1.0f, fabsf(n0)) &&
         fabsf(n1 - t1) <= ITER_TOL32 * fmaxf(1.0f, fabsf(n1));
}
// The coordinate iteration may also stop on an estimate of its remaining error: two successive
// updates d_prev, d of a linearly converging iteration give its rate as about d / d_prev, so
// the error left after the latest one is about d^2 / d_prev. Stop when sixteen times that is
// below ITER_TOL32 (cell units). After the first metric evaluation at the midpoint, d_prev is
// the particle's whole move and d about rho times it (rho ~ dt |dV/dx|, 1e-3 or less off the
// guard zones), so most warps stop there instead of running a third evaluation for the few
// lanes whose update is still above the plain rule's bound.
__device__ __forceinline__ bool settled32_rate(float d, float d_prev) {
  return 16.0f * d * d <= ITER_TOL32 * d_prev;
}

// |n - t| <= tol max(1, |n|): the difference in FP64 (n and t agree to about tol), the test
// in FP32 on truncated values (the bound moves by less than 2^-22 of itself)
__device__ __forceinline__ bool converged(double n, double t, float tol) {
  return fabsf(f32_trunc(n - t)) <= tol * fmaxf(1.0f, fabsf(f32_trunc(n)));
}
// the largest eigenvalue modulus of a 2 x 2 matrix: the asymptotic contraction of a map
// with that Jacobian
__device__ __forceinline__ float spectral_radius(const float J[2][2]) {
  const float tr = J[0][0] + J[1][1], det = fmaf(J[0][0], J[1][1], -J[0][1] * J[1][0]);
  const float disc = fmaf(tr, tr, -4.0f * det);
  return disc >= 0.0f ? 0.5f * (fabsf(tr) + sqrtf(disc)) : sqrtf(fmaxf(det, 0.0f));
}
// Whether the method's n_iter iterations from its start come within a tenth of tol of the
// fixed point, so that the refined result stands for the method's n_iter result: d1 is the
// method's first update (from the FP32 predictor's first step), rho the contraction (the
// spectral radius of J), the remainder d1 rho^n_iter.
__device__ __forceinline__ bool method_converges(float d1, float rho, int n_iter, float tol,
                                                 double s0, double s1) {
  if (!(rho < 0.5f)) return false;
  if (!(rho > 0.0f)) return true;
  const float scale = fmaxf(1.0f, fmaxf(fabsf(f32_trunc(s0)), fabsf(f32_trunc(s1))));
  return d1 * exp2f((float)n_iter * log2f(rho)) <= 0.1f * tol * scale;
}
// t + (I - J)^{-1} (n - t): the Newton step of t = G(t) from the residual n - t; the plain
// iteration step (n itself) when the result is not finite
__device__ __forceinline__ void newton_step(const float J[2][2], double t0, double t1, double n0,
                                            double n1, double &s0, double &s1) {
  const float a = 1.0f - J[0][0], d = 1.0f - J[1][1];
  const float idet = 1.0f / fmaf(a, d, -J[0][1] * J[1][0]);
  const double r0 = n0 - t0, r1 = n1 - t1;
  s0 = t0 + fma(f64_widen(idet * d), r0, f64_widen(idet * J[0][1]) * r1);
  s1 = t1 + fma(f64_widen(idet * J[1][0]), r0, f64_widen(idet * a) * r1);
  if (!(finite64(s0) && finite64(s1))) {
    s0 = n0;
    s1 = n1;
  }
}

__device__ __forceinline__ DF df_half(DF a) { return DF(0.5f * a.hi, 0.5f * a.lo); }

// t + (I - J)^{-1} (n - t) in pairs, the matrix from the FP32 Jacobian
__device__ __forceinline__ void newton_df(const float J[2][2], DF t0, DF t1, DF n0, DF n1,
                                          DF &s0, DF &s1) {
  const float a = 1.0f - J[0][0], d = 1.0f - J[1][1];
  const float idet = 1.0f / fmaf(a, d, -J[0][1] * J[1][0]);
  const DF r0 = n0 - t0, r1 = n1 - t1;
  s0 = t0 + (DF(idet * d) * r0 + DF(idet * J[0][1]) * r1);
  s1 = t1 + (DF(idet * J[1][0]) * r0 + DF(idet * a) * r1);
}

// dt/2 times the derivative of the coordinate velocity V of Eq. (discretized-geodesic-x) at
// the point of L for the momentum u: the Jacobian of the map t -> x^n + dt V((x^n + t)/2).
// V^1 = (alpha/gamma) (h^11 u_1 + h^13 u_3) - beta^1, V^2 = (alpha/gamma) h^22 u_2, with
// alpha/gamma = (q / alpha^2)^(-1/2), q = m2 + h^ij u_i u_j.
__device__ __forceinline__ void coord_jacobian(const GridP &g, const Local<float> &L,
                                               const float u[3], float m2, float J[2][2]) {
  const Geo<float> &o = L.G;
  const float uu = 2.0f * u[0] * u[2], u00 = u[0] * u[0], u11 = u[1] * u[1], u22 = u[2] * u[2];
  const float q = fmaf(o.H11, u00, fmaf(o.H22, u11, fmaf(o.H33, u22, fmaf(o.H13, uu, m2))));
  const float ag = rsqrtf(o.opz * q);
  const float w1 = fmaf(o.H11, u[0], o.H13 * u[2]), w2 = o.H22 * u[1];
  const float ia = L.alpha * o.opz;           // 1 / alpha
  const float hq = 0.5f * ag * ag * o.opz;    // 1 / (2 q)
  const float hdt = 0.5f * g.f_dt;
  const float dH11[2] = {L.d1H11, L.d2H11}, dH22[2] = {L.d1H22, L.d2H22};
  const float dH33[2] = {L.d1H33, L.d2H33}, dH13[2] = {L.d1H13, L.d2H13};
  const float dal[2] = {L.d1alpha, L.d2alpha}, dbe[2] = {L.d1beta1, L.d2beta1};
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float dq = fmaf(dH11[j], u00, fmaf(dH22[j], u11, fmaf(dH33[j], u22, dH13[j] * uu)));
    const float dag = ag * fmaf(dal[j], ia, -dq * hq);
    J[0][j] = hdt * (fmaf(dag, w1, ag * fmaf(dH11[j], u[0], dH13[j] * u[2])) - dbe[j]);
    J[1][j] = hdt * fmaf(dag, w2, ag * dH22[j] * u[1]);
  }
}

}  // namespace
