// push_inc.cuh -- one particle of the FP64 path in the increment form (inc.cuh), included by
// particles.cu.
#pragma once
#include "inc.cuh"

namespace {

// An FP32 estimate of whether a Boris half step stays below INC_MAX (fields of one node, no
// interpolation): where it does not, the warp goes to push64 at once. Only speed depends on it.
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

// Whether a particle is likely to take the increment form: off the axis rows (where the
// refined iterations do not apply either), and with small increments.
__device__ __forceinline__ bool inc_fit(const GridP &g, const FieldPtrsT<double> &F,
                                        const PushTables &tb, const SpeciesDevT<double> &s,
                                        int64_t kp) {
  const int i1 = s.i1[kp], i2 = s.i2[kp];
  return i2 >= 2 && i2 < g.n_th - 2 && i1 >= 0 && i1 < g.n_r &&
         (s.m2 == 0.0 || inc_small(g, F, tb, i1, i2, s.f_qm));
}

// floor of t in (-2, 2), on the integer pipe
__device__ __forceinline__ int inc_cell(double t) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(t);
  const unsigned long long a = b & 0x7fffffffffffffffull, one = 0x3ff0000000000000ull;
  if (a == b) return a >= one ? 1 : 0;
  return a == 0 ? 0 : (a > one ? -2 : -1);
}

// One particle (inc_fit) in the increment form; false: nothing stored, push64 has to take it.
template <bool DEPOSIT>
__device__ __forceinline__ bool push_inc(const GridP &g, const FieldPtrsT<double> &F,
                                         const PushTables &tb, const SpeciesDevT<double> &s,
                                         int64_t kp, unsigned long long *diag) {
  const int i1 = s.i1[kp], i2 = s.i2[kp];
  const bool em = s.m2 != 0.0;
  const double dx1 = s.dx1[kp], dx2 = s.dx2[kp];
  const IncC k = inc_c(g);
  const DF o1 = df_of(dx1), o2 = df_of(dx2);
  const double u64[3] = {s.u1[kp], s.u2[kp], s.u3[kp]};
  const DF u[3] = {df_of(u64[0]), df_of(u64[1]), df_of(u64[2])};
  DF du[3] = {DF(0.0f), DF(0.0f), DF(0.0f)};
  {
    Local<DF> L;
    {
      DF r, sn, cs;
      if (!inc_point(k, tb, i1, i2, o1, o2, r, sn, cs)) return false;
      inc_local(k, r, sn, cs, L);
    }
    DF eD[3], eB[3];
    if (em) {
      IncLerp l;
      inc_lerp(i1, i2, o1, o2, l);
      const DF e = df_scale(df_of(s.qm) * L.alpha * k.dt, 0.25f);  // half of qm alpha dt/2
      DF V[3] = {inc_interp(F.Bn[0], g.NX, l, 0, 1), inc_interp(F.Bn[1], g.NX, l, 1, 0),
                 inc_interp(F.Bn[2], g.NX, l, 1, 1)};
      vec_hat(L, V, eB);
      V[0] = inc_interp(F.D[0], g.NX, l, 1, 0);
      V[1] = inc_interp(F.D[1], g.NX, l, 0, 1);
      V[2] = inc_interp(F.D[2], g.NX, l, 0, 0);
      vec_hat(L, V, eD);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        eB[q] = e * eB[q];
        eD[q] = e * eD[q];
      }
      if (!inc_boris(L, eD, eB, u, du)) return false;
    }
    const float m2f = em ? 1.0f : 0.0f;
    DF un[3] = {u[0] + du[0], u[1] + du[1], u[2] + du[2]};
    if (!inc_geodesic(g, k, L, un, m2f, du[0], du[1])) return false;
    if (em) {
      un[0] = u[0] + du[0];
      un[1] = u[1] + du[1];
      if (!inc_boris(L, eD, eB, un, du)) return false;
    }
  }
  const double un[3] = {u64[0] + df_to_double(du[0]), u64[1] + df_to_double(du[1]),
                        u64[2] + df_to_double(du[2])};
  const DF ud[3] = {u[0] + du[0], u[1] + du[1], u[2] + du[2]};
  double t1, t2, v3;
  if (!inc_coord<false>(g, k, tb, g.n_iter, g.f_iter_tol, i1, i2, dx1, dx2, o1, o2, un, ud, s.m2,
                        em ? 1.0f : 0.0f, t1, t2, v3))
    return false;
  if (!(finite64(un[0]) && finite64(un[1]) && finite64(un[2]))) return false;
  const int c1 = inc_cell(t1), c2 = inc_cell(t2);
  const int j1 = i1 + c1, j2 = i2 + c2;
  if (j2 < 0 || j2 >= g.n_th) return false;
  const double e1 = t1 - (double)c1, e2 = t2 - (double)c2;
  s.i1[kp] = j1; s.i2[kp] = j2; s.dx1[kp] = e1; s.dx2[kp] = e2;
  s.u1[kp] = un[0]; s.u2[kp] = un[1]; s.u3[kp] = un[2];
  if (j1 < 0) { s.tag[kp] = 2; count(diag, DG_LEFT_INNER); }
  else if (j1 >= g.n_r) { s.tag[kp] = 2; count(diag, DG_LEFT_OUTER); }
  s.phi[kp] = s.phi[kp] + g.dt * v3;
  if (DEPOSIT)
    deposit64(g, F, s.qc * s.w[kp], i1, i2, i1 + dx1, i2 + dx2, j1, j2, j1 + e1, j2 + e2, v3);
  return true;
}

}  // namespace
