// dual_df.cuh -- pairs of floats (dfloat.cuh) with their derivatives along two directions,
// the derivatives pairs too: what the adjoint differentiates the pusher's increment form
// (inc.cuh) with. Only the operations that form uses are defined.
#pragma once
#include "dfloat.cuh"

namespace {

struct D2F {
  DF v, d0, d1;
  D2F() = default;
  __device__ __forceinline__ D2F(DF a) : v(a), d0(0.0f), d1(0.0f) {}
  __device__ __forceinline__ D2F(float a) : v(a), d0(0.0f), d1(0.0f) {}
  __device__ __forceinline__ D2F(DF a, DF x, DF y) : v(a), d0(x), d1(y) {}
};

__device__ __forceinline__ D2F operator+(D2F a, D2F b) {
  return D2F(a.v + b.v, a.d0 + b.d0, a.d1 + b.d1);
}
__device__ __forceinline__ D2F operator+(D2F a, DF b) { return D2F(a.v + b, a.d0, a.d1); }
__device__ __forceinline__ D2F operator-(D2F a) { return D2F(-a.v, -a.d0, -a.d1); }
__device__ __forceinline__ D2F operator-(D2F a, D2F b) { return a + (-b); }
__device__ __forceinline__ D2F operator-(D2F a, DF b) { return a + (-b); }
__device__ __forceinline__ D2F operator*(D2F a, D2F b) {
  return D2F(a.v * b.v, fma_(a.d0, b.v, a.v * b.d0), fma_(a.d1, b.v, a.v * b.d1));
}
__device__ __forceinline__ D2F operator*(DF a, D2F b) { return D2F(a * b.v, a * b.d0, a * b.d1); }
__device__ __forceinline__ D2F operator*(D2F a, DF b) { return b * a; }
__device__ __forceinline__ D2F fma_(D2F a, D2F b, D2F c) {
  return D2F(fma_(a.v, b.v, c.v), fma_(a.d0, b.v, fma_(a.v, b.d0, c.d0)),
             fma_(a.d1, b.v, fma_(a.v, b.d1, c.d1)));
}
__device__ __forceinline__ D2F fma_(DF a, D2F b, D2F c) {
  return D2F(fma_(a, b.v, c.v), fma_(a, b.d0, c.d0), fma_(a, b.d1, c.d1));
}
__device__ __forceinline__ D2F fma_(D2F a, DF b, D2F c) { return fma_(b, a, c); }
__device__ __forceinline__ D2F df_scale(D2F a, float p2) {
  return D2F(df_scale(a.v, p2), df_scale(a.d0, p2), df_scale(a.d1, p2));
}
__device__ __forceinline__ D2F df_rcp(D2F b) {
  const DF r = df_rcp(b.v), k = -(r * r);
  return D2F(r, k * b.d0, k * b.d1);
}
__device__ __forceinline__ D2F df_rsqrt(D2F x) {
  const DF r = df_rsqrt(x.v), k = df_scale(r * r * r, -0.5f);
  return D2F(r, k * x.d0, k * x.d1);
}
__device__ __forceinline__ D2F rsqrt_(D2F x) { return df_rsqrt(x); }

}  // namespace
