// fields.cu -- metric tables, initial fields and the GR field solver of Sec. 3.3 of
// arXiv:2511.17701 (Faraday, Ampere, auxiliary E and H with volume-weighted averages,
// axis treatment, horizon layer and absorbing layer), plus the loop steps 2 and 5-8 of
// Sec. 3.4. Grid work is a small fraction of a step at the particle counts this library
// targets (tens of particles per cell): one thread per grid point, metric from tables.
#include "grpic_internal.cuh"

namespace {

constexpr int TPB = 256;

// ---------------------------------------------------------------------------------
// Coefficient tables of the field solver, T_... (grpic_internal.cuh): per component of
// Eqs. (discretized-auxE), (discretized-auxH) the factor of every field value that enters it
// (alpha h_ii; alpha sqrt(h~) h_13 / (2 sqrt(h~)) and sqrt(h~ h) beta^1 / (2 sqrt(h~)) of both
// neighbours of an average), and dt / sqrt(h) of the curls, each formed in FP64 and rounded
// once; the polar area A(x1) = dr (r^2 + a^2) sqrt(1 + 2 M r/(r^2 + a^2))
// (1 - cos(theta(x2 = 1/2))) (App. A, per unit phi; theta(1/2) = dtheta/2 on the plain grid).
//
// Why whole coefficients: GB300's FP64 rate is 2 operations per clock and SM, so on 2048^2
// points one FP64 operation per point costs 8 us, as much as 1.6 planes of HBM traffic. With
// the metric factors tabulated one by one (alpha, h_11, h_22, h_33, weights) an auxiliary-field
// kernel took ~50 FP64 operations per point and 13 table planes; a component as a sum of
// coefficient x field products takes 11 and 11. With the boundary writes folded into the
// curl kernels (put, below) and the launches that read the same fields merged, a vacuum step
// on 2048^2 points went from 2220 to 1025 us in FP64, one on 500 x 300 points in FP32 (bound by
// launches) from 90 to 49 us: 7 launches a step where there were 18.
//
// FP32 planes keep the metric factors one by one (MetricTab): their kernels are bound by HBM
// and launches, not by arithmetic, and next to the axes the curls amplify every FP32 rounding,
// so that a regrouping moves a run's small components (B^3 of the 2048^2 workload after 10
// steps: by up to 8.4e-4 of its rms) without making them better.
// ---------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T tabv(const T *tab, int64_t ps, int q, int64_t k) {
  return __ldg(tab + q * ps + k);
}

// FP32: the factor q of Yee class cls
struct MetricTab {
  const float *tab;
  int64_t ps;
  __device__ __forceinline__ float operator()(int cls, int q, int64_t k) const {
    return __ldg(tab + (int64_t)(cls * M_NQ + q) * ps + k);
  }
};
// v + dt c / sqrt(h) at the points of a component: T_... in FP64, 1/sqrt(h) of Yee class cls in
// FP32 (in the order of operations of the factors one by one)
__device__ __forceinline__ double curl_step(const GridP &, const double *tab, int64_t ps, int q,
                                            int, int64_t k, double c, double v) {
  return fma(c, tabv(tab, ps, q, k), v);
}
__device__ __forceinline__ float curl_step(const GridP &g, const float *tab, int64_t ps, int,
                                           int cls, int64_t k, float c, float v) {
  return fmaf((float)g.dt * c, MetricTab{tab, ps}(cls, M_ISH, k), v);
}

// The absorbing layer (MATCH, Sec. 3.3.3): a field value v relaxes towards its initial value
// vi as v - k (v - vi), k = absorb_coef x^3, x = (r - r_absorb) / (r_max - r_absorb) capped at
// 1, beyond r_absorb. k depends on x1 alone, so it is tabulated per column.
__device__ __forceinline__ double absorb_factor(const GridP &g, double x1) {
  if (!(g.r_absorb < g.r_max)) return 0.0;
  const double r = g.r0 + map_e(g, x1);
  if (r <= g.r_absorb) return 0.0;
  double x = (r - g.r_absorb) / (g.r_max - g.r_absorb);
  x = fmin(x, 1.0);
  return g.absorb_coef * x * x * x;
}

// the polar area and the absorbing layer's factors of column i
template <typename T>
__device__ __forceinline__ void polar_row(const GridP &g, int i, T *polar) {
  const double e = map_e(g, i + 0.5), r = g.r0 + e, a2 = g.a * g.a;
  polar[i + G_] = (T)(g.dxi * e * (r * r + a2) * sqrt(1.0 + 2.0 * g.M * r / (r * r + a2)) *
                      (1.0 - cos(map_theta(g, 0.5))));
  polar[g.NX + i + G_] = (T)absorb_factor(g, i);
  polar[2 * g.NX + i + G_] = (T)absorb_factor(g, i + 0.5);
}

// Each lane evaluates the metric at its column's four Yee points and takes the averaged terms of
// the columns next to it from its neighbours: a warp covers 30 columns of a row.
__global__ void k_metric_tables(GridP g, double *tab, double *polar) {
  constexpr unsigned FULL = 0xffffffffu;
  const int64_t ps = plane_size(g);
  const int lane = threadIdx.x & 31, tiles = (g.NX + 29) / 30;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
  for (int64_t t = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
       t < (int64_t)tiles * g.NY; t += warps) {
    const int i = (int)(t % tiles) * 30 + lane - 1 - G_, j = (int)(t / tiles) - G_;
    MetricV nn, hn, nh, hh;
    metric_eval<false>(g, i, j, false, nn, nullptr);
    metric_eval<false>(g, i + 0.5, j, false, hn, nullptr);
    metric_eval<false>(g, i, j + 0.5, false, nh, nullptr);
    metric_eval<false>(g, i + 0.5, j + 0.5, false, hh, nullptr);
    // [sqrt(h~) h_13] and [sqrt(h~ h) beta^1] here and at the neighbours half a cell away
    const auto t13 = [](const MetricV &m) { return m.sqrt_ht * m.h13; };
    const auto tb1 = [](const MetricV &m) { return m.sqrt_ht * m.sqrt_h * m.beta1; };
    const double nn13 = t13(nn), nnb = tb1(nn), hn13 = t13(hn), hnb = tb1(hn);
    const double nh13 = t13(nh), nhb = tb1(nh), hh13 = t13(hh), hhb = tb1(hh);
    const double hn13l = __shfl_up_sync(FULL, hn13, 1), hnbl = __shfl_up_sync(FULL, hnb, 1);
    const double hh13l = __shfl_up_sync(FULL, hh13, 1), hhbl = __shfl_up_sync(FULL, hhb, 1);
    const double nn13r = __shfl_down_sync(FULL, nn13, 1), nnbr = __shfl_down_sync(FULL, nnb, 1);
    const double nh13r = __shfl_down_sync(FULL, nh13, 1), nhbr = __shfl_down_sync(FULL, nhb, 1);
    if (lane == 0 || lane == 31 || i > g.n_r + G_) continue;
    double *o = tab + sidx(g, i, j);
    double w = 0.5 / nn.sqrt_ht, wa = w * nn.alpha;
    o[T_E3D3 * ps] = nn.alpha * nn.h33;
    o[T_E3D1L * ps] = wa * hn13l;
    o[T_E3D1R * ps] = wa * hn13;
    o[T_E3B2L * ps] = w * hnbl;
    o[T_E3B2R * ps] = w * hnb;
    o[T_D3 * ps] = g.dt / nn.sqrt_h;
    w = 0.5 / hn.sqrt_ht;
    wa = w * hn.alpha;
    o[T_E1D1 * ps] = hn.alpha * hn.h11;
    o[T_E1D3L * ps] = wa * nn13;
    o[T_E1D3R * ps] = wa * nn13r;
    o[T_H2B2 * ps] = hn.alpha * hn.h22;
    o[T_H2D3L * ps] = w * nnb;
    o[T_H2D3R * ps] = w * nnbr;
    o[T_B2D1 * ps] = g.dt / hn.sqrt_h;
    w = 0.5 / nh.sqrt_ht;
    wa = w * nh.alpha;
    o[T_E2D2 * ps] = nh.alpha * nh.h22;
    o[T_E2B3L * ps] = w * hhbl;
    o[T_E2B3R * ps] = w * hhb;
    o[T_H1B1 * ps] = nh.alpha * nh.h11;
    o[T_H1B3L * ps] = wa * hh13l;
    o[T_H1B3R * ps] = wa * hh13;
    o[T_B1D2 * ps] = g.dt / nh.sqrt_h;
    w = 0.5 / hh.sqrt_ht;
    wa = w * hh.alpha;
    o[T_H3B3 * ps] = hh.alpha * hh.h33;
    o[T_H3B1L * ps] = wa * nh13;
    o[T_H3B1R * ps] = wa * nh13r;
    o[T_H3D2L * ps] = w * nhb;
    o[T_H3D2R * ps] = w * nhbr;
    o[T_B3 * ps] = g.dt / hh.sqrt_h;
    if (j == 0) polar_row(g, i, polar);
  }
}

// alpha, h_11, h_22, h_33, 1/(2 sqrt(h~)), [sqrt(h~) h_13], [sqrt(h~ h) beta^1] and 1/sqrt(h) per
// Yee class, and the polar rows
__global__ void k_metric_tables(GridP g, float *tab, float *polar) {
  const int64_t ps = plane_size(g);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 4 * ps;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int cls = (int)(t / ps);
    const int64_t q = t - cls * ps;
    const int i = (int)(q % g.NX) - G_, j = (int)(q / g.NX) - G_;
    const double s1 = (cls == CLS_HN || cls == CLS_HH) ? 0.5 : 0.0;
    const double s2 = (cls == CLS_NH || cls == CLS_HH) ? 0.5 : 0.0;
    MetricV m;
    metric_eval<false>(g, i + s1, j + s2, false, m, nullptr);
    float *o = tab + (int64_t)cls * M_NQ * ps + q;
    o[M_ALPHA * ps] = (float)m.alpha;
    o[M_H11 * ps] = (float)m.h11;
    o[M_H22 * ps] = (float)m.h22;
    o[M_H33 * ps] = (float)m.h33;
    o[M_IHT2 * ps] = (float)(0.5 / m.sqrt_ht);
    o[M_WT13 * ps] = (float)(m.sqrt_ht * m.h13);
    o[M_WB1 * ps] = (float)(m.sqrt_ht * m.sqrt_h * m.beta1);
    o[M_ISH * ps] = (float)(1.0 / m.sqrt_h);
    if (cls == CLS_HN && j == 0) polar_row(g, i, polar);
  }
}

// dt = cfl * min over cell centres of 1 / (alpha sqrt(h^11 + h^22) + |beta^1|); positive
// doubles order like their bit patterns, so the minimum is an integer atomicMin.
__global__ void k_dt_min(GridP g, unsigned long long *out) {
  __shared__ unsigned long long sm[TPB];
  unsigned long long best = 0x7FF0000000000000ull;  // +inf
  const int64_t n = (int64_t)g.n_r * g.n_th;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % g.n_r), j = (int)(t / g.n_r);
    MetricV m;
    metric_eval<false>(g, i + 0.5, j + 0.5, false, m, nullptr);
    const double v = 1.0 / (m.alpha * sqrt(m.H11 + m.H22) + fabs(m.beta1));
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    best = b < best ? b : best;
  }
  sm[threadIdx.x] = best;
  __syncthreads();
  for (int s = TPB / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s && sm[threadIdx.x + s] < sm[threadIdx.x]) sm[threadIdx.x] = sm[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicMin(out, sm[0]);
}

// D at a Yee point from the inverse of Eq. (aux) with E_i = d_i A_0, E_3 = 0 and
// sqrt(h) B^2 = -d_1 A_3, sqrt(h) B^3 = -d_2 A_1 (no division by sqrt(h) on the axis).
__device__ void d_from_potential(const GridP &g, int kind, double B0, double x1, double x2,
                                 int comp, double &out) {
  Pot p;
  potential(g, kind, B0, x1, x2, true, p);
  MetricV m;
  metric_eval<false>(g, x1, x2, false, m, nullptr);
  if (comp == 0) out = (m.H11 * p.d1A0 + m.H13 * m.beta1 * p.d1A3) / m.alpha;
  else if (comp == 1) out = m.H22 * (p.d2A0 - m.beta1 * p.d2A1) / m.alpha;
  else out = (m.H13 * p.d1A0 + m.H33 * m.beta1 * p.d1A3) / m.alpha;
}

__device__ double inv_sqrt_h(const GridP &g, double x1, double x2) {
  MetricV m;
  metric_eval<false>(g, x1, x2, false, m, nullptr);
  return 1.0 / m.sqrt_h;
}

// theta_j + theta_{j+1} and theta_{j+1} - theta_j of two face rows; with h0 the cubic's
// difference p(eta + d) - p(eta) = d (pi^2 - 6 pi eta + 6 eta^2) + d^2 (6 eta - 3 pi) + 2 d^3
// (p(eta) = eta (pi - 2 eta)(pi - eta)) is expanded so that nothing cancels
__device__ double theta_sum(const GridP &g, int j) {
  const double de = g.dth, e0 = j * de, e1 = (j + 1) * de, k = 2.0 * g.h0 / (GRPIC_PI * GRPIC_PI);
  const double p0 = e0 * (GRPIC_PI - 2.0 * e0) * (GRPIC_PI - e0);
  const double p1 = e1 * (GRPIC_PI - 2.0 * e1) * (GRPIC_PI - e1);
  return (2 * j + 1) * de + k * (p0 + p1);
}
__device__ double theta_diff(const GridP &g, int j) {
  const double de = g.dth, e0 = j * de, k = 2.0 * g.h0 / (GRPIC_PI * GRPIC_PI);
  return de + k * (de * (GRPIC_PI * GRPIC_PI - 6.0 * GRPIC_PI * e0 + 6.0 * e0 * e0) +
                   de * de * (6.0 * e0 - 3.0 * GRPIC_PI) + 2.0 * de * de * de);
}

// A_1(x1, theta_{j+1}) - A_1(x1, theta_j) of the Wald potential (Eq. Wald) for the discrete
// curl that gives B^3, in product form: with A_1 = (B0/2) a f (2 M r (1 + cos^2)/Sigma -
// sin^2) and sin^2(b) - sin^2(a) = sin(b - a) sin(b + a) = -(cos^2(b) - cos^2(a)),
//   dA_1 = -(B0/2) a f D (1 + 2 M r (r^2 - a^2) / (Sigma_a Sigma_b)),
//   D = sin(theta_{j+1} - theta_j) sin(theta_{j+1} + theta_j);
// the plain difference loses ~1/dth^2 of its digits next to the axes (A_1 ~ theta^2 there).
// A_3(x1, theta_{j+1}) - A_3(x1, theta_j) for the discrete curl that gives B^1; for the
// monopole, -B0 (cos(theta_{j+1}) - cos(theta_j)) = 2 B0 sin((theta_j + theta_{j+1}) / 2)
// sin((theta_{j+1} - theta_j) / 2) in product form (the plain difference of the cosines
// loses ~1/dth^2 of its digits next to the axes)
__device__ double dA3_theta(const GridP &g, int kind, double B0, int i, int j) {
  if (kind == GRPIC_FIELD_MONOPOLE)
    return 2.0 * B0 * sin(0.5 * theta_sum(g, j)) * sin(0.5 * theta_diff(g, j));
  Pot pa, pb;
  potential(g, kind, B0, i, j, false, pa);
  potential(g, kind, B0, i, j + 1, false, pb);
  return pb.A3 - pa.A3;
}

__device__ double dA1_theta(const GridP &g, int kind, double B0, double x1, int j) {
  if (kind != GRPIC_FIELD_WALD) return 0.0;  // the vertical field has A_1 = 0
  const double a = g.a, M = g.M;
  const double e = map_e(g, x1), r = g.r0 + e, f = g.dxi * e;
  const double ca = cos(map_theta(g, j)), cb = cos(map_theta(g, j + 1));
  const double Sa = r * r + a * a * ca * ca, Sb = r * r + a * a * cb * cb;
  const double D = sin(theta_diff(g, j)) * sin(theta_sum(g, j));
  return -0.5 * B0 * a * f * D * (1.0 + 2.0 * M * r * (r * r - a * a) / (Sa * Sb));
}

template <typename T>
__global__ void k_init_fields(GridP g, FieldPtrsT<T> F, int kind, double B0) {
  const int ni = g.n_r + 2 * G_ + 1, nj = g.n_th + 1;
  const int64_t n = (int64_t)ni * nj;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % ni) - G_, j = (int)(t / ni);
    const int64_t k = sidx(g, i, j);
    const bool axis = (j == 0 || j == g.n_th);
    Pot pa, pb;
    if (j < g.n_th) {
      F.B[0][k] = (T)(dA3_theta(g, kind, B0, i, j) * inv_sqrt_h(g, i, j + 0.5));
      F.B[2][k] = (T)(-dA1_theta(g, kind, B0, i + 0.5, j) * inv_sqrt_h(g, i + 0.5, j + 0.5));
      double d;
      d_from_potential(g, kind, B0, i, j + 0.5, 1, d);
      F.D[1][k] = (T)d;
    }
    if (!axis) {
      potential(g, kind, B0, i, j, false, pa);
      potential(g, kind, B0, i + 1, j, false, pb);
      F.B[1][k] = (T)(-(pb.A3 - pa.A3) * inv_sqrt_h(g, i + 0.5, j));
      double d;
      d_from_potential(g, kind, B0, i, j, 2, d);
      F.D[2][k] = (T)d;
    } else {
      F.B[1][k] = (T)0;
      F.D[2][k] = (T)0;
    }
    double d0;
    d_from_potential(g, kind, B0, i + 0.5, j, 0, d0);
    F.D[0][k] = (T)d0;
  }
}

// ---------------------------------------------------------------------------------
// Boundary conditions (Sec. 3.3.3).
// ---------------------------------------------------------------------------------
// Horizon layer: cells i1 in [-G, n_f] copy cell n_f + 1, all rows.
template <typename T>
__global__ void k_horizon(GridP g, T *p0, T *p1, T *p2) {
  const int nl = g.n_f + 1 + G_, nj = g.NY;
  const int64_t n = (int64_t)nl * nj * 3;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t / ((int64_t)nl * nj));
    const int64_t q = t - c * (int64_t)nl * nj;
    const int i = (int)(q % nl) - G_, j = (int)(q / nl) - G_;
    T *p = c == 0 ? p0 : (c == 1 ? p1 : p2);
    p[sidx(g, i, j)] = p[sidx(g, g.n_f + 1, j)];
  }
}

// Axis ghost rows by reflection (Fig. 1): r components even, theta and phi components
// odd; half rows (x2 = j + 1/2) and node rows mirror differently. isB selects the B
// classes (B^1 half, B^2 node, B^3 half) or the D classes (D^1 node, D^2 half, D^3 node).
template <typename T>
__global__ void k_axis(GridP g, T *p0, T *p1, T *p2, int isB) {
  const int ni = g.NX;
  const int nrow = 2 * G_ + 1;  // rows written per component (2 below, 3 above)
  const int64_t n = (int64_t)ni * nrow * 3;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t / ((int64_t)ni * nrow));
    const int64_t q = t - c * (int64_t)ni * nrow;
    const int i = (int)(q % ni) - G_, rr = (int)(q / ni);
    T *p = c == 0 ? p0 : (c == 1 ? p1 : p2);
    const bool half = isB ? (c != 1) : (c == 1);
    const T par = (c == 0) ? (T)1 : (T)-1;
    const int N = g.n_th;
    if (!half) {
      if (rr < G_) {  // rows -1, -2 from 1, 2
        const int k = rr + 1;
        p[sidx(g, i, -k)] = par * p[sidx(g, i, k)];
      } else if (rr < 2 * G_) {  // rows N+1, N+2 from N-1, N-2
        const int k = rr - G_ + 1;
        p[sidx(g, i, N + k)] = par * p[sidx(g, i, N - k)];
      }
    } else {
      if (rr < G_) {  // rows -1, -2 from 0, 1
        p[sidx(g, i, -1 - rr)] = par * p[sidx(g, i, rr)];
      } else {  // rows N, N+1, N+2 from N-1, N-2, N-3
        const int k = rr - G_;
        p[sidx(g, i, N + k)] = par * p[sidx(g, i, N - 1 - k)];
      }
    }
  }
}

// ---------------------------------------------------------------------------------
// Field kernels. One thread per point of a row; a block covers TPBX x TPBY points, so no
// index is divided and the x2 neighbours of a block's rows are in its cache.
//
// Two time levels: a field that enters as the mean of two levels is read from a and b
// (MEAN), one that enters as itself from a alone; which one is known at compile time, since a
// multiplication by a weight of 1 would cost an FP64 operation per value.
// ---------------------------------------------------------------------------------
constexpr int TPBX = 64, TPBY = 4;  // the largest block

template <typename T>
struct Pair3 {
  const T *a[3], *b[3];
};
template <bool MEAN, typename T>
__device__ __forceinline__ T pv(const Pair3<T> &P, int c, int64_t k) {
  if (MEAN) return (T)0.5 * (__ldg(P.a[c] + k) + __ldg(P.b[c] + k));
  return __ldg(P.a[c] + k);
}

// v - 4 pi J
template <bool MEAN, typename T>
__device__ __forceinline__ T less_4pi_j(const Pair3<T> &J, int c, int64_t k, T v) {
  return fma((T)(-4.0 * GRPIC_PI), pv<MEAN>(J, c, k), v);
}

// E_1 at (i+1/2, j) = alpha [h_11 D^1 + <h_13 D^3>], E_3 at (i, j) = alpha [h_33 D^3 +
// <h_13 D^1>] + <sqrt(h) beta^1 B^2> (zero on the axes), E_2 at (i, j+1/2) = alpha h_22 D^2 -
// <sqrt(h) beta^1 B^3>; Eq. (discretized-auxE)
template <bool DMEAN>
__device__ __forceinline__ void aux_E(const GridP &g, const Pair3<double> &B,
                                      const Pair3<double> &D, const double *tab, int64_t ps, int j,
                                      int64_t k, double *E1, double *E2, double *E3) {
  using T = double;
  const T d1 = pv<DMEAN>(D, 0, k), d3 = pv<DMEAN>(D, 2, k);
  E1[k] = fma(tabv(tab, ps, T_E1D1, k), d1,
              fma(tabv(tab, ps, T_E1D3L, k), d3,
                  tabv(tab, ps, T_E1D3R, k) * pv<DMEAN>(D, 2, k + 1)));
  E3[k] = (j == 0 || j == g.n_th)
              ? (T)0
              : fma(tabv(tab, ps, T_E3D3, k), d3,
                    fma(tabv(tab, ps, T_E3D1L, k), pv<DMEAN>(D, 0, k - 1),
                        tabv(tab, ps, T_E3D1R, k) * d1)) +
                    fma(tabv(tab, ps, T_E3B2L, k), pv<false>(B, 1, k - 1),
                        tabv(tab, ps, T_E3B2R, k) * pv<false>(B, 1, k));
  if (j < g.n_th)
    E2[k] = fma(tabv(tab, ps, T_E2D2, k), pv<DMEAN>(D, 1, k),
                -fma(tabv(tab, ps, T_E2B3L, k), pv<false>(B, 2, k - 1),
                     tabv(tab, ps, T_E2B3R, k) * pv<false>(B, 2, k)));
}

// H_1 at (i, j+1/2) = alpha [h_11 B^1 + <h_13 B^3>], H_3 at (i+1/2, j+1/2) = alpha [h_33 B^3 +
// <h_13 B^1>] - <sqrt(h) beta^1 D^2>, H_2 at (i+1/2, j) = alpha h_22 B^2 +
// <sqrt(h) beta^1 D^3>; Eq. (discretized-auxH)
__device__ __forceinline__ void aux_H(const GridP &g, const Pair3<double> &B,
                                      const Pair3<double> &D, const double *tab, int64_t ps, int j,
                                      int64_t k, double *H1, double *H2, double *H3) {
  using T = double;
  if (j < g.n_th) {
    const T b1 = pv<false>(B, 0, k), b3 = pv<false>(B, 2, k);
    H1[k] = fma(tabv(tab, ps, T_H1B1, k), b1,
                fma(tabv(tab, ps, T_H1B3L, k), pv<false>(B, 2, k - 1),
                    tabv(tab, ps, T_H1B3R, k) * b3));
    H3[k] = fma(tabv(tab, ps, T_H3B3, k), b3,
                fma(tabv(tab, ps, T_H3B1L, k), b1,
                    tabv(tab, ps, T_H3B1R, k) * pv<false>(B, 0, k + 1))) -
            fma(tabv(tab, ps, T_H3D2L, k), pv<false>(D, 1, k),
                tabv(tab, ps, T_H3D2R, k) * pv<false>(D, 1, k + 1));
  }
  H2[k] = fma(tabv(tab, ps, T_H2B2, k), pv<false>(B, 1, k),
              fma(tabv(tab, ps, T_H2D3L, k), pv<false>(D, 2, k),
                  tabv(tab, ps, T_H2D3R, k) * pv<false>(D, 2, k + 1)));
}

// The same in FP32, from the factors one by one (explicit fused multiply-adds: a fixed order of
// roundings, see above on the axes).
__device__ __forceinline__ float two_terms(float t0, float v0, float t1, float v1, float w) {
  return fmaf(t1, v1, t0 * v0) * w;  // an average of two weighted neighbours
}
template <bool DMEAN>
__device__ __forceinline__ void aux_E(const GridP &g, const Pair3<float> &B, const Pair3<float> &D,
                                      const float *tab, int64_t ps, int j, int64_t k, float *E1,
                                      float *E2, float *E3) {
  const MetricTab m{tab, ps};
  const float d1 = pv<DMEAN>(D, 0, k), d3 = pv<DMEAN>(D, 2, k);
  E1[k] = m(CLS_HN, M_ALPHA, k) *
          fmaf(m(CLS_HN, M_H11, k), d1,
               two_terms(m(CLS_NN, M_WT13, k), d3, m(CLS_NN, M_WT13, k + 1),
                         pv<DMEAN>(D, 2, k + 1), m(CLS_HN, M_IHT2, k)));
  if (j == 0 || j == g.n_th) {
    E3[k] = 0.0f;
  } else {
    const float w2 = m(CLS_NN, M_IHT2, k);
    const float a13 = two_terms(m(CLS_HN, M_WT13, k), d1, m(CLS_HN, M_WT13, k - 1),
                                pv<DMEAN>(D, 0, k - 1), w2);
    const float ab2 = two_terms(m(CLS_HN, M_WB1, k - 1), pv<false>(B, 1, k - 1),
                                m(CLS_HN, M_WB1, k), pv<false>(B, 1, k), w2);
    E3[k] = fmaf(m(CLS_NN, M_ALPHA, k), fmaf(m(CLS_NN, M_H33, k), d3, a13), ab2);
  }
  if (j < g.n_th)
    E2[k] = fmaf(m(CLS_NH, M_ALPHA, k) * m(CLS_NH, M_H22, k), pv<DMEAN>(D, 1, k),
                 -two_terms(m(CLS_HH, M_WB1, k - 1), pv<false>(B, 2, k - 1), m(CLS_HH, M_WB1, k),
                            pv<false>(B, 2, k), m(CLS_NH, M_IHT2, k)));
}
__device__ __forceinline__ void aux_H(const GridP &g, const Pair3<float> &B, const Pair3<float> &D,
                                      const float *tab, int64_t ps, int j, int64_t k, float *H1,
                                      float *H2, float *H3) {
  const MetricTab m{tab, ps};
  if (j < g.n_th) {
    const float b1 = pv<false>(B, 0, k), b3 = pv<false>(B, 2, k), w3 = m(CLS_HH, M_IHT2, k);
    H1[k] = m(CLS_NH, M_ALPHA, k) *
            fmaf(m(CLS_NH, M_H11, k), b1,
                 two_terms(m(CLS_HH, M_WT13, k - 1), pv<false>(B, 2, k - 1), m(CLS_HH, M_WT13, k),
                           b3, m(CLS_NH, M_IHT2, k)));
    const float b13 = two_terms(m(CLS_NH, M_WT13, k), b1, m(CLS_NH, M_WT13, k + 1),
                                pv<false>(B, 0, k + 1), w3);
    const float bd2 = two_terms(m(CLS_NH, M_WB1, k), pv<false>(D, 1, k), m(CLS_NH, M_WB1, k + 1),
                                pv<false>(D, 1, k + 1), w3);
    H3[k] = fmaf(m(CLS_HH, M_ALPHA, k), fmaf(m(CLS_HH, M_H33, k), b3, b13), -bd2);
  }
  H2[k] = fmaf(m(CLS_HN, M_ALPHA, k) * m(CLS_HN, M_H22, k), pv<false>(B, 1, k),
               two_terms(m(CLS_NN, M_WB1, k), pv<false>(D, 2, k), m(CLS_NN, M_WB1, k + 1),
                         pv<false>(D, 2, k + 1), m(CLS_HN, M_IHT2, k)));
}

// The auxiliary fields on stored i in [-1, n_r + 1], rows [0, n_theta]: E, H or both (both
// read the same B and D, so one launch reads them once).
template <typename T, bool DOE, bool DOH, bool DMEAN>
__global__ void __launch_bounds__(TPBX *TPBY) k_aux(GridP g, Pair3<T> B, Pair3<T> D, const T *tab,
                                                    T *E1, T *E2, T *E3, T *H1, T *H2, T *H3) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - 1;
  const int64_t ps = plane_size(g);
  for (int j = blockIdx.y * blockDim.y + threadIdx.y; j <= g.n_th; j += gridDim.y * blockDim.y) {
    if (i > g.n_r + 1) return;
    const int64_t k = sidx(g, i, j);
    if (DOE) aux_E<DMEAN>(g, B, D, tab, ps, j, k, E1, E2, E3);
    if (DOH) aux_H(g, B, D, tab, ps, j, k, H1, H2, H3);
  }
}

// MATCH absorbing layer (reading of paper I's form): F <- F - lambda (F - F_init),
// lambda = coef min(1, ((r - r_abs)/(r_max - r_abs)))^3 for r > r_absorb, rows [0, n_theta].
// The initial value is read only inside the layer (the factor is zero elsewhere).
template <typename T>
__device__ __forceinline__ T match(const GridP &g, T v, const T *init, int64_t idx,
                                   const T *absorb, int i, int j) {
  if (j < 0 || j > g.n_th) return v;
  const T k = __ldg(absorb + i + G_);  // the factor at this column (absorb_factor)
  return k == (T)0 ? v : v - k * (v - __ldg(init + idx));
}

// Stores a point's new value together with every boundary value it determines, so that the
// curl kernels need no boundary launches (k_horizon, then k_axis): the columns [-G, n_f] of
// the horizon layer copy column n_f + 1, and the rows across the axes mirror rows inside
// (half rows -1-r <- r, n+r <- n-1-r; node rows -r <- r, n+r <- n-r) with parity par. The
// points that are written here by others are not stored by their own threads
// (boundary_point). AXIS false: the horizon layer alone.
template <bool AXIS>
__device__ __forceinline__ bool boundary_point(const GridP &g, bool half, int i, int j) {
  return i <= g.n_f || (AXIS && (j < 0 || j > g.n_th - (half ? 1 : 0)));
}
template <typename T>
__device__ __forceinline__ void put_row(const GridP &g, T *p, int i, int j, T v) {
  p[sidx(g, i, j)] = v;
  if (i == g.n_f + 1)
    for (int q = -G_; q <= g.n_f; ++q) p[sidx(g, q, j)] = v;
}
template <bool AXIS, typename T>
__device__ __forceinline__ void put(const GridP &g, T *p, bool half, T par, int i, int j, T v) {
  if (boundary_point<AXIS>(g, half, i, j)) return;
  put_row(g, p, i, j, v);
  if (!AXIS) return;
  const int N = g.n_th;
  if (half) {
    if (j < G_) put_row(g, p, i, -1 - j, par * v);
    if (N - 1 - j <= G_) put_row(g, p, i, N + (N - 1 - j), par * v);
  } else {
    if (j >= 1 && j <= G_) put_row(g, p, i, -j, par * v);
    if (N - j >= 1 && N - j <= G_) put_row(g, p, i, N + (N - j), par * v);
  }
}

// Faraday, Eq. (discretized-faraday): Bout = Bin - dt curl E / sqrt(h) on the evolved points,
// Bout = Bin elsewhere; B^2 is not evolved on the axes.
template <typename T, bool MEAN, bool MATCH>
__device__ __forceinline__ void faraday(const GridP &g, const Pair3<T> &Bin, const T *E1,
                                        const T *E2, const T *E3, const T *tab, const T *absorb,
                                        T *const B[3], T *const Bi[3], int64_t ps, int i, int j,
                                        int64_t k) {
  T b1 = pv<MEAN>(Bin, 0, k), b2 = pv<MEAN>(Bin, 1, k), b3 = pv<MEAN>(Bin, 2, k);
  const bool rows_half = (j >= 0 && j < g.n_th);
  if (rows_half && i >= 0 && i <= g.n_r) {
    const T e3 = __ldg(E3 + k);
    b1 = curl_step(g, tab, ps, T_B1D2, CLS_NH, k, -(__ldg(E3 + k + g.NX) - e3), b1);
    if (i < g.n_r) {
      if (j >= 1) b2 = curl_step(g, tab, ps, T_B2D1, CLS_HN, k, __ldg(E3 + k + 1) - e3, b2);
      b3 = curl_step(g, tab, ps, T_B3, CLS_HH, k,
                     -((__ldg(E2 + k + 1) - __ldg(E2 + k)) - (__ldg(E1 + k + g.NX) - __ldg(E1 + k))),
                     b3);
    }
  }
  if (MATCH) {
    b1 = match(g, b1, Bi[0], k, absorb, i, j);
    b2 = match(g, b2, Bi[1], k, absorb + g.NX, i, j);
    b3 = match(g, b3, Bi[2], k, absorb + g.NX, i, j);
  }
  put<true>(g, B[0], true, (T)1, i, j, b1);
  put<true>(g, B[1], false, (T)-1, i, j, b2);
  put<true>(g, B[2], true, (T)-1, i, j, b3);
}

// Ampere, Eq. (discretized-ampere): Dout = Din + dt (curl H - 4 pi J) / sqrt(h); on the
// axes D^1 follows the integral form of Sec. 3.3.2 with the polar area (reading: the
// whole radial flux into the half cell, coefficient 4 pi; -H_3 at theta = pi) and D^3
// is not evolved. MEAN: Din and J are means of two time levels, and only the horizon layer
// follows; else the absorbing layer and both boundaries do.
template <typename T, bool MEAN>
__device__ __forceinline__ void ampere(const GridP &g, const Pair3<T> &Din, const T *H1,
                                       const T *H2, const T *H3, const Pair3<T> &J, const T *tab,
                                       const T *polar, T *const D[3], T *const Di[3], int64_t ps,
                                       int i, int j, int64_t k) {
  T d1 = pv<MEAN>(Din, 0, k), d2 = pv<MEAN>(Din, 1, k), d3 = pv<MEAN>(Din, 2, k);
  if (i >= 0 && i <= g.n_r && j >= 0 && j <= g.n_th) {
    if (i < g.n_r) {
      if (j == 0)
        d1 += (T)g.dt * less_4pi_j<MEAN>(J, 0, k, __ldg(H3 + k)) / __ldg(polar + i + G_);
      else if (j == g.n_th)
        d1 += (T)g.dt * less_4pi_j<MEAN>(J, 0, k, -__ldg(H3 + k - g.NX)) / __ldg(polar + i + G_);
      else
        d1 = curl_step(g, tab, ps, T_B2D1, CLS_HN, k,
                       less_4pi_j<MEAN>(J, 0, k, __ldg(H3 + k) - __ldg(H3 + k - g.NX)), d1);
    }
    if (j < g.n_th) {
      d2 = curl_step(g, tab, ps, T_B1D2, CLS_NH, k,
                     less_4pi_j<MEAN>(J, 1, k, __ldg(H3 + k - 1) - __ldg(H3 + k)), d2);
      if (j >= 1)
        d3 = curl_step(g, tab, ps, T_D3, CLS_NN, k,
                       less_4pi_j<MEAN>(J, 2, k, (__ldg(H2 + k) - __ldg(H2 + k - 1)) -
                                                     (__ldg(H1 + k) - __ldg(H1 + k - g.NX))),
                       d3);
    }
  }
  if (!MEAN) {
    d1 = match(g, d1, Di[0], k, polar + 2 * g.NX, i, j);
    d2 = match(g, d2, Di[1], k, polar + g.NX, i, j);
    d3 = match(g, d3, Di[2], k, polar + g.NX, i, j);
  }
  put<!MEAN>(g, D[0], false, (T)1, i, j, d1);
  put<!MEAN>(g, D[1], true, (T)-1, i, j, d2);
  put<!MEAN>(g, D[2], false, (T)-1, i, j, d3);
}

template <typename T>
struct Planes3 {
  T *p[3];
};

// Every stored point. The predict's Faraday: B^{n-1} -> B^n, no absorbing layer.
template <typename T>
__global__ void __launch_bounds__(TPBX *TPBY) k_faraday(GridP g, Pair3<T> Bin, Planes3<T> E,
                                                        const T *tab, Planes3<T> Bout) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - G_;
  const int64_t ps = plane_size(g);
  for (int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - G_; j <= g.n_th + G_;
       j += gridDim.y * blockDim.y) {
    if (i > g.n_r + G_) return;
    faraday<T, true, false>(g, Bin, E.p[0], E.p[1], E.p[2], tab, nullptr, Bout.p, Bout.p, ps, i,
                            j, sidx(g, i, j));
  }
}
// Step 6's Faraday B^{n-1/2} -> B^{n+1/2} and step 7's auxiliary Ampere D^{n-1/2} ->
// D^{n+1/2}: independent of one another, one launch.
template <typename T>
__global__ void __launch_bounds__(TPBX *TPBY) k_faraday_ampere(
    GridP g, Pair3<T> Bin, Planes3<T> E, Planes3<T> Bout, Planes3<T> Bi, Pair3<T> Din,
    Planes3<T> H, Pair3<T> J, Planes3<T> Dout, const T *tab, const T *polar) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - G_;
  const int64_t ps = plane_size(g);
  for (int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - G_; j <= g.n_th + G_;
       j += gridDim.y * blockDim.y) {
    if (i > g.n_r + G_) return;
    const int64_t k = sidx(g, i, j);
    faraday<T, false, true>(g, Bin, E.p[0], E.p[1], E.p[2], tab, polar + g.NX, Bout.p, Bi.p, ps,
                            i, j, k);
    ampere<T, true>(g, Din, H.p[0], H.p[1], H.p[2], J, tab, polar, Dout.p, Dout.p, ps, i, j, k);
  }
}
// The final Ampere D^n -> D^{n+1}.
template <typename T>
__global__ void __launch_bounds__(TPBX *TPBY) k_ampere(GridP g, Pair3<T> Din, Planes3<T> H,
                                                       Pair3<T> J, const T *tab, const T *polar,
                                                       Planes3<T> Dout, Planes3<T> Di) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - G_;
  const int64_t ps = plane_size(g);
  for (int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - G_; j <= g.n_th + G_;
       j += gridDim.y * blockDim.y) {
    if (i > g.n_r + G_) return;
    ampere<T, false>(g, Din, H.p[0], H.p[1], H.p[2], J, tab, polar, Dout.p, Di.p, ps, i, j,
                     sidx(g, i, j));
  }
}

template <typename T>
__global__ void k_copy3(int64_t n, const T *a0, const T *a1, const T *a2, T *b0, T *b1, T *b2) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x) {
    b0[t] = a0[t]; b1[t] = a1[t]; b2[t] = a2[t];
  }
}

template <typename T>
__global__ void k_zero(T *p, int64_t n) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n;
       t += (int64_t)gridDim.x * blockDim.x)
    p[t] = (T)0;
}

int blocks_for(int64_t n) {
  int64_t b = (n + TPB - 1) / TPB;
  if (b > N_SM * 32) b = N_SM * 32;
  return (int)(b < 1 ? 1 : b);
}

template <typename T>
Pair3<T> pair(T *const p[3], T *const q[3]) {
  Pair3<T> P;
  for (int c = 0; c < 3; ++c) { P.a[c] = p[c]; P.b[c] = q[c]; }
  return P;
}
template <typename T>
Pair3<T> one(T *const p[3]) {
  return pair(p, p);
}
template <typename T>
Planes3<T> planes(T *const p[3]) {
  return {{p[0], p[1], p[2]}};
}

template <typename T>
void horizon(const GridP &g, T *const p[3], cudaStream_t st) {
  const int64_t n = (int64_t)(g.n_f + 1 + G_) * g.NY * 3;
  k_horizon<T><<<blocks_for(n), TPB, 0, st>>>(g, p[0], p[1], p[2]);
  COUNT_LAUNCH(1);
}
template <typename T>
void axis(const GridP &g, T *const p[3], int isB, cudaStream_t st) {
  const int64_t n = (int64_t)g.NX * (2 * G_ + 1) * 3;
  k_axis<T><<<blocks_for(n), TPB, 0, st>>>(g, p[0], p[1], p[2], isB);
  COUNT_LAUNCH(1);
}

// Blocks covering ni x nj points: TPBX x TPBY, or 32 x 2 on grids that would not give every SM
// two of those (64^2 cells were 34 or 36 blocks, 8 warps of FP64 work on each of as many SMs);
// rows beyond the grid's limit in y are taken by the kernels' row loop
struct Tiles {
  dim3 grid, block;
};
Tiles tiles_for(int ni, int nj) {
  const bool few = (int64_t)ni * nj < 2 * N_SM * TPBX * TPBY;
  const int bx = few ? 32 : TPBX, by = few ? 2 : TPBY, ny = (nj + by - 1) / by;
  return {dim3((ni + bx - 1) / bx, ny > 65535 ? 65535 : ny), dim3(bx, by)};
}

template <bool DOE, bool DOH, bool DMEAN, typename T>
void aux(const GridP &g, const Pair3<T> &B, const Pair3<T> &D, const FieldPtrsT<T> &F,
         cudaStream_t st) {
  const Tiles t = tiles_for(g.n_r + 3, g.n_th + 1);
  k_aux<T, DOE, DOH, DMEAN><<<t.grid, t.block, 0, st>>>(
      g, B, D, F.tab, F.E[0], F.E[1], F.E[2], F.H[0], F.H[1], F.H[2]);
  COUNT_LAUNCH(1);
}

}  // namespace

template <typename T>
cudaError_t launch_metric_tables(const GridP &g, T *tab, T *polar, cudaStream_t st) {
  k_metric_tables<<<blocks_for(plane_size(g)), TPB, 0, st>>>(g, tab, polar);
  COUNT_LAUNCH(1);
  return cudaGetLastError();
}

cudaError_t launch_dt_min(const GridP &g, double *scratch, int, double *out, cudaStream_t st) {
  unsigned long long *u = reinterpret_cast<unsigned long long *>(scratch);
  const unsigned long long inf = 0x7FF0000000000000ull;
  cudaMemcpyAsync(u, &inf, sizeof(inf), cudaMemcpyHostToDevice, st);
  k_dt_min<<<blocks_for((int64_t)g.n_r * g.n_th), TPB, 0, st>>>(g, u);
  COUNT_LAUNCH(1);
  cudaMemcpyAsync(out, u, sizeof(double), cudaMemcpyDeviceToHost, st);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_zero(T *p, int64_t n, cudaStream_t st) {
  k_zero<T><<<blocks_for(n), TPB, 0, st>>>(p, n);
  COUNT_LAUNCH(1);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init_fields(const GridP &g, const FieldPtrsT<T> &F, int kind, double B0,
                               cudaStream_t st) {
  const int64_t ps = plane_size(g);
  for (int c = 0; c < 3; ++c) {
    launch_zero(F.B[c], ps, st);
    launch_zero(F.D[c], ps, st);
  }
  if (kind == GRPIC_FIELD_WALD || kind == GRPIC_FIELD_VERTICAL || kind == GRPIC_FIELD_MONOPOLE) {
    const int64_t n = (int64_t)(g.n_r + 2 * G_ + 1) * (g.n_th + 1);
    k_init_fields<T><<<blocks_for(n), TPB, 0, st>>>(g, F, kind, B0);
    COUNT_LAUNCH(1);
  }
  return cudaGetLastError();
}

// After em holds the initial B, D: boundary fills, em0 = em, initial-field copy,
// cur0 = cur = 0, B^n = B.
template <typename T>
cudaError_t launch_field_finish_init(const GridP &g, const FieldPtrsT<T> &F, int, cudaStream_t st) {
  const int64_t ps = plane_size(g);
  horizon(g, F.B, st);
  horizon(g, F.D, st);
  axis(g, F.B, 1, st);
  axis(g, F.D, 0, st);
  k_copy3<T><<<blocks_for(ps), TPB, 0, st>>>(ps, F.B[0], F.B[1], F.B[2], F.B0[0], F.B0[1], F.B0[2]);
  k_copy3<T><<<blocks_for(ps), TPB, 0, st>>>(ps, F.D[0], F.D[1], F.D[2], F.D0[0], F.D0[1], F.D0[2]);
  k_copy3<T><<<blocks_for(ps), TPB, 0, st>>>(ps, F.B[0], F.B[1], F.B[2], F.Bi[0], F.Bi[1], F.Bi[2]);
  k_copy3<T><<<blocks_for(ps), TPB, 0, st>>>(ps, F.D[0], F.D[1], F.D[2], F.Di[0], F.Di[1], F.Di[2]);
  k_copy3<T><<<blocks_for(ps), TPB, 0, st>>>(ps, F.B[0], F.B[1], F.B[2], F.Bn[0], F.Bn[1], F.Bn[2]);
  COUNT_LAUNCH(5);
  for (int c = 0; c < 3; ++c) {
    launch_zero(F.J[c], ps, st);
    launch_zero(F.J0[c], ps, st);
    launch_zero(F.E[c], ps, st);
    launch_zero(F.H[c], ps, st);
    launch_zero(F.Dh[c], ps, st);
  }
  return cudaGetLastError();
}

// Loop step 2 of Sec. 3.4: B^{n-1} = (B^{n-3/2} + B^{n-1/2})/2, D^{n-1/2} = (D^{n-1} + D^n)/2,
// E^{n-1/2} from {B^{n-1/2}, D^{n-1/2}}, auxiliary Faraday B^{n-1} -> B^n (BN planes).
template <typename T>
cudaError_t launch_predict(const GridP &g, const FieldPtrsT<T> &F, cudaStream_t st) {
  aux<true, false, true>(g, one(F.B), pair(F.D0, F.D), F, st);
  const Tiles all = tiles_for(g.NX, g.NY);
  k_faraday<T><<<all.grid, all.block, 0, st>>>(g, pair(F.B0, F.B), planes(F.E), F.tab, planes(F.Bn));
  COUNT_LAUNCH(1);
  return cudaGetLastError();
}

// Loop steps 5-7 of Sec. 3.4 (J holds J^{n+1/2}). Writes B^{n+1/2} into the B0 planes and
// D^{n+1} into the D0 planes; the caller then swaps em/em0 and cur/cur0.
template <typename T>
cudaError_t launch_advance(const GridP &g, const FieldPtrsT<T> &F, cudaStream_t st) {
  const Tiles all = tiles_for(g.NX, g.NY);
  // step 6: E^n, H^n from {B^n, D^n}; Faraday B^{n-1/2} -> B^{n+1/2}; step 7: auxiliary Ampere
  // D^{n-1/2} -> D^{n+1/2} with H^n and J^n = (J^{n-1/2} + J^{n+1/2})/2
  aux<true, true, false>(g, one(F.Bn), one(F.D), F, st);
  k_faraday_ampere<T><<<all.grid, all.block, 0, st>>>(g, one(F.B), planes(F.E), planes(F.B0), planes(F.Bi),
                                            pair(F.D0, F.D), planes(F.H), pair(F.J0, F.J),
                                            planes(F.Dh), F.tab, F.polar);
  COUNT_LAUNCH(1);
  // H^{n+1/2} from {B^{n+1/2}, D^{n+1/2}}; final Ampere D^n -> D^{n+1} with J^{n+1/2}
  aux<false, true, false>(g, one(F.B0), one(F.Dh), F, st);
  k_ampere<T><<<all.grid, all.block, 0, st>>>(g, one(F.D), planes(F.H), one(F.J), F.tab, F.polar,
                                    planes(F.D0), planes(F.Di));
  COUNT_LAUNCH(1);
  return cudaGetLastError();
}

// The auxiliary fields E and H (Eqs. discretized-auxE, discretized-auxH) of the em planes as
// they stand (B^{n+1/2} and D^{n+1} after a step), into the E and H scratch planes.
template <typename T>
cudaError_t launch_aux_fields(const GridP &g, const FieldPtrsT<T> &F, cudaStream_t st) {
  aux<true, true, false>(g, one(F.B), one(F.D), F, st);
  return cudaGetLastError();
}

#define INSTANTIATE_FIELDS(T)                                                                    \
  template cudaError_t launch_metric_tables<T>(const GridP &, T *, T *, cudaStream_t);         \
  template cudaError_t launch_zero<T>(T *, int64_t, cudaStream_t);                              \
  template cudaError_t launch_init_fields<T>(const GridP &, const FieldPtrsT<T> &, int, double, \
                                             cudaStream_t);                                     \
  template cudaError_t launch_field_finish_init<T>(const GridP &, const FieldPtrsT<T> &, int,   \
                                                   cudaStream_t);                               \
  template cudaError_t launch_predict<T>(const GridP &, const FieldPtrsT<T> &, cudaStream_t);   \
  template cudaError_t launch_advance<T>(const GridP &, const FieldPtrsT<T> &, cudaStream_t);   \
  template cudaError_t launch_aux_fields<T>(const GridP &, const FieldPtrsT<T> &, cudaStream_t);
INSTANTIATE_FIELDS(double)
INSTANTIATE_FIELDS(float)
