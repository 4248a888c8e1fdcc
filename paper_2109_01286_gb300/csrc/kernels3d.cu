// CUDA kernels (sm_103a) of the three-dimensional extension of the Hermite FD residual and
// SSP-RK3 step; FP64 state, fluxes and sums.  Per Runge-Kutta stage:
//   k3_vertex  one thread per vertex: the vertex-major copy of the 20 unknowns and the analytic
//              flux vectors F, G, K (Sec. 2.3, vertex fluxes, in 3D);
//   k3_edge    one thread per edge: Alg. 1 in 3D (Roe average of the edge ends, five-wave
//              characteristic projection along the edge, uniform WENO5 weights as the sensor --
//              taken in FP32 and again in FP64 inside a band around each threshold -- 5-node
//              Hermite value or weighted 3-node value per component and side,
//              back-projection, positivity fallback) and Roe's flux with Harten's fix;
//   k3_div_fx  8 lanes per vertex: the CSR gather of the least-squares divergence rows
//              d_0, d_x, d_y, d_z over the vertex fluxes and edge fluxes (Eq.
//              (flux_polynomials) in 3D) in fixed point, fused with the SSP-RK3 stage update;
//   k3_div     the same gather in FP64, 1, 2 or 4 lanes per vertex (chosen lanes, long rows).
// The characteristic projection uses the closed forms of the left and right eigenvectors of
// the flux Jacobian along n with the frame (n, t1, t2): waves q_n - c, entropy, shear along
// t1, shear along t2, q_n + c.
#include <cuda_runtime.h>

#include "fixed_point.cuh"
#include "fp_convert.cuh"
#include "kernels3d.hpp"
#include "mbar.cuh"

namespace hfd {
namespace {

constexpr unsigned kErrNonfinite = 1u, kErrPositivity = 2u, kErrIndex = 4u;

__device__ __forceinline__ bool finite3(double x) { return isfinite(x); }

// The eigen-structure of one Roe state along the frame (n, t1, t2), and the two states'
// reciprocal densities and pressures (shared with the normal fluxes).
struct Eig {
  double u[3], H, c, qn, q1, q2, K, b1, b2, ic;
  double n[3], t1[3], t2[3];
  double irl, irr, pl, pr;
};

// One reciprocal square root per state gives sqrt(rho) and 1/rho, one more gives c and 1/c
// (the CUDA math library's rsqrt); one division forms the Roe weights.
__device__ __forceinline__ void roe_state(const double* wl, const double* wr, double g1, Eig& s) {
  const double sl = rsqrt(wl[0]), sr = rsqrt(wr[0]);
  s.irl = sl * sl;
  s.irr = sr * sr;
  s.pl = g1 * (wl[4] - 0.5 * (wl[1] * wl[1] + wl[2] * wl[2] + wl[3] * wl[3]) * s.irl);
  s.pr = g1 * (wr[4] - 0.5 * (wr[1] * wr[1] + wr[2] * wr[2] + wr[3] * wr[3]) * s.irr);
  const double is = 1.0 / (wl[0] * sl + wr[0] * sr);
#pragma unroll
  for (int k = 0; k < 3; ++k) s.u[k] = (wl[k + 1] * sl + wr[k + 1] * sr) * is;
  s.H = ((wl[4] + s.pl) * sl + (wr[4] + s.pr) * sr) * is;
  s.K = s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2];
  const double c2 = g1 * (s.H - 0.5 * s.K);
  s.ic = rsqrt(c2);
  s.c = c2 * s.ic;
  s.qn = s.u[0] * s.n[0] + s.u[1] * s.n[1] + s.u[2] * s.n[2];
  s.q1 = s.u[0] * s.t1[0] + s.u[1] * s.t1[1] + s.u[2] * s.t1[2];
  s.q2 = s.u[0] * s.t2[0] + s.u[1] * s.t2[1] + s.u[2] * s.t2[2];
  s.b1 = g1 * s.ic * s.ic;
  s.b2 = 0.5 * s.b1 * s.K;
}

// c = L a for the five conserved components a.
__device__ __forceinline__ void to_char(const Eig& s, const double* a, double* c) {
  const double um = s.u[0] * a[1] + s.u[1] * a[2] + s.u[2] * a[3];
  const double nm = (s.n[0] * a[1] + s.n[1] * a[2] + s.n[2] * a[3]) * s.ic;
  const double t1m = s.t1[0] * a[1] + s.t1[1] * a[2] + s.t1[2] * a[3];
  const double t2m = s.t2[0] * a[1] + s.t2[1] * a[2] + s.t2[2] * a[3];
  const double qc = s.qn * s.ic;
  c[0] = 0.5 * ((s.b2 + qc) * a[0] - s.b1 * um - nm + s.b1 * a[4]);
  c[1] = (1.0 - s.b2) * a[0] + s.b1 * um - s.b1 * a[4];
  c[2] = t1m - s.q1 * a[0];
  c[3] = t2m - s.q2 * a[0];
  c[4] = 0.5 * ((s.b2 - qc) * a[0] - s.b1 * um + nm + s.b1 * a[4]);
}

// w = R c.
__device__ __forceinline__ void from_char(const Eig& s, const double* c, double* w) {
  w[0] = c[0] + c[1] + c[4];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    w[k + 1] = (c[0] + c[1] + c[4]) * s.u[k] + (c[4] - c[0]) * s.c * s.n[k] + c[2] * s.t1[k] +
               c[3] * s.t2[k];
  w[4] = (c[0] + c[4]) * s.H + (c[4] - c[0]) * s.c * s.qn + c[1] * (0.5 * s.K) + c[2] * s.q1 +
         c[3] * s.q2;
}

// The FP32 copy of an eigen-structure for the sensor, rounded by integer operations.
struct EigF {
  float u[3], n[3], t1[3], t2[3], ic, qn, q1, q2, b1, b2;
};

__device__ __forceinline__ void to_f32(const Eig& s, EigF& f) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    f.u[k] = d2f_rn(s.u[k]);
    f.n[k] = d2f_rn(s.n[k]);
    f.t1[k] = d2f_rn(s.t1[k]);
    f.t2[k] = d2f_rn(s.t2[k]);
  }
  f.ic = d2f_rn(s.ic);
  f.qn = d2f_rn(s.qn);
  f.q1 = d2f_rn(s.q1);
  f.q2 = d2f_rn(s.q2);
  f.b1 = d2f_rn(s.b1);
  f.b2 = d2f_rn(s.b2);
}

// c = L a in FP32 (the formulas of to_char).
__device__ __forceinline__ void to_char_f(const EigF& s, const float* a, float* c) {
  const float um = s.u[0] * a[1] + s.u[1] * a[2] + s.u[2] * a[3];
  const float nm = (s.n[0] * a[1] + s.n[1] * a[2] + s.n[2] * a[3]) * s.ic;
  const float t1m = s.t1[0] * a[1] + s.t1[1] * a[2] + s.t1[2] * a[3];
  const float t2m = s.t2[0] * a[1] + s.t2[1] * a[2] + s.t2[2] * a[3];
  const float qc = s.qn * s.ic;
  c[0] = 0.5f * ((s.b2 + qc) * a[0] - s.b1 * um - nm + s.b1 * a[4]);
  c[1] = (1.0f - s.b2) * a[0] + s.b1 * um - s.b1 * a[4];
  c[2] = t1m - s.q1 * a[0];
  c[3] = t2m - s.q2 * a[0];
  c[4] = 0.5f * ((s.b2 - qc) * a[0] - s.b1 * um + nm + s.b1 * a[4]);
}

// rho > 0 and p > 0 (R16): p has the sign of E rho - |m|^2 / 2 when rho > 0.
__device__ __forceinline__ bool admissible3(const double* w) {
  return w[0] > 0.0 && w[4] * w[0] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]) > 0.0;
}

// Uniform WENO5 on the five values u0..u4 (Jiang-Shu indicators, linear weights 1/16, 10/16,
// 5/16) with every weight multiplied by (eps+b1)^2 (eps+b2)^2 (eps+b3)^2, so that the sensor
// needs no division: t[i] is weight i times that product and S their sum; omega_i = t[i] / S.
__device__ __forceinline__ void weno3(double u0, double u1, double u2, double u3, double u4,
                                      double eps, double* t, double& S) {
  const double e1 = u0 - 2.0 * u1 + u2, f1 = u0 - 4.0 * u1 + 3.0 * u2;
  const double e2 = u1 - 2.0 * u2 + u3, f2 = u1 - u3;
  const double e3 = u2 - 2.0 * u3 + u4, f3 = 3.0 * u2 - 4.0 * u3 + u4;
  const double b1 = 13.0 / 12.0 * (e1 * e1) + 0.25 * (f1 * f1);
  const double b2 = 13.0 / 12.0 * (e2 * e2) + 0.25 * (f2 * f2);
  const double b3 = 13.0 / 12.0 * (e3 * e3) + 0.25 * (f3 * f3);
  double s1 = eps + b1, s2 = eps + b2, s3 = eps + b3;
  s1 *= s1;
  s2 *= s2;
  s3 *= s3;
  t[0] = (1.0 / 16.0) * (s2 * s3);
  t[1] = (10.0 / 16.0) * (s1 * s3);
  t[2] = (5.0 / 16.0) * (s1 * s2);
  S = t[0] + t[1] + t[2];
}

// weno3 in FP32, for the sensor's first pass.
__device__ __forceinline__ void weno3f(float u0, float u1, float u2, float u3, float u4, float eps,
                                       float& t0, float& S) {
  const float e1 = u0 - 2.0f * u1 + u2, f1 = u0 - 4.0f * u1 + 3.0f * u2;
  const float e2 = u1 - 2.0f * u2 + u3, f2 = u1 - u3;
  const float e3 = u2 - 2.0f * u3 + u4, f3 = 3.0f * u2 - 4.0f * u3 + u4;
  float s1 = eps + (13.0f / 12.0f * (e1 * e1) + 0.25f * (f1 * f1));
  float s2 = eps + (13.0f / 12.0f * (e2 * e2) + 0.25f * (f2 * f2));
  float s3 = eps + (13.0f / 12.0f * (e3 * e3) + 0.25f * (f3 * f3));
  s1 *= s1;
  s2 *= s2;
  s3 *= s3;
  t0 = 0.0625f * (s2 * s3);
  S = t0 + 0.625f * (s1 * s3) + 0.3125f * (s1 * s2);
}

// Relative width of the band around each sensor threshold inside which the FP32 decision is
// taken again in FP64.
constexpr float kGuard3 = 1e-3f;

// F_n(w) from the state, its reciprocal density and its pressure.
__device__ __forceinline__ void normal_flux3(const double* w, double ir, double p, const double* n,
                                             double* f) {
  const double un = (w[1] * n[0] + w[2] * n[1] + w[3] * n[2]) * ir;
  f[0] = w[0] * un;
#pragma unroll
  for (int k = 0; k < 3; ++k) f[k + 1] = w[k + 1] * un + p * n[k];
  f[4] = (w[4] + p) * un;
}

// ------------------------------------------------------------------ k3_vertex
// A 5-vector's record in fixed point: its pairs and the codes of mass, momentum (one for the three: each row
// reads fluxes in all directions, so every momentum sum has pressure-sized terms) and energy.
constexpr int kBits3 = 29;
__device__ __forceinline__ void st_record3(int4* rec, size_t i, const double* f) {
  const int E0 = fx_code(f[0]), E1 = max(fx_code(f[1]), max(fx_code(f[2]), fx_code(f[3]))), E2 = fx_code(f[4]);
  const int2 p0 = fx_encode(f[0], E0, kBits3), p1 = fx_encode(f[1], E1, kBits3), p2 = fx_encode(f[2], E1, kBits3);
  const int2 p3 = fx_encode(f[3], E1, kBits3), p4 = fx_encode(f[4], E2, kBits3);
  int4* o = rec + 3 * i;
  o[0] = make_int4(p0.x, p0.y, p1.x, p1.y);
  o[1] = make_int4(p2.x, p2.y, p3.x, p3.y);
  o[2] = make_int4(p4.x, p4.y, (int)((unsigned)E0 | ((unsigned)E1 << 16)), E2);
}

// Ua: 20 values per vertex (160 B); FGK: F, G, K per vertex at a stride of 16 (128 B); FX: records 3 v,
// 3 v + 1, 3 v + 2 instead.
template <bool FX>
__global__ void __launch_bounds__(256) k3_vertex(int V, const double* __restrict__ U,
                                                 double* __restrict__ Ua, double* __restrict__ FGK,
                                                 int4* __restrict__ rec, double g1) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  double w[20];
#pragma unroll
  for (int r = 0; r < 20; ++r) w[r] = U[(size_t)r * V + v];
  double2* ua = reinterpret_cast<double2*>(Ua + (size_t)20 * v);
#pragma unroll
  for (int i = 0; i < 10; ++i) ua[i] = make_double2(w[2 * i], w[2 * i + 1]);
  const double ir = 1.0 / w[0];
  const double u = w[1] * ir, vv = w[2] * ir, ww = w[3] * ir;
  const double p = g1 * (w[4] - 0.5 * (w[1] * u + w[2] * vv + w[3] * ww));
  const double f[16] = {w[1], w[1] * u + p, w[2] * u, w[3] * u, (w[4] + p) * u,
                        w[2], w[1] * vv, w[2] * vv + p, w[3] * vv, (w[4] + p) * vv,
                        w[3], w[1] * ww, w[2] * ww, w[3] * ww + p, (w[4] + p) * ww, 0.0};
  if (FX) {
#pragma unroll
    for (int p = 0; p < 3; ++p) st_record3(rec, (size_t)3 * v + p, f + 5 * p);
  } else {
    double2* o = reinterpret_cast<double2*>(FGK + (size_t)16 * v);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = make_double2(f[2 * i], f[2 * i + 1]);
  }
}

// ------------------------------------------------------------------ k3_edge
// One thread per edge.  Stencil ids (6 x E), frame (9 x E), w5 (40 x E) and w3 (18 x E) are
// structure-of-arrays streams; node data are gathered from Ua.  h: 8 doubles per edge (5 used); FX:
// record 3 V + e instead.
template <bool FX>
__global__ void __launch_bounds__(128) k3_edge(int E, int V, const int32_t* __restrict__ sten,
                                               const double* __restrict__ frame,
                                               const double* __restrict__ w5,
                                               const double* __restrict__ w3,
                                               const double* __restrict__ Ua,
                                               double* __restrict__ h, int4* __restrict__ rec,
                                               Phys3 ph, unsigned* __restrict__ err) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  int s[6];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    s[k] = __ldg(sten + (size_t)k * E + e);
    bad |= (unsigned)s[k] >= (unsigned)V;
  }
  if (bad) {
    atomicOr(err, kErrIndex);
    return;
  }
  const double g1 = ph.g1;
  Eig st;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    st.n[k] = __ldg(frame + (size_t)k * E + e);
    st.t1[k] = __ldg(frame + (size_t)(3 + k) * E + e);
    st.t2[k] = __ldg(frame + (size_t)(6 + k) * E + e);
  }
  double wi[5], wj[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    wi[q] = __ldg(Ua + (size_t)20 * s[2] + q);
    wj[q] = __ldg(Ua + (size_t)20 * s[3] + q);
  }
  roe_state(wi, wj, g1, st);
  // FP32 sensor: characteristic values of the six nodes' differences from the tail state (the
  // WENO indicators see differences only), each difference formed in FP64 and rounded once;
  // and the 5-node sums of both sides in conservative variables, in FP64
  EigF sf;
  to_f32(st, sf);
  float cf[6][5];
  double W[2][5];
#pragma unroll
  for (int q = 0; q < 5; ++q) W[0][q] = W[1][q] = 0.0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double a[20];
    const double2* src = reinterpret_cast<const double2*>(Ua + (size_t)20 * s[k]);
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      const double2 t = __ldg(src + i);
      a[2 * i] = t.x;
      a[2 * i + 1] = t.y;
    }
    float d[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) d[q] = d2f_rn(a[q] - wi[q]);
    to_char_f(sf, d, cf[k]);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int j = k - side;                 // node index within this side's five
      if (j < 0 || j > 4) continue;
#pragma unroll
      for (int dd = 0; dd < 4; ++dd) {
        const double wt = __ldg(w5 + (size_t)(20 * side + 4 * j + dd) * E + e);
#pragma unroll
        for (int q = 0; q < 5; ++q) W[side][q] = fma(wt, a[5 * dd + q], W[side][q]);
      }
    }
  }
  // per side and characteristic component: FP32 decision, taken again in FP64 (on the node
  // values' characteristic values, as the 3-node candidates need) inside the guard band or on a
  // non-finite FP32 sum; weighted 3-node values where the decision is rough
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    unsigned flag = 0;                        // rough in FP32, or undecided
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (ph.force_branch == 1) break;
      if (ph.force_branch == 2) {
        flag |= 1u << q;
        continue;
      }
      float t0, S;
      if (side == 0) weno3f(cf[0][q], cf[1][q], cf[2][q], cf[3][q], cf[4][q], ph.epsf, t0, S);
      else           weno3f(cf[5][q], cf[4][q], cf[3][q], cf[2][q], cf[1][q], ph.epsf, t0, S);
      const float mlo = t0 - ph.sens_lof * S, mhi = ph.sens_hif * S - t0;
      const bool smooth = mlo > 0.f && mhi > 0.f;
      const bool clear = isfinite(S) && fabsf(mlo) > kGuard3 * S && fabsf(mhi) > kGuard3 * S;
      if (!smooth || !clear) flag |= 1u << q;
    }
    if (!flag) continue;
    double C[5];
    to_char(st, W[side], C);
    bool any = false;
    const double* w = w3 + (size_t)(9 * side) * E + e;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (!((flag >> q) & 1u)) continue;
      double cq[5];
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const int k = side == 0 ? j : 5 - j;
        double a[5], c[5];
#pragma unroll
        for (int r = 0; r < 5; ++r) a[r] = __ldg(Ua + (size_t)20 * s[k] + r);
        to_char(st, a, c);
        cq[j] = c[q];
      }
      double o[3], S;
      weno3(cq[0], cq[1], cq[2], cq[3], cq[4], ph.eps, o, S);
      const bool smooth = o[0] > ph.sens_lo * S && o[0] < ph.sens_hi * S;
      if (ph.force_branch != 2 && smooth) continue;
      const double iS = 1.0 / S;
      double wt[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) wt[i] = __ldg(w + (size_t)i * E);
      const double c1 = wt[0] * cq[0] + wt[1] * cq[1] + wt[2] * cq[2];
      const double c2 = wt[3] * cq[1] + wt[4] * cq[2] + wt[5] * cq[3];
      const double c3 = wt[6] * cq[2] + wt[7] * cq[3] + wt[8] * cq[4];
      C[q] = (o[0] * iS) * c1 + (o[1] * iS) * c2 + (o[2] * iS) * c3;
      any = true;
    }
    if (any) from_char(st, C, W[side]);
  }
  // positivity (R16): fall back to the end state of that side
  if (!admissible3(W[0]))
#pragma unroll
    for (int q = 0; q < 5; ++q) W[0][q] = wi[q];
  if (!admissible3(W[1]))
#pragma unroll
    for (int q = 0; q < 5; ++q) W[1][q] = wj[q];
  // Roe's flux along n with Harten's fix on all five waves
  Eig r;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.n[k] = st.n[k];
    r.t1[k] = st.t1[k];
    r.t2[k] = st.t2[k];
  }
  roe_state(W[0], W[1], g1, r);
  double dw[5], al[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) dw[q] = W[1][q] - W[0][q];
  to_char(r, dw, al);
  const double lam[5] = {r.qn - r.c, r.qn, r.qn, r.qn, r.qn + r.c};
  const double del = ph.harten * r.c, i2del = ph.half_inv_harten * r.ic;
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    double a = fabs(lam[i]);
    if (a < del) a = (lam[i] * lam[i] + del * del) * i2del;
    al[i] *= a;
  }
  double diss[5], fl[5], fr[5];
  from_char(r, al, diss);
  normal_flux3(W[0], r.irl, r.pl, r.n, fl);
  normal_flux3(W[1], r.irr, r.pr, r.n, fr);
  double hq[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) hq[q] = 0.5 * (fl[q] + fr[q]) - 0.5 * diss[q];
  if (FX) {
    st_record3(rec, (size_t)3 * V + e, hq);
    return;
  }
  double* o = h + (size_t)8 * e;
  reinterpret_cast<double2*>(o)[0] = make_double2(hq[0], hq[1]);
  reinterpret_cast<double2*>(o)[1] = make_double2(hq[2], hq[3]);
  o[4] = hq[4];
}

// ------------------------------------------------------------------ k3_div
// G lanes per vertex (G = 1, 2 or 4, consecutive threads): the lanes take the vertex's entries
// in turn (lane l the entries l, l + G, ...; adjacent lanes read adjacent coefficient blocks),
// each accumulates acc[5 r + q] over its entries of the row r (d_0, d_x, d_y, d_z): 12
// coefficients per vertex entry against F, G, K of the entry's vertex and 4 per edge entry
// against h of the entry's edge.  The lanes' sums are combined by a fixed butterfly, so the
// result is deterministic.  R = -acc; mode 0 writes R; mode 1 writes the stage update
// b (Us + dt R) + a Un (a = 0: Un is not read) with explicit roundings; lane l writes the
// rows l, l + G, ...
template <int G>
__global__ void __launch_bounds__(128) k3_div(int V, int E, const int32_t* __restrict__ vptr,
                                              const int32_t* __restrict__ vidx,
                                              const double* __restrict__ cv,
                                              const int32_t* __restrict__ eptr,
                                              const int32_t* __restrict__ eidx,
                                              const double* __restrict__ ce,
                                              const double* __restrict__ FGK,
                                              const double* __restrict__ h, int mode,
                                              const double* __restrict__ Us, const double* Un,
                                              double* out, double a, double b, double dt,
                                              unsigned* __restrict__ err) {
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int v = gt / G, lane = gt % G;
  // whole groups stay in the warp for the shuffles (V * G threads rounded up to the block)
  const bool live = v < V;
  double acc[20];
#pragma unroll
  for (int i = 0; i < 20; ++i) acc[i] = 0.0;
  unsigned bad = 0;
  if (live) {
    const int j0 = __ldg(vptr + v), j1 = __ldg(vptr + v + 1);
    for (int j = j0 + lane; j < j1; j += G) {
      const int u = __ldg(vidx + j);
      if ((unsigned)u >= (unsigned)V) {
        bad |= kErrIndex;
        continue;
      }
      double c[12], f[16];
      const double2* cs = reinterpret_cast<const double2*>(cv + (size_t)12 * j);
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        const double2 t = __ldg(cs + i);
        c[2 * i] = t.x;
        c[2 * i + 1] = t.y;
      }
      const double2* fs = reinterpret_cast<const double2*>(FGK + (size_t)16 * u);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const double2 t = __ldg(fs + i);
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 5; ++q)
          acc[5 * r + q] = fma(c[3 * r], f[q], fma(c[3 * r + 1], f[5 + q], fma(c[3 * r + 2], f[10 + q], acc[5 * r + q])));
    }
    const int k0 = __ldg(eptr + v), k1 = __ldg(eptr + v + 1);
    for (int j = k0 + lane; j < k1; j += G) {
      const int ed = __ldg(eidx + j);
      if ((unsigned)ed >= (unsigned)E) {
        bad |= kErrIndex;
        continue;
      }
      const double2 c01 = __ldg(reinterpret_cast<const double2*>(ce + (size_t)4 * j));
      const double2 c23 = __ldg(reinterpret_cast<const double2*>(ce + (size_t)4 * j) + 1);
      const double* hp = h + (size_t)8 * ed;
      const double2 h01 = __ldg(reinterpret_cast<const double2*>(hp));
      const double2 h23 = __ldg(reinterpret_cast<const double2*>(hp) + 1);
      const double hq[5] = {h01.x, h01.y, h23.x, h23.y, __ldg(hp + 4)};
      const double cr[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int q = 0; q < 5; ++q) acc[5 * r + q] = fma(cr[r], hq[q], acc[5 * r + q]);
    }
  }
  // butterfly over the group: every lane ends with the group's sums, in the same order
#pragma unroll
  for (int off = 1; off < G; off <<= 1)
#pragma unroll
    for (int i = 0; i < 20; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off, G);
  if (!live) return;
#pragma unroll
  for (int i = 0; i < 20; ++i) {
    if (i % G != lane) continue;
    const double R = -acc[i];
    const size_t idx = (size_t)i * V + v;
    double o;
    if (mode == 0) {
      o = R;
    } else {
      o = __dmul_rn(b, __fma_rn(dt, R, Us[idx]));
      if (a != 0.0) o = __fma_rn(a, Un[idx], o);
    }
    out[idx] = o;
    if (!finite3(o)) bad |= kErrNonfinite;
    if (mode == 1 && i == 0 && !(o > 0.0)) bad |= kErrPositivity;
  }
  if (bad) atomicOr(err, bad);
}

// ------------------------------------------------------------------ k3_div_fx
// The same gather with the sums on the integer pipe (fixed_point.cuh, L = 29).  A row of 65 vertices
// and 304 edges is 9980 products: in FP64 the pipe (2 lanes per clock and SM) takes 5000 clocks of an
// SM for them, while its 18 KB of coefficients and indices need about 1000 of the SM's share of the HBM.
// 24^3 (13,824 rows): 102 us, the FP64 kernel 294 us.
//
// F, G and K of a vertex are records like the edges' fluxes, so a row is one list of products of a
// record with a coefficient of each d_k.  8 lanes share a row: lane l takes stream l / 2 of the
// list and d_0, d_x (l even) or d_y, d_z (l odd), so that its sums take 40 registers and not 80; the 8
// lanes read 128 contiguous bytes of coefficients each time.  A chunk's records and coefficients are
// copied to shared memory one chunk ahead, its record ids are read two ahead (each warp its own
// rows: no block barrier).  What is left is the gathers: an L1 hit rate of one half, 43% of the issue
// slots used.  Measured slower: records loaded to registers four at a time (145 us; 190 us with
// vertex entries of 128 bytes and two edges at a time), records past L1 (149 us), ids read with their
// records (126 us), coefficients prefetched into L2 a row at a time (121 us: they evict one another)
// or 3 to 12 chunks ahead (110 us), 20 warps an SM (138 us).  Blocks of 1, 2, 4 warps: no difference.
// Bounds: k3_pack scales each d_k so that its coefficients add up to 127 times the scale at most, which keeps
// the high sums below 2^63; the cross sums are carried over every 40 products (42 fit).
constexpr int kWarps3 = 4;                      // warps of a block, 4 rows each
struct Ring3 {                                  // one chunk of each row of a block
  int4 rec[kWarps3][4][3][16];                      // [warp][product][piece][row of the warp, stream]
  int4 c[kWarps3][4][32];                           // [warp][product][lane]
};
struct Fx3Args {
  Div3Fx fx;
  const int32_t *vptr, *vidx, *eptr, *eidx;       // the FP64 rows, for fallback3
  const double *cv, *ce;
};

__device__ __forceinline__ uint2 max3(uint2 a, int x, int y) {
  return make_uint2(__vmaxu2(a.x, (unsigned)x), max(a.y, (unsigned)y));
}

// One sum (row d_k, component q) of a row some of whose fluxes are not finite, as k3_div takes it.
__device__ __noinline__ double fallback3(const Fx3Args& m, int V, int v, int k, int q) {
  auto value = [&](size_t i) {
    const int2* p = reinterpret_cast<const int2*>(m.fx.rec + 3 * i);
    const int c = q == 0 ? p[5].x & 0xffff : q < 4 ? (int)((unsigned)p[5].x >> 16) : p[5].y;
    return fx_decode(p[q], c, kBits3);
  };
  double s = 0.0;
  for (int j = m.vptr[v]; j < m.vptr[v + 1]; ++j)
#pragma unroll 1
    for (int d = 2; d >= 0; --d)
      s = fma(m.cv[(size_t)12 * j + 3 * k + d], value((size_t)3 * m.vidx[j] + d), s);
  for (int j = m.eptr[v]; j < m.eptr[v + 1]; ++j)
    s = fma(m.ce[(size_t)4 * j + k], value((size_t)3 * V + m.eidx[j]), s);
  return s;
}

// 16 bytes global -> shared, asynchronously, with and without a copy left in L1.
__device__ __forceinline__ void copy16_l1(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copies_wait_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

__global__ void __launch_bounds__(32 * kWarps3, 16 / kWarps3) k3_div_fx(int V, Fx3Args m, int mode, const double* __restrict__ Us,
                                                    const double* Un, double* out, double a, double b,
                                                    double dt, unsigned* __restrict__ err) {
  constexpr int L = kBits3;
  const int gt = blockIdx.x * blockDim.x + threadIdx.x;
  const int v = gt >> 3, lane = gt & 7;
  const bool live = v < V;                     // whole groups stay in the warp for the shuffles
  const int tid = threadIdx.x, wp = tid >> 5, slot = (tid & 31) >> 1;
  const unsigned group = 0xffu << (tid & 24);
  __shared__ Ring3 ring[2];
  int c0 = 0, c1 = 0;
  int2 ke = make_int2(0, 0);
  if (live) {
    c0 = __ldg(m.fx.ptr + v);
    c1 = __ldg(m.fx.ptr + v + 1);
    ke = __ldg(m.fx.cexp + v);
  }
  // the row's scale: the largest code of its records
  uint2 E = make_uint2(0x00010001u, 1u);
  const int2* ids = reinterpret_cast<const int2*>(m.fx.id) + lane;   // two of the stream's four records
#pragma unroll 8
  for (int c = c0; c < c1; ++c) {
    const int2 i = __ldg(ids + (size_t)8 * c);
    const int2 w0 = __ldg(reinterpret_cast<const int2*>(m.fx.rec + (size_t)3 * i.x + 2) + 1);
    const int2 w1 = __ldg(reinterpret_cast<const int2*>(m.fx.rec + (size_t)3 * i.y + 2) + 1);
    E = max3(max3(E, w0.x, w0.y), w1.x, w1.y);
  }
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const unsigned x = __shfl_xor_sync(0xffffffffu, E.x, o), y = __shfl_xor_sync(0xffffffffu, E.y, o);
    E = max3(E, (int)x, (int)y);
  }
  const bool odd = (E.x & 0xffffu) == kFxRaw || (E.x >> 16) == kFxRaw || E.y == kFxRaw;
  // one chunk: a lane copies half of its stream's records and its own coefficients
  auto fetch = [&](int c, int b, int2 i) {
    const int n = 2 * (lane & 1);
    const int4 *r0 = m.fx.rec + (size_t)3 * i.x, *r1 = m.fx.rec + (size_t)3 * i.y;
    const int4* k = m.fx.c + (size_t)32 * c + lane;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      copy16_l1(&ring[b].rec[wp][n][t][slot], r0 + t);
      copy16_l1(&ring[b].rec[wp][n + 1][t][slot], r1 + t);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) copy16(&ring[b].c[wp][t][tid & 31], k + 8 * t);
  };
  long long hh[10], x[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) hh[i] = x[i] = 0;
  if (!odd && c1 > c0) {
    int2 next = __ldg(ids + (size_t)8 * c0);     // ids are read two chunks ahead, records one
    fetch(c0, 0, next);
    copies_commit();
    next = __ldg(ids + (size_t)8 * min(c0 + 1, c1 - 1));
    int left = 10;                             // chunks until the cross sums are carried over
#pragma unroll 1
    for (int c = c0; c < c1; ++c) {
      const int b = (c - c0) & 1;
      if (c + 1 < c1) {
        fetch(c + 1, b ^ 1, next);
        next = __ldg(ids + (size_t)8 * min(c + 2, c1 - 1));
      }
      copies_commit();
      copies_wait_but_one();
      __syncwarp(group);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int4 k = ring[b].c[wp][i][tid & 31];
        const int4 r0 = ring[b].rec[wp][i][0][slot], r1 = ring[b].rec[wp][i][1][slot], r2 = ring[b].rec[wp][i][2][slot];
        int2 p[5] = {make_int2(r0.x, r0.y), make_int2(r0.z, r0.w), make_int2(r1.x, r1.y), make_int2(r1.z, r1.w),
                     make_int2(r2.x, r2.y)};
        const unsigned t = E.x - (unsigned)r2.z;
        int d[3] = {(int)(t & 0xffffu), (int)(t >> 16), (int)(E.y - (unsigned)r2.w)};
        if (((t & 0xffe0ffe0u) | ((unsigned)d[2] & ~31u)) != 0u) {      // a shift of 32 or more
          int s[3] = {d[1], d[1], d[1]};
          fx_far(p[0].x, p[0].y, d[0]);
#pragma unroll
          for (int q = 0; q < 3; ++q) fx_far(p[1 + q].x, p[1 + q].y, s[q]);
          fx_far(p[4].x, p[4].y, d[2]);
          d[1] = s[0];
        }
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          fx_limbs(p[q].x, p[q].y, d[q == 0 ? 0 : q < 4 ? 1 : 2], L);
          fx_fma(hh[q], x[q], k.x, k.y, p[q].x, p[q].y);
          fx_fma(hh[5 + q], x[5 + q], k.z, k.w, p[q].x, p[q].y);
        }
      }
      __syncwarp(group);
      if (--left == 0) {
        left = 10;
#pragma unroll
        for (int i = 0; i < 10; ++i) x[i] = fx_carry(hh[i], x[i], L);
      }
    }
  }
  // the four streams' sums, exactly: lanes with bit 2 clear keep the first of their two rows, the
  // others the second; bit 1 then shares the row's components
  unsigned lo[10];
#pragma unroll
  for (int i = 0; i < 10; ++i) lo[i] = fx_carry(hh[i], x[i], L);
  const bool second = (lane & 4) != 0;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const long long sh = second ? hh[q] : hh[5 + q];
    const unsigned sl = second ? lo[q] : lo[5 + q];
    hh[q] = (second ? hh[5 + q] : hh[q]) + __shfl_xor_sync(0xffffffffu, sh, 4);
    lo[q] = (second ? lo[5 + q] : lo[q]) + __shfl_xor_sync(0xffffffffu, sl, 4);
    hh[q] += __shfl_xor_sync(0xffffffffu, hh[q], 2);
    lo[q] += __shfl_xor_sync(0xffffffffu, lo[q], 2);
  }
  if (!live) return;
  const int row = 2 * (lane & 1) + (second ? 1 : 0);
  const int kr = (lane & 1) ? ke.y : ke.x;
  const int unit = (second ? kr >> 16 : (kr << 16) >> 16) + L - 1022 - 2 * (2 * L - 1);
  unsigned bad = 0;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    if ((q >= 3) != ((lane & 2) != 0)) continue;
    const int code = q == 0 ? (int)(E.x & 0xffffu) : q < 4 ? (int)(E.x >> 16) : (int)E.y;
    const double s = odd ? fallback3(m, V, v, row, q) : fx_to_double(hh[q], lo[q], code + unit, L);
    const double R = -s;
    const size_t idx = (size_t)(5 * row + q) * V + v;
    double o;
    if (mode == 0) {
      o = R;
    } else {
      o = __dmul_rn(b, __fma_rn(dt, R, Us[idx]));
      if (a != 0.0) o = __fma_rn(a, Un[idx], o);
    }
    out[idx] = o;
    if (!finite3(o)) bad |= kErrNonfinite;
    if (mode == 1 && row == 0 && q == 0 && !(o > 0.0)) bad |= kErrPositivity;
  }
  if (bad) atomicOr(err, bad);
}

// One warp per row: the list of products, the coefficients as limbs at the scale of their d_k.
__global__ void k3_pack(int V, const int32_t* __restrict__ vptr, const int32_t* __restrict__ vidx,
                        const int32_t* __restrict__ eptr, const int32_t* __restrict__ eidx,
                        const double* __restrict__ cv, const double* __restrict__ ce, Div3Fx fx, int* flag) {
  const int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (v >= V) return;
  const int j0 = vptr[v], K1 = 3 * (vptr[v + 1] - j0), k0 = eptr[v], K = K1 + eptr[v + 1] - k0;
  auto coef = [&](int i, int k) {                // product i of the row: vertices' F, G, K, then edges
    return i < K1 ? cv[(size_t)12 * (j0 + i / 3) + 3 * k + i % 3] : ce[(size_t)4 * (k0 + i - K1) + k];
  };
  int e[4];
  bool bad = false;
  for (int k = 0; k < 4; ++k) {
    int t = -10000;
    double sum = 0.0;
    for (int i = lane; i < K; i += 32) {
      const double c = coef(i, k);
      bad |= !isfinite(c);
      t = max(t, exp_above(c));
      sum += fabs(c);
    }
    for (int o = 16; o > 0; o >>= 1) {
      t = max(t, __shfl_xor_sync(0xffffffffu, t, o));
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
    }
    e[k] = t == -10000 ? 0 : t;
    bad |= !(sum < 1e150) || abs(e[k]) > 400;
    if (!bad)
      while (sum > scalbn(127.0, e[k])) ++e[k];
  }
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) *flag = 1;
    return;
  }
  if (lane == 0)
    fx.cexp[v] = make_int2((e[0] & 0xffff) | (int)((unsigned)e[1] << 16), (e[2] & 0xffff) | (int)((unsigned)e[3] << 16));
  const int c0 = fx.ptr[v], nc = fx.ptr[v + 1] - c0;
  int32_t* id = reinterpret_cast<int32_t*>(fx.id);
  for (int j = lane; j < 16 * nc; j += 32) {
    const bool pad = j >= K;                     // padding stays within the row's scale
    const int i = pad ? 0 : j, n = (j >> 2) & 3, s = j & 3;
    const size_t ch = (size_t)c0 + (j >> 4);
    id[16 * ch + 4 * s + n] = i < K1 ? 3 * vidx[j0 + i / 3] + i % 3 : 3 * V + eidx[k0 + i - K1];
    for (int hf = 0; hf < 2; ++hf) {
      const int2 p = pad ? make_int2(0, 0) : coef_limbs(coef(i, 2 * hf), e[2 * hf], kBits3);
      const int2 q = pad ? make_int2(0, 0) : coef_limbs(coef(i, 2 * hf + 1), e[2 * hf + 1], kBits3);
      fx.c[32 * ch + 8 * n + 2 * s + hf] = make_int4(p.x, p.y, q.x, q.y);
    }
  }
}

}  // namespace

cudaError_t launch3_pack(const DevMesh3& m, int* flag, cudaStream_t s) {
  k3_pack<<<(m.V + 3) / 4, 128, 0, s>>>(m.V, m.vptr, m.vidx, m.eptr, m.eidx, m.cv, m.ce, m.fx, flag);
  return cudaGetLastError();
}

cudaError_t launch3_vertex(const DevMesh3& m, const double* U, const Phys3& ph, cudaStream_t s) {
  if (m.V == 0) return cudaSuccess;
  const unsigned nb = (unsigned)((m.V + 255) / 256);
  if (div3_lanes(m) == 0) k3_vertex<true><<<nb, 256, 0, s>>>(m.V, U, m.Ua, m.FGK, m.fx.rec, ph.g1);
  else                    k3_vertex<false><<<nb, 256, 0, s>>>(m.V, U, m.Ua, m.FGK, m.fx.rec, ph.g1);
  return cudaGetLastError();
}

cudaError_t launch3_edge(const DevMesh3& m, const Phys3& ph, cudaStream_t s) {
  if (m.E == 0) return cudaSuccess;
  const unsigned nb = (unsigned)((m.E + 127) / 128);
  if (div3_lanes(m) == 0)
    k3_edge<true><<<nb, 128, 0, s>>>(m.E, m.V, m.sten, m.frame, m.w5, m.w3, m.Ua, m.h, m.fx.rec, ph,
                                     m.err);
  else
    k3_edge<false><<<nb, 128, 0, s>>>(m.E, m.V, m.sten, m.frame, m.w5, m.w3, m.Ua, m.h, m.fx.rec, ph,
                                     m.err);
  return cudaGetLastError();
}

cudaError_t launch3_div(const DevMesh3& m, const double* Us, const double* Un, double* out,
                        int mode, double a, double b, double dt, cudaStream_t s) {
  if (m.V == 0) return cudaSuccess;
  const int lanes = div3_lanes(m);
  const int64_t threads = (int64_t)m.V * (lanes ? lanes : 8);
  const unsigned blocks = (unsigned)((threads + 127) / 128);
  if (lanes == 0) {
    constexpr int nt = 32 * kWarps3;
    const Fx3Args f = {m.fx, m.vptr, m.vidx, m.eptr, m.eidx, m.cv, m.ce};
    k3_div_fx<<<(unsigned)((threads + nt - 1) / nt), nt, 0, s>>>(m.V, f, mode, Us, Un, out, a, b, dt, m.err);
  } else if (lanes == 4)
    k3_div<4><<<blocks, 128, 0, s>>>(m.V, m.E, m.vptr, m.vidx, m.cv, m.eptr, m.eidx, m.ce, m.FGK,
                                     m.h, mode, Us, Un, out, a, b, dt, m.err);
  else if (lanes == 2)
    k3_div<2><<<blocks, 128, 0, s>>>(m.V, m.E, m.vptr, m.vidx, m.cv, m.eptr, m.eidx, m.ce, m.FGK,
                                     m.h, mode, Us, Un, out, a, b, dt, m.err);
  else
    k3_div<1><<<blocks, 128, 0, s>>>(m.V, m.E, m.vptr, m.vidx, m.cv, m.eptr, m.eidx, m.ce, m.FGK,
                                     m.h, mode, Us, Un, out, a, b, dt, m.err);
  return cudaGetLastError();
}

}  // namespace hfd
