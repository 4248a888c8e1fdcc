// The edge fluxes of the three-dimensional extension: Alg. 1 in 3D (Roe average of the edge ends, five-wave
// characteristic projection along the edge, uniform WENO5 weights as the sensor, 5-node Hermite value or
// weighted 3-node value per component and side, back-projection, positivity fallback) and Roe's
// flux with Harten's fix.
//
// What bounds it.  The two 5-node sums of 5 components are 200 DFMA, and the rest of Alg. 1 with the sensor's
// 3-node branch was another 500 to 2500 FP64 instructions a warp; an SM takes one in 16 clocks, and a
// warp alone 64.  So the sums run on the integer pipe (fixed_point.cuh; nodes as pairs with codes per
// component, weights as limbs), the sensor's differences are integer differences rounded once to
// FP32, the flux is formed from primitive jumps (150 FP64 instructions), and edges with a 3-node (or
// undecided) component are listed for a second kernel of two lanes an edge.
// 24^3 (96,768 edges, 1.5% listed): 93 us, before (one kernel, one thread an edge) 150 us; 12^3: 50 against 67 us.
#include <cuda_runtime.h>

#include <algorithm>

#include "fixed_point.cuh"
#include "fp64_roots.cuh"
#include "fp_convert.cuh"
#include "kernels3d.hpp"
#include "mbar.cuh"
#include "record3.cuh"

namespace hfd {
namespace {

constexpr unsigned kErrIndex = 4u;
// Relative width of the band around each sensor threshold inside which the FP32 decision is taken again
// in FP64 (1e-3 covers the projections' rounding; the Roe state in FP32 is given three times that).
constexpr float kGuard3 = 4e-3f;

constexpr int kEdgeThreads3 = 128;

// ---- states
struct Prim3 {       // of a state w: 1/rho, sqrt(rho), velocity, pressure, E + p, enthalpy
  double ir, r, u[3], p, Ep, H;
};
__device__ __forceinline__ Prim3 prim3(const double* w, double g1) {
  Prim3 a;
  const double y = rsqrt64(w[0]);
  a.r = w[0] * y;
  a.ir = y * y;
#pragma unroll
  for (int k = 0; k < 3; ++k) a.u[k] = w[k + 1] * a.ir;
  a.p = g1 * fma(-0.5, fma(w[1], a.u[0], fma(w[2], a.u[1], w[3] * a.u[2])), w[4]);
  a.Ep = w[4] + a.p;
  a.H = a.Ep * a.ir;
  return a;
}

struct Roe3 {        // the Roe average and the velocity jump
  double u[3], du[3], K, H, c, ic, qn;
};
__device__ __forceinline__ Roe3 roe3(const Prim3& L, const Prim3& R, const double* n, double g1) {
  Roe3 a;
  const double f = R.r * rcp64(L.r + R.r);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    a.du[k] = R.u[k] - L.u[k];
    a.u[k] = fma(f, a.du[k], L.u[k]);
  }
  a.H = fma(f, R.H - L.H, L.H);
  a.K = fma(a.u[0], a.u[0], fma(a.u[1], a.u[1], a.u[2] * a.u[2]));
  const double c2 = g1 * fma(-0.5, a.K, a.H);
  a.ic = rsqrt64(c2);
  a.c = c2 * a.ic;
  a.qn = fma(a.u[0], n[0], fma(a.u[1], n[1], a.u[2] * n[2]));
  return a;
}

// Roe's flux along n with Harten's fix on all five waves, from the primitive jumps: the acoustic and entropy
// strengths from dp, du_n and drho, the two shear waves together as the tangential velocity jump.
__device__ __forceinline__ void roe_flux3(const double* wl, const double* wr, const Prim3& L, const Prim3& R,
                                          const double* n, const Phys3& ph, double* hq) {
  const Roe3 a = roe3(L, R, n, ph.g1);
  const double dun = fma(a.du[0], n[0], fma(a.du[1], n[1], a.du[2] * n[2]));
  // wave strengths with the flux's factor 1/2
  const double hrho = 0.5 * (L.r * R.r), hp = 0.25 * ((R.p - L.p) * (a.ic * a.ic));
  const double rc = (0.5 * hrho) * (a.ic * dun);
  const double a1 = fma(0.5, wr[0] - wl[0], -2.0 * hp);
  const double lam[3] = {a.qn - a.c, a.qn, a.qn + a.c};
  const double del = ph.harten * a.c;
  double al[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    al[i] = fabs(lam[i]);
    if (al[i] < del) al[i] = fma(lam[i], lam[i], del * del) * (ph.half_inv_harten * a.ic);
  }
  const double k0 = al[0] * (hp - rc), k1 = al[1] * a1, k4 = al[2] * (hp + rc), sh = al[1] * hrho;
  double t[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) t[k] = sh * fma(-dun, n[k], a.du[k]);
  const double s04 = k0 + k4, s = s04 + k1, d = (k4 - k0) * a.c;
  const double unl = fma(L.u[0], n[0], fma(L.u[1], n[1], L.u[2] * n[2]));
  const double unr = fma(R.u[0], n[0], fma(R.u[1], n[1], R.u[2] * n[2]));
  const double ml = wl[0] * unl, mr = wr[0] * unr, ps = L.p + R.p;
  hq[0] = fma(0.5, ml + mr, -s);
#pragma unroll
  for (int k = 0; k < 3; ++k)
    hq[k + 1] = fma(0.5, fma(ps, n[k], fma(mr, R.u[k], ml * L.u[k])), -fma(a.u[k], s, fma(d, n[k], t[k])));
  const double ut = fma(a.u[0], t[0], fma(a.u[1], t[1], a.u[2] * t[2]));
  hq[4] = fma(0.5, fma(R.Ep, unr, L.Ep * unl), -fma(a.H, s04, fma(d, a.qn, fma(0.5 * a.K, k1, ut))));
}

// rho > 0 and p > 0 (R16).
__device__ __forceinline__ bool admissible3(const double* w, const Prim3& a) {
  return positive_bits(w[0]) && positive_bits(a.p);
}

__device__ __forceinline__ void ld5(const double* __restrict__ Ua, int v, double* w) {
  const double2* p = reinterpret_cast<const double2*>(Ua + (size_t)20 * v);
  const double2 a = __ldg(p), b = __ldg(p + 1);
  w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
  w[4] = __ldg(Ua + (size_t)20 * v + 4);
}

__device__ __forceinline__ void store_flux3(int e, int V, const double* hq, double* __restrict__ h,
                                            int4* __restrict__ rec) {
  if (rec) {
    st_record3(rec, (size_t)3 * V + e, hq);
    return;
  }
  double* o = h + (size_t)8 * e;
  reinterpret_cast<double2*>(o)[0] = make_double2(hq[0], hq[1]);
  reinterpret_cast<double2*>(o)[1] = make_double2(hq[2], hq[3]);
  o[4] = hq[4];
}

// ---- the sensor in FP32
struct EigF {
  float u[3], n[3], t1[3], t2[3], ic, qn, q1, q2, b1, b2;
};
__device__ __forceinline__ float dot3(const float* a, const float* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

__device__ __forceinline__ void eig32(const float* wl, const float* wr, const float* __restrict__ framef, int E,
                                      int e, float g1, EigF& s) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    s.n[k] = __ldg(framef + (size_t)k * E + e);
    s.t1[k] = __ldg(framef + (size_t)(3 + k) * E + e);
    s.t2[k] = __ldg(framef + (size_t)(6 + k) * E + e);
  }
  const float sl = rsqrtf(wl[0]), sr = rsqrtf(wr[0]);
  const float pl = g1 * (wl[4] - 0.5f * (dot3(wl + 1, wl + 1) * (sl * sl)));
  const float pr = g1 * (wr[4] - 0.5f * (dot3(wr + 1, wr + 1) * (sr * sr)));
  const float is = 1.0f / (wl[0] * sl + wr[0] * sr);
#pragma unroll
  for (int k = 0; k < 3; ++k) s.u[k] = (wl[k + 1] * sl + wr[k + 1] * sr) * is;
  const float H = ((wl[4] + pl) * sl + (wr[4] + pr) * sr) * is, K = dot3(s.u, s.u);
  s.ic = rsqrtf(g1 * (H - 0.5f * K));
  s.qn = dot3(s.u, s.n);
  s.q1 = dot3(s.u, s.t1);
  s.q2 = dot3(s.u, s.t2);
  s.b1 = g1 * s.ic * s.ic;
  s.b2 = 0.5f * s.b1 * K;
}

// c = L a.
__device__ __forceinline__ void to_char32(const EigF& s, const float* a, float* c) {
  const float um = dot3(s.u, a + 1), nm = dot3(s.n, a + 1) * s.ic, qc = s.qn * s.ic;
  c[0] = 0.5f * ((s.b2 + qc) * a[0] - s.b1 * um - nm + s.b1 * a[4]);
  c[1] = (1.0f - s.b2) * a[0] + s.b1 * um - s.b1 * a[4];
  c[2] = dot3(s.t1, a + 1) - s.q1 * a[0];
  c[3] = dot3(s.t2, a + 1) - s.q2 * a[0];
  c[4] = 0.5f * ((s.b2 - qc) * a[0] - s.b1 * um + nm + s.b1 * a[4]);
}

// Uniform WENO5 on the five values u0..u4 (Jiang-Shu indicators, linear weights 1/16, 10/16, 5/16) with every
// weight multiplied by (eps+b1)^2 (eps+b2)^2 (eps+b3)^2, so that the sensor needs no division: t[i] is
// weight i times that product and S their sum; omega_i = t[i] / S.
__device__ __forceinline__ void weno3_32(float u0, float u1, float u2, float u3, float u4, float eps, float* t, float& S) {
  const float e1 = u0 - 2.0f * u1 + u2, f1 = u0 - 4.0f * u1 + 3.0f * u2;
  const float e2 = u1 - 2.0f * u2 + u3, f2 = u1 - u3;
  const float e3 = u2 - 2.0f * u3 + u4, f3 = 3.0f * u2 - 4.0f * u3 + u4;
  float s1 = eps + ((13.0f / 12.0f) * (e1 * e1) + 0.25f * (f1 * f1));
  float s2 = eps + ((13.0f / 12.0f) * (e2 * e2) + 0.25f * (f2 * f2));
  float s3 = eps + ((13.0f / 12.0f) * (e3 * e3) + 0.25f * (f3 * f3));
  s1 *= s1;
  s2 *= s2;
  s3 *= s3;
  t[0] = 0.0625f * (s2 * s3);
  t[1] = 0.625f * (s1 * s3);
  t[2] = 0.3125f * (s1 * s2);
  S = t[0] + t[1] + t[2];
}

// The same from the differences of neighbours, with 33 instead of 45 FP64 instructions.
__device__ __forceinline__ void weno3_64(const double (*c)[5], int q, double eps, double* t, double& S) {
  const double d0 = c[1][q] - c[0][q], d1 = c[2][q] - c[1][q], d2 = c[3][q] - c[2][q], d3 = c[4][q] - c[3][q];
  auto ind = [&](double e, double f) {
    const double b = fma(0.25 * f, f, fma((13.0 / 12.0) * e, e, eps));
    return b * b;
  };
  const double s1 = ind(d1 - d0, fma(3.0, d1, -d0)), s2 = ind(d2 - d1, d1 + d2), s3 = ind(d3 - d2, fma(-3.0, d2, d3));
  t[0] = 0.0625 * (s2 * s3);
  t[1] = 0.625 * (s1 * s3);
  t[2] = 0.3125 * (s1 * s2);
  S = t[0] + t[1] + t[2];
}

// ---- the 5-node sums
// Both sides' sums and the sensor's characteristic differences in FP64 / FP32 from the FP64 states: where a
// weight or a node's value does not fit fixed point.
__device__ __noinline__ void sums64(int e, int E, const int* s, const double* __restrict__ Ua,
                                    const double* __restrict__ w5, const float* __restrict__ framef, float g1,
                                    double* W, float* cf) {
  double wi[5], wj[5];
  ld5(Ua, s[2], wi);
  ld5(Ua, s[3], wj);
  float fi[5], fj[5];
  for (int q = 0; q < 5; ++q) {
    fi[q] = d2f_rn(wi[q]);
    fj[q] = d2f_rn(wj[q]);
    W[q] = W[5 + q] = 0.0;
  }
  EigF sf;
  eig32(fi, fj, framef, E, e, g1, sf);
#pragma unroll 1
  for (int k = 0; k < 6; ++k) {
    const double* a = Ua + (size_t)20 * s[k];
    float d[5];
    for (int q = 0; q < 5; ++q) d[q] = d2f_rn(a[q] - wi[q]);
    to_char32(sf, d, cf + 5 * k);
    for (int side = 0; side < 2; ++side) {
      const int j = k - side;
      if (j < 0 || j > 4) continue;
      for (int g = 0; g < 4; ++g) {
        const double w = w5[(size_t)(20 * side + 4 * j + g) * E + e];
        for (int q = 0; q < 5; ++q) W[5 * side + q] = fma(w, a[5 * g + q], W[5 * side + q]);
      }
    }
  }
}

struct Codes3 { unsigned c[5]; };
__device__ __forceinline__ Codes3 ld_codes3(const uint4* uc, int v) {
  const uint4 a = __ldg(uc + (size_t)2 * v);
  return {{a.x, a.y, a.z, a.w, __ldg(reinterpret_cast<const unsigned*>(uc + (size_t)2 * v + 1))}};
}
__device__ __forceinline__ Codes3 max_codes3(const Codes3& a, const Codes3& b) {
  Codes3 m;
#pragma unroll
  for (int q = 0; q < 5; ++q) m.c[q] = __vmaxu2(a.c[q], b.c[q]);
  return m;
}
__device__ __forceinline__ bool any_raw3(const Codes3& E) {
  const unsigned m = __vmaxu2(__vmaxu2(__vmaxu2(E.c[0], E.c[1]), __vmaxu2(E.c[2], E.c[3])), E.c[4]);
  return (m & 0xffffu) == kFxRaw || (m >> 16) == kFxRaw;
}

// The same in fixed point.  Weights: one exponent per side for the values (we.x: 16 bits each) and d = we.y
// above it for the derivatives of both; all products of component q share the scale
// top_q = max(value code, derivative code + d).  False: some value is not finite, or a side lies too far below
// the scale, which covers the far node of the other side.
__device__ __forceinline__ bool sums_fixed(int e, int E, const int* s, const Edge3Fx& fx, const int4* w5, float g1,
                                           double (*W)[5], float (*cf)[5]) {
  constexpr int L = kBits3;
  Codes3 M = ld_codes3(fx.uc, s[1]);               // of the four nodes that both sides read
#pragma unroll
  for (int k = 2; k < 5; ++k) M = max_codes3(M, ld_codes3(fx.uc, s[k]));
  const Codes3 M0 = max_codes3(M, ld_codes3(fx.uc, s[0])), M1 = max_codes3(M, ld_codes3(fx.uc, s[5]));
  if (any_raw3(max_codes3(M0, M1))) return false;
  const int2 we = __ldg(fx.w5e + e);
  // a component may lie two codes below the scale, a momentum as far as sqrt(rho E) of its side reaches (as in 2D,
  // edge64.cuh: FP64 sums are the more accurate ones below that)
  int top[5], t0[5], t1[5];
  float unit[5];                                   // FP32 value of 2^-(L-1) of the scale
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    t0[q] = max((int)(M0.c[q] & 0xffffu), (int)(M0.c[q] >> 16) + we.y);
    t1[q] = max((int)(M1.c[q] & 0xffffu), (int)(M1.c[q] >> 16) + we.y);
    top[q] = max(t0[q], t1[q]);
    unit[q] = exp2_f32(top[q] - 1022 - (L - 1));
  }
  const int m0 = (t0[0] + t0[4]) >> 1, m1 = (t1[0] + t1[4]) >> 1;
  bool apart = false;
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    const bool mom = q >= 1 && q < 4;
    apart |= top[q] - min(mom ? max(t0[q], m0) : t0[q], mom ? max(t1[q], m1) : t1[q]) > 2;
  }
  if (apart) return false;
  // a pair's limbs at its component's scale (far: some shift of the node is 32 or more)
  auto limbs = [&](int hi, int lo, int d, bool far, int& bh, int& bl) {
    if (far) fx_far(hi, lo, d);
    fx_limbs(hi, lo, d, L);
    bh = hi;
    bl = lo;
  };
  auto shifts = [&](int v, int* dv, int* dd) {
    const Codes3 c = ld_codes3(fx.uc, v);
    int any = 0;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      dv[q] = top[q] - (int)(c.c[q] & 0xffffu);
      dd[q] = top[q] - we.y - (int)(c.c[q] >> 16);
      any |= dv[q] | dd[q];
    }
    return (any & ~31) != 0;
  };
  constexpr float kLow = 1.0f / (1 << L);
  copies_wait();                                   // the thread's own weights
  int ih[5], il[5];
  EigF sf;
  {
    float f[2][5];
#pragma unroll
    for (int k = 1; k >= 0; --k) {                 // the head's values, then the tail's (kept)
      int dv[5], dd[5];
      const bool far = shifts(s[2 + k], dv, dd);
      const int4* src = fx.uf + (size_t)10 * s[2 + k];
      const int4 a = __ldg(src), b = __ldg(src + 1), c = __ldg(src + 8);
      limbs(a.x, a.y, dv[0], far, ih[0], il[0]);
      limbs(a.z, a.w, dv[1], far, ih[1], il[1]);
      limbs(b.x, b.y, dv[2], far, ih[2], il[2]);
      limbs(b.z, b.w, dv[3], far, ih[3], il[3]);
      limbs(c.x, c.y, dv[4], far, ih[4], il[4]);
#pragma unroll
      for (int q = 0; q < 5; ++q) f[k][q] = fmaf((float)il[q], kLow, (float)ih[q]) * unit[q];
    }
    eig32(f[0], f[1], fx.framef, E, e, g1, sf);
  }
  long long hh[2][5], x[2][5];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int q = 0; q < 5; ++q) hh[i][q] = x[i][q] = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    int dv[5], dd[5];
    const bool far = shifts(s[k], dv, dd);
    const int4* src = fx.uf + (size_t)10 * s[k];
    const int4 c0 = __ldg(src + 8), c1 = __ldg(src + 9);      // component 4
    const int2 last[4] = {make_int2(c0.x, c0.y), make_int2(c0.z, c0.w), make_int2(c1.x, c1.y), make_int2(c1.z, c1.w)};
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int4 a = __ldg(src + 2 * g), b = __ldg(src + 2 * g + 1);
      const int* d = g ? dd : dv;
      int bh[5], bl[5];
      limbs(a.x, a.y, d[0], far, bh[0], bl[0]);
      limbs(a.z, a.w, d[1], far, bh[1], bl[1]);
      limbs(b.x, b.y, d[2], far, bh[2], bl[2]);
      limbs(b.z, b.w, d[3], far, bh[3], bl[3]);
      limbs(last[g].x, last[g].y, d[4], far, bh[4], bl[4]);
      if (g == 0) {
        float f[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) f[q] = fmaf((float)(bl[q] - il[q]), kLow, (float)(bh[q] - ih[q])) * unit[q];
        to_char32(sf, f, cf[k]);
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (k < side || k > 4 + side) continue;
        const int2 w = reinterpret_cast<const int2*>(w5 + kEdgeThreads3 * (10 * side + 2 * (k - side) + (g >> 1)))[g & 1];
#pragma unroll
        for (int q = 0; q < 5; ++q) fx_fma(hh[side][q], x[side][q], w.x, w.y, bh[q], bl[q]);
      }
    }
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int ew = side == 0 ? (we.x << 16) >> 16 : we.x >> 16;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      const unsigned lo = fx_carry(hh[side][q], x[side][q], L);
      W[side][q] = fx_to_double(hh[side][q], lo, top[q] + ew + L - 1022 - 2 * (2 * L - 1), L);
    }
  }
  return true;
}

// ------------------------------------------------------------------ k3_edge
// One thread per edge.  Stencil ids (6 x E), frame (9 x E), weights (40 x E) and w3 (18 x E) are
// structure-of-arrays streams; node data are gathered.  A thread's 40 weights are copied to shared memory at
// its start (40 KB a block): loaded where they are used, they cost 12 us more.  h: 8
// doubles per edge (5 used), or rec: record 3 V + e instead.
__global__ void __launch_bounds__(kEdgeThreads3, 3) k3_edge(int E, int V, const int32_t* __restrict__ sten,
                                                  const double* __restrict__ frame,
                                                  const double* __restrict__ w5,
                                                  const double* __restrict__ Ua, double* __restrict__ h,
                                                  int4* __restrict__ rec, Edge3Fx fx, Phys3 ph,
                                                  unsigned* __restrict__ err) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  __shared__ int4 w5s[20 * kEdgeThreads3];
  if (fx.uf) {
#pragma unroll
    for (int i = 0; i < 20; ++i) copy16(w5s + kEdgeThreads3 * i + threadIdx.x, fx.w5f + (size_t)i * E + e);
  }
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
  double W[2][5];
  float cf[6][5];
  if (!fx.uf || !sums_fixed(e, E, s, fx, w5s + threadIdx.x, ph.g1f, W, cf)) {
    double W1[10];
    float c1[30];
    sums64(e, E, s, Ua, w5, fx.framef, ph.g1f, W1, c1);
#pragma unroll
    for (int i = 0; i < 10; ++i) W[i / 5][i % 5] = W1[i];
#pragma unroll
    for (int i = 0; i < 30; ++i) cf[i / 5][i % 5] = c1[i];
  }
  // components to list: rough in FP32, or undecided
  unsigned flag = ph.force_branch == 2 ? 0x3ffu : 0u;
  if (ph.force_branch == 0) {
#pragma unroll
    for (int side = 0; side < 2; ++side)
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        float t[3], S;
        if (side == 0) weno3_32(cf[0][q], cf[1][q], cf[2][q], cf[3][q], cf[4][q], ph.epsf, t, S);
        else           weno3_32(cf[5][q], cf[4][q], cf[3][q], cf[2][q], cf[1][q], ph.epsf, t, S);
        const float mlo = t[0] - ph.sens_lof * S, mhi = ph.sens_hif * S - t[0];
        const bool clear = isfinite(S) && mlo > kGuard3 * S && mhi > kGuard3 * S;
        if (!clear) flag |= 1u << (5 * side + q);
      }
  }
  if (flag) {
    const int i = atomicAdd(fx.count, 1);
    fx.list[i] = make_int2(e, (int)flag);
    double2* o = reinterpret_cast<double2*>(fx.listw + (size_t)12 * i);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      o[3 * side] = make_double2(W[side][0], W[side][1]);
      o[3 * side + 1] = make_double2(W[side][2], W[side][3]);
      o[3 * side + 2] = make_double2(W[side][4], 0.0);
    }
    return;
  }
  Prim3 L = prim3(W[0], ph.g1), R = prim3(W[1], ph.g1);
  // positivity (R16): fall back to the end state of that side
  if (!admissible3(W[0], L)) {
    ld5(Ua, s[2], W[0]);
    L = prim3(W[0], ph.g1);
  }
  if (!admissible3(W[1], R)) {
    ld5(Ua, s[3], W[1]);
    R = prim3(W[1], ph.g1);
  }
  const double n[3] = {__ldg(frame + e), __ldg(frame + (size_t)E + e), __ldg(frame + (size_t)2 * E + e)};
  double hq[5];
  roe_flux3(W[0], W[1], L, R, n, ph, hq);
  store_flux3(e, V, hq, h, rec);
}

// ------------------------------------------------------------------ k3_edge_weno
// The listed edges, two lanes each (one a side), with their 5-node sums from k3_edge: the smooth edges of a
// warp do not wait for the 3-node branch.  16 lanes an edge (one a component and side) make the FP64 chain
// shorter but repeat half of it in every lane: 61 us for 3700 edges, 36 us with two.
__global__ void __launch_bounds__(64) k3_edge_weno(int E, int V, const int32_t* __restrict__ sten,
                                                   const double* __restrict__ frame,
                                                   const double* __restrict__ w3,
                                                   const double* __restrict__ Ua, double* __restrict__ h,
                                                   int4* __restrict__ rec, Edge3Fx fx, Phys3 ph) {
  const int n = *fx.count;
  const int side = threadIdx.x & 1;
  const double g1 = ph.g1;
  const int groups = gridDim.x * (blockDim.x >> 1);
  auto other = [](double x) { return __shfl_xor_sync(0xffffffffu, x, 1); };
  auto other_side = [&](const Prim3& p) {
    Prim3 o;
    o.ir = other(p.ir); o.r = other(p.r); o.p = other(p.p); o.Ep = other(p.Ep); o.H = other(p.H);
#pragma unroll
    for (int k = 0; k < 3; ++k) o.u[k] = other(p.u[k]);
    return o;
  };
  // whole warps run the same number of rounds (shuffles)
  for (int i0 = (blockIdx.x * blockDim.x + (threadIdx.x & ~31)) >> 1; i0 < n; i0 += groups) {
    const bool live = i0 + ((threadIdx.x & 31) >> 1) < n;
    const int i = live ? i0 + ((threadIdx.x & 31) >> 1) : i0;
    const int2 item = fx.list[i];
    const int e = item.x;
    const unsigned mine = ((unsigned)item.y >> (5 * side)) & 0x1fu;
    int s[5];                                      // this side's nodes in WENO order; s[2] is its end
#pragma unroll
    for (int j = 0; j < 5; ++j) s[j] = __ldg(sten + (size_t)(side == 0 ? j : 5 - j) * E + e);
    double nv[3], w[5], end[5];
#pragma unroll
    for (int k = 0; k < 3; ++k) nv[k] = __ldg(frame + (size_t)k * E + e);
    {
      const double2* src = reinterpret_cast<const double2*>(fx.listw + (size_t)12 * i + 6 * side);
      const double2 a = src[0], b = src[1];
      w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
      w[4] = src[2].x;
    }
    ld5(Ua, s[2], end);
    const Prim3 pe = prim3(end, g1), po = other_side(pe);
    const Roe3 a = roe3(side == 0 ? pe : po, side == 0 ? po : pe, nv, g1);
    if (mine) {
      double t1[3], t2[3], hu[3], n1[3], q1 = 0.0, q2 = 0.0;
      const double h3 = 0.5 * g1 * (a.ic * a.ic), hic = 0.5 * a.ic, h0 = 0.5 * (h3 * a.K), n0 = hic * a.qn;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        t1[k] = __ldg(frame + (size_t)(3 + k) * E + e);
        t2[k] = __ldg(frame + (size_t)(6 + k) * E + e);
        hu[k] = h3 * a.u[k];
        n1[k] = hic * nv[k];
        q1 = fma(a.u[k], t1[k], q1);
        q2 = fma(a.u[k], t2[k], q2);
      }
      // c = L v
      auto to_char = [&](const double* v, double* c) {
        const double A = fma(h0, v[0], fma(-hu[0], v[1], fma(-hu[1], v[2], fma(-hu[2], v[3], h3 * v[4]))));
        const double N = fma(n0, v[0], fma(-n1[0], v[1], fma(-n1[1], v[2], -n1[2] * v[3])));
        c[0] = A + N;
        c[1] = fma(-2.0, A, v[0]);
        c[2] = fma(t1[0], v[1], fma(t1[1], v[2], fma(t1[2], v[3], -q1 * v[0])));
        c[3] = fma(t2[0], v[1], fma(t2[1], v[2], fma(t2[2], v[3], -q2 * v[0])));
        c[4] = A - N;
      };
      double C[5], c[5][5];
      to_char(w, C);
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        double v[5];
        ld5(Ua, s[j], v);
        to_char(v, c[j]);
      }
      bool taken = false;
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        if (!((mine >> q) & 1u)) continue;
        double o[3], S;
        weno3_64(c, q, ph.eps, o, S);
        const bool smooth = o[0] > ph.sens_lo * S && o[0] < ph.sens_hi * S;
        if (smooth && ph.force_branch != 2) continue;
        const double* k3 = w3 + (size_t)(9 * side) * E + e;
        auto k = [&](int m) { return __ldg(k3 + (size_t)m * E); };
        const double c1 = k(0) * c[0][q] + k(1) * c[1][q] + k(2) * c[2][q];
        const double c2 = k(3) * c[1][q] + k(4) * c[2][q] + k(5) * c[3][q];
        const double c3 = k(6) * c[2][q] + k(7) * c[3][q] + k(8) * c[4][q];
        const double iS = rcp64(S);
        C[q] = (o[0] * iS) * c1 + (o[1] * iS) * c2 + (o[2] * iS) * c3;
        taken = true;
      }
      if (taken) {                                 // w = R C
        const double s04 = C[0] + C[4], sum = s04 + C[1], d = (C[4] - C[0]) * a.c;
#pragma unroll
        for (int k = 0; k < 3; ++k)
          w[k + 1] = fma(a.u[k], sum, fma(d, nv[k], fma(C[2], t1[k], C[3] * t2[k])));
        w[0] = sum;
        w[4] = fma(a.H, s04, fma(d, a.qn, fma(0.5 * a.K, C[1], fma(q1, C[2], q2 * C[3]))));
      }
    }
    Prim3 pw = prim3(w, g1);
    if (!admissible3(w, pw)) {                     // positivity (R16)
#pragma unroll
      for (int r = 0; r < 5; ++r) w[r] = end[r];
      pw = pe;
    }
    __syncwarp();
    const Prim3 px = other_side(pw);
    double x[5], hq[5];
#pragma unroll
    for (int r = 0; r < 5; ++r) x[r] = other(w[r]);
    if (live && side == 0) {
      roe_flux3(w, x, pw, px, nv, ph, hq);
      store_flux3(e, V, hq, h, rec);
    }
  }
}

// One thread per edge: the 40 weights of its sides (side * 20 + node * 4 + {value, x, y, z}) as limbs, and
// the frame in FP32.  Exponents: one per side for the values, one offset for the derivatives of both.
__global__ void k3_pack_w5(int E, const double* __restrict__ w5, const double* __restrict__ frame, Edge3Fx fx,
                           int* flag) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  for (int k = 0; k < 9; ++k) fx.framef[(size_t)k * E + e] = d2f_rn(frame[(size_t)k * E + e]);
  if (!fx.w5f) return;
  int ev[2] = {-10000, -10000}, off = -10000;
  bool bad = false;
  for (int s = 0; s < 2; ++s) {
    int ed = -10000;
    for (int j = 0; j < 20; ++j) {
      const double w = w5[(size_t)(20 * s + j) * E + e];
      bad |= !isfinite(w);
      if (j % 4 == 0) ev[s] = max(ev[s], exp_above(w));
      else ed = max(ed, exp_above(w));
    }
    bad |= ev[s] == -10000 || abs(ev[s]) > 500;
    if (ed != -10000) off = max(off, ed - ev[s]);
  }
  if (off == -10000) off = 0;
  if (bad || abs(off) > 500) {
    *flag = 1;
    return;
  }
  for (int s = 0; s < 2; ++s)
    for (int j = 0; j < 20; j += 2) {
      const int2 a = coef_limbs(w5[(size_t)(20 * s + j) * E + e], ev[s] + (j % 4 ? off : 0), kBits3);
      const int2 b = coef_limbs(w5[(size_t)(20 * s + j + 1) * E + e], ev[s] + off, kBits3);
      fx.w5f[(size_t)(10 * s + j / 2) * E + e] = make_int4(a.x, a.y, b.x, b.y);
    }
  fx.w5e[e] = make_int2((ev[0] & 0xffff) | (int)((unsigned)ev[1] << 16), off);
}

}  // namespace

cudaError_t launch3_pack_w5(const DevMesh3& m, int* flag, cudaStream_t s) {
  if (m.E == 0) return cudaSuccess;
  k3_pack_w5<<<(m.E + 127) / 128, 128, 0, s>>>(m.E, m.w5, m.frame, m.ex, flag);
  return cudaGetLastError();
}

// Threads per block of k3_edge: an SM partition has its own FP64 unit, so blocks of 32 spread a small mesh best.
cudaError_t launch3_edge(const DevMesh3& m, const Phys3& ph, cudaStream_t s) {
  if (m.E == 0) return cudaSuccess;
  const Edge3Fx fx = edge3_fx(m);
  int4* rec = div3_lanes(m) == 0 ? m.fx.rec : nullptr;
  const int nt = m.E <= kSms * 64 ? 32 : m.E <= kSms * 128 ? 64 : kEdgeThreads3;
  k3_edge<<<(unsigned)((m.E + nt - 1) / nt), nt, 0, s>>>(m.E, m.V, m.sten, m.frame, m.w5, m.Ua, m.h, rec, fx, ph,
                                                         m.err);
  const cudaError_t st = cudaGetLastError();
  if (st != cudaSuccess) return st;
  const int64_t blocks = std::min<int64_t>(((int64_t)m.E * 2 + 63) / 64, kSms * 8);
  k3_edge_weno<<<(unsigned)blocks, 64, 0, s>>>(m.E, m.V, m.sten, m.frame, m.w3, m.Ua, m.h, rec, fx, ph);
  return cudaGetLastError();
}

}  // namespace hfd
