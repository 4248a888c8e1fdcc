// The FP64 edge's interpolation shared by the forward kernels (kernels.cu) and the adjoint
// (adjoint.cu): states, sensor, and the 5-node sums in fixed point.
#pragma once
#include "fixed_point.cuh"
#include "fp_convert.cuh"
#include "kernels.hpp"

namespace hfd {

// ------------------------------------------------------------------ physics (Sec. 2.3)
template <typename T>
__device__ __forceinline__ T pressure(const T* w, T g1) {
  return g1 * (w[3] - T(0.5) * (w[1] * w[1] + w[2] * w[2]) / w[0]);
}

// Roe-averaged u, v, H, c of two states (Alg. 1, first step; also the Riemann flux).
template <typename T>
__device__ __forceinline__ void roe_avg(const T* wl, const T* wr, T g1, T& u, T& v, T& H, T& c) {
  T rl = sqrt(wl[0]), rr = sqrt(wr[0]);
  T irl = T(1) / rl, irr = T(1) / rr, is = T(1) / (rl + rr);
  T pl = pressure(wl, g1), pr = pressure(wr, g1);
  u = (wl[1] * irl + wr[1] * irr) * is;
  v = (wl[2] * irl + wr[2] * irr) * is;
  H = ((wl[3] + pl) * irl + (wr[3] + pr) * irr) * is;
  c = sqrt(g1 * (H - T(0.5) * (u * u + v * v)));
}

// Left eigenvectors (rows of L = R^-1) of the Euler flux Jacobian along n (Alg. 1, step 2).
template <typename T>
__device__ __forceinline__ void left_ev(T u, T v, T c, T nx, T ny, T g1, T (*L)[4]) {
  T qn = u * nx + v * ny, qt = -u * ny + v * nx;
  T ic = T(1) / c;
  T b1 = g1 * ic * ic, b2 = T(0.5) * b1 * (u * u + v * v);
  L[0][0] = T(0.5) * (b2 + qn * ic);
  L[0][1] = T(-0.5) * (b1 * u + nx * ic);
  L[0][2] = T(-0.5) * (b1 * v + ny * ic);
  L[0][3] = T(0.5) * b1;
  L[1][0] = T(1) - b2;
  L[1][1] = b1 * u;
  L[1][2] = b1 * v;
  L[1][3] = -b1;
  L[2][0] = -qt;
  L[2][1] = -ny;
  L[2][2] = nx;
  L[2][3] = T(0);
  L[3][0] = T(0.5) * (b2 - qn * ic);
  L[3][1] = T(-0.5) * (b1 * u - nx * ic);
  L[3][2] = T(-0.5) * (b1 * v - ny * ic);
  L[3][3] = T(0.5) * b1;
}

constexpr float kGuard = 1e-3f;

// Jiang-Shu smoothness indicators of the three sub-stencils of u0..u4 (uniform WENO5, R2).
template <typename T>
__device__ __forceinline__ void smoothness(T u0, T u1, T u2, T u3, T u4, T* b) {
  T a = u0 - T(2) * u1 + u2, e = u0 - T(4) * u1 + T(3) * u2;
  b[0] = T(13.0 / 12.0) * a * a + T(0.25) * e * e;
  a = u1 - T(2) * u2 + u3;
  e = u1 - u3;
  b[1] = T(13.0 / 12.0) * a * a + T(0.25) * e * e;
  a = u2 - T(2) * u3 + u4;
  e = T(3) * u2 - T(4) * u3 + u4;
  b[2] = T(13.0 / 12.0) * a * a + T(0.25) * e * e;
}

// ---- FP64 edges
// What the FP64 edge kernel reads and writes beside the plain arrays (null: not used): the vertex
// fluxes of the folded double-float divergence; the fixed-point divergence's vertex codes and edge
// codes; the nodes' stored pairs and codes and the 5-node weights in fixed point.
struct EdgeFx {
  const double* FGd = nullptr;
  const uint2* ex = nullptr;
  uint2* ee = nullptr;
  const int4* uf = nullptr;        // [V][12] pairs: w, w_x, w_y
  const uint4* uc = nullptr;       // [V] 8 codes of 16 bits: w (4), w_x and w_y together (4)
  const int2* w5f = nullptr;       // [30][Ef] limb pairs, order of w5
  const int2* w5e = nullptr;       // [Ef] exponents (see pack_w5)
  int2* list = nullptr;            // edges left to k_edge_weno: {edge, components}
  int* count = nullptr;
};

// The sensor in FP32 on one component's five differences: the 3-node branch, and the guard band.
__device__ __forceinline__ void sensor_bits(float u0, float u1, float u2, float u3, float u4, const Phys& ph,
                                            bool& rough, bool& amb) {
  float b[3];
  smoothness(u0, u1, u2, u3, u4, b);
  const float eps = ph.epsf;
  float s0 = eps + b[0], s1 = eps + b[1], s2 = eps + b[2];
  s0 *= s0; s1 *= s1; s2 *= s2;
  const float t0 = 0.0625f * s1 * s2, t1 = 0.625f * s0 * s2, t2 = 0.3125f * s0 * s1;
  const float S = t0 + t1 + t2;
  const float mlo = t0 - ph.sens_lof * S, mhi = ph.sens_hif * S - t0;
  rough = !(mlo > 0.f && mhi > 0.f);
  amb = !(fabsf(mlo) > kGuard * S && fabsf(mhi) > kGuard * S);
}

// Bits (side*4+q) of the sensor in FP32 on the characteristic values cf of the nodes' differences from
// the tail state: the 3-node branch, and the guard band.
__device__ __forceinline__ void sensor32(const float (*cf)[4], const Phys& ph, unsigned& rough, unsigned& amb) {
  rough = amb = 0;
#pragma unroll
  for (int side = 0; side < 2; ++side)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float u0, u1, u2, u3, u4;
      if (side == 0) { u0 = cf[0][q]; u1 = cf[1][q]; u2 = cf[2][q]; u3 = cf[3][q]; u4 = cf[4][q]; }
      else           { u0 = cf[5][q]; u1 = cf[4][q]; u2 = cf[3][q]; u3 = cf[2][q]; u4 = cf[1][q]; }
      bool r, m;
      sensor_bits(u0, u1, u2, u3, u4, ph, r, m);
      const unsigned bit = 1u << (side * 4 + q);
      if (r) rough |= bit;
      if (m) amb |= bit;
    }
  if (ph.force_branch == 1) rough = amb = 0u;                 // every side 5-node
  else if (ph.force_branch == 2) { rough = 0xffu; amb = 0u; } // every side 3-node WENO
}

// Eight codes of 16 bits: the larger of each; true if one is kFxRaw.
__device__ __forceinline__ uint4 max_codes8(uint4 a, uint4 b) {
  return make_uint4(__vmaxu2(a.x, b.x), __vmaxu2(a.y, b.y), __vmaxu2(a.z, b.z), __vmaxu2(a.w, b.w));
}
__device__ __forceinline__ bool any_raw8(uint4 a) {
  const unsigned m = __vmaxu2(__vmaxu2(a.x, a.y), __vmaxu2(a.z, a.w));
  return (m & 0xffffu) == kFxRaw || (m >> 16) == kFxRaw;
}

// A side's sum is cut at 2^-57 of the scale that it shares with the other side, whose far node it does not
// read.  True if no component of either side lies more than two codes (a factor of four) below that scale:
// over the weights of a 16x16 mesh and values within a factor e, the sums' errors in units of 2^-53 of the
// value are then 0.70 rms and 3.0 at most, those of FP64 sums 1.07 and 5.1 (at the scale itself 0.43 and
// 1.2, three codes below it 1.17 and 5.7).  A momentum is compared with sqrt(rho E) of its side
// too, the size of the terms that it is added to in the flux, so that momenta around zero send no edge to
// FP64.  m: codes of the four middle nodes, a, b: of the far ones (values, then derivatives), d: how far the
// derivatives' weights lie above the values'; top: the components' scales, 16 bits each.
__device__ __forceinline__ bool sides_in_range(uint4 m, uint4 a, uint4 b, int d, uint2& top) {
  const unsigned dd = (unsigned)d & 0xffffu, d2 = dd | (dd << 16);
  auto tops = [&](const uint4& n) {
    return make_uint2(__vmaxs2(__vmaxu2(m.x, n.x), __vadd2(__vmaxu2(m.z, n.z), d2)),
                      __vmaxs2(__vmaxu2(m.y, n.y), __vadd2(__vmaxu2(m.w, n.w), d2)));
  };
  auto refs = [](const uint2& t) {
    const unsigned mom = ((t.x & 0xffffu) + (t.y >> 16)) >> 1;       // of density and energy (both positive codes)
    return make_uint2(__vmaxs2(t.x, mom << 16), __vmaxs2(t.y, mom));
  };
  const uint2 ta = tops(a), tb = tops(b), ra = refs(ta), rb = refs(tb);
  top = make_uint2(__vmaxs2(ta.x, tb.x), __vmaxs2(ta.y, tb.y));
  return (__vcmpgts2(__vsub2(top.x, __vmins2(ra.x, rb.x)), 0x00020002u) |
          __vcmpgts2(__vsub2(top.y, __vmins2(ra.y, rb.y)), 0x00020002u)) == 0u;
}

// The 5-node sums of both sides in fixed point (fixed_point.cuh): 120 DFMA, half of the smooth edge's
// FP64 instructions, become 360 integer multiply-adds.  The nodes' 12 values are stored as pairs with
// two codes per component (values; derivatives), the weights as limbs with one exponent per side
// for the values (we.x: 16 bits each) and d = we.y above it for the derivatives (one d for both
// sides, so that one alignment of the nodes serves both).  All products of component q then share the
// scale top_q = max(value code, derivative code + d).  Also the sensor's characteristic values of
// the differences from the tail state: the integer differences, rounded to FP32.  False: some value
// is not finite or a side lies too far below the common scale, and nothing is written.
// SHARED: the thread's weights are in shared memory (stage_w5), at ws.
constexpr int kEdgeBlock = 128;                    // threads of a block that stages them, at most
__device__ __forceinline__ void stage_w5(int2* ws, const EdgeFx& fx, int Ef, int e) {
#pragma unroll
  for (int i = 0; i < 30; ++i)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(ws + kEdgeBlock * i)),
                 "l"(fx.w5f + (size_t)i * Ef + e)
                 : "memory");
}
template <bool SHARED>
__device__ __forceinline__ bool edge_fixed64(int e, int Ef, const int* s, const EdgeFx& fx, float nx, float ny,
                                             const Phys& ph, double (*W)[4], float (*cf)[4],
                                             const int2* ws = nullptr) {
  constexpr int L = kFxBits;
  uint4 E = __ldg(fx.uc + s[1]);
#pragma unroll
  for (int k = 2; k < 5; ++k) E = max_codes8(E, __ldg(fx.uc + s[k]));
  const uint4 far0 = __ldg(fx.uc + s[0]), far1 = __ldg(fx.uc + s[5]);
  const int2 we = __ldg(fx.w5e + e);
  uint2 tops;
  if (any_raw8(max_codes8(E, max_codes8(far0, far1))) || !sides_in_range(E, far0, far1, we.y, tops)) return false;
  int top[4];
  float unit[4];                                   // FP32 value of 2^-(L-1) of the scale
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    top[q] = (int)((q & 2 ? tops.y : tops.x) >> (16 * (q & 1))) & 0xffff;
    unit[q] = exp2_f32(top[q] - 1022 - (L - 1));
  }
  // a node's codes, read again where they are used (L1) rather than held for all six nodes; its shifts;
  // and the limbs of its four values (g = 0), x derivatives (1) or y derivatives (2)
  auto shifts = [&](int k, int* dw, int* dd) {
    uint4 c;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(c.x), "=r"(c.y), "=r"(c.z), "=r"(c.w) : "l"(fx.uc + s[k]));
    dw[0] = top[0] - (int)(c.x & 0xffffu);
    dw[1] = top[1] - (int)(c.x >> 16);
    dw[2] = top[2] - (int)(c.y & 0xffffu);
    dw[3] = top[3] - (int)(c.y >> 16);
    dd[0] = top[0] - we.y - (int)(c.z & 0xffffu);
    dd[1] = top[1] - we.y - (int)(c.z >> 16);
    dd[2] = top[2] - we.y - (int)(c.w & 0xffffu);
    dd[3] = top[3] - we.y - (int)(c.w >> 16);
    return ((dw[0] | dw[1] | dw[2] | dw[3] | dd[0] | dd[1] | dd[2] | dd[3]) & ~31) != 0;
  };
  auto group = [&](int k, int g, const int* d0, bool far, int* bh, int* bl) {
    const int4* src = fx.uf + 6 * (size_t)s[k] + 2 * g;
    const int4 a = __ldg(src), b = __ldg(src + 1);
    int d[4] = {d0[0], d0[1], d0[2], d0[3]};
    bh[0] = a.x; bl[0] = a.y; bh[1] = a.z; bl[1] = a.w;
    bh[2] = b.x; bl[2] = b.y; bh[3] = b.z; bl[3] = b.w;
    if (far) {
#pragma unroll
      for (int q = 0; q < 4; ++q) fx_far(bh[q], bl[q], d[q]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) fx_limbs(bh[q], bl[q], d[q], L);
  };
  constexpr float kLow = 1.0f / (1 << L);
  int ih[4], il[4];
  float Lf[4][4];
  {
    int jh[4], jl[4], dw[4], dd[4];
    bool far = shifts(2, dw, dd);
    group(2, 0, dw, far, ih, il);
    far = shifts(3, dw, dd);
    group(3, 0, dw, far, jh, jl);
    float fi[4], fj[4], u, v, H, cs;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      fi[q] = fmaf((float)il[q], kLow, (float)ih[q]) * unit[q];
      fj[q] = fmaf((float)jl[q], kLow, (float)jh[q]) * unit[q];
    }
    roe_avg(fi, fj, ph.g1f, u, v, H, cs);
    left_ev(u, v, cs, nx, ny, ph.g1f, Lf);
  }
  if (SHARED) asm volatile("cp.async.wait_all;" ::: "memory");
  long long hh[2][4], x[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) hh[i][q] = x[i][q] = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    int dw[4], dd[4];
    const bool far = shifts(k, dw, dd);
#pragma unroll
    for (int g = 0; g < 3; ++g) {
      int bh[4], bl[4];
      group(k, g, g ? dd : dw, far, bh, bl);
      if (g == 0) {
        float d[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          d[q] = fmaf((float)(bl[q] - il[q]), kLow, (float)(bh[q] - ih[q])) * unit[q];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          cf[k][q] = Lf[q][0] * d[0] + Lf[q][1] * d[1] + Lf[q][2] * d[2] + Lf[q][3] * d[3];
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        if (k < side || k > 4 + side) continue;
        const int i = 15 * side + 3 * (k - side) + g;
        const int2 w = SHARED ? ws[kEdgeBlock * i] : __ldg(fx.w5f + (size_t)i * Ef + e);
#pragma unroll
        for (int q = 0; q < 4; ++q) fx_fma(hh[side][q], x[side][q], w.x, w.y, bh[q], bl[q]);
      }
    }
  }
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int ew = side == 0 ? (we.x << 16) >> 16 : we.x >> 16;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const unsigned lo = fx_carry(hh[side][q], x[side][q], L);
      W[side][q] = fx_to_double(hh[side][q], lo, top[q] + ew + L - 1022 - 2 * (2 * L - 1), L);
    }
  }
  return true;
}

}  // namespace hfd
