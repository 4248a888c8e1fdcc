// CUDA kernels (sm_103a) of the three-dimensional extension of the Hermite FD residual and
// SSP-RK3 step; FP64 state, fluxes and sums.  Per Runge-Kutta stage:
//   k3_vertex  one thread per vertex: the vertex-major copy of the 20 unknowns and the analytic
//              flux vectors F, G, K (Sec. 2.3, vertex fluxes, in 3D);
//   k3_edge    edge fluxes (edge3d.cu);
//   k3_div_fx  8 lanes per vertex: the CSR gather of the least-squares divergence rows
//              d_0, d_x, d_y, d_z over the vertex fluxes and edge fluxes (Eq.
//              (flux_polynomials) in 3D) in fixed point, fused with the SSP-RK3 stage update;
//   k3_div     the same gather in FP64, 1, 2 or 4 lanes per vertex (chosen lanes; meshes without the fixed-point form).
#include <cuda_runtime.h>

#include "fixed_point.cuh"
#include "fp64_roots.cuh"
#include "kernels3d.hpp"
#include "mbar.cuh"
#include "record3.cuh"

namespace hfd {
namespace {

constexpr unsigned kErrNonfinite = 1u, kErrPositivity = 2u, kErrIndex = 4u;

__device__ __forceinline__ bool finite3(double x) { return isfinite(x); }

// ------------------------------------------------------------------ k3_vertex
// Ua: 20 values per vertex (160 B); FGK: F, G, K per vertex at a stride of 16 (128 B); FX: records 3 v,
// 3 v + 1, 3 v + 2 instead.
template <bool FX>
__global__ void __launch_bounds__(256) k3_vertex(int V, const double* __restrict__ U,
                                                 double* __restrict__ Ua, double* __restrict__ FGK,
                                                 int4* __restrict__ rec, Edge3Fx ex, double g1) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= V) return;
  double w[20];
#pragma unroll
  for (int r = 0; r < 20; ++r) w[r] = U[(size_t)r * V + v];
  double2* ua = reinterpret_cast<double2*>(Ua + (size_t)20 * v);
#pragma unroll
  for (int i = 0; i < 10; ++i) ua[i] = make_double2(w[2 * i], w[2 * i + 1]);
  if (v == 0) *ex.count = 0;                     // the edge kernel's list starts empty
  if (ex.uf) {                                   // pairs and codes for the edge kernel
    int Ev[5], Ed[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      Ev[q] = fx_code(w[q]);
      Ed[q] = max(fx_code(w[5 + q]), max(fx_code(w[10 + q]), fx_code(w[15 + q])));
    }
    int4* o = ex.uf + (size_t)10 * v;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int* E = g ? Ed : Ev;
      const double* a = w + 5 * g;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int2 s = fx_encode(a[2 * i], E[2 * i], kBits3), t = fx_encode(a[2 * i + 1], E[2 * i + 1], kBits3);
        o[2 * g + i] = make_int4(s.x, s.y, t.x, t.y);
      }
    }
    const int2 e0 = fx_encode(w[4], Ev[4], kBits3), e1 = fx_encode(w[9], Ed[4], kBits3);
    const int2 e2 = fx_encode(w[14], Ed[4], kBits3), e3 = fx_encode(w[19], Ed[4], kBits3);
    o[8] = make_int4(e0.x, e0.y, e1.x, e1.y);
    o[9] = make_int4(e2.x, e2.y, e3.x, e3.y);
    unsigned c[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) c[q] = (unsigned)Ev[q] | ((unsigned)Ed[q] << 16);
    ex.uc[2 * (size_t)v] = make_uint4(c[0], c[1], c[2], c[3]);
    ex.uc[2 * (size_t)v + 1] = make_uint4(c[4], 0u, 0u, 0u);
  }
  const double ir = rcp64(w[0]);
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
  for (int j = m.vptr[v]; j < m.vptr[v + 1] && !isnan(s); ++j)      // NaN stays NaN
#pragma unroll 1
    for (int d = 2; d >= 0; --d)
      s = fma(m.cv[(size_t)12 * j + 3 * k + d], value((size_t)3 * m.vidx[j] + d), s);
  for (int j = m.eptr[v]; j < m.eptr[v + 1] && !isnan(s); ++j)
    s = fma(m.ce[(size_t)4 * j + k], value((size_t)3 * V + m.eidx[j]), s);
  return s;
}

// copy16 with a copy left in L1.
__device__ __forceinline__ void copy16_l1(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
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
  if (div3_lanes(m) == 0) k3_vertex<true><<<nb, 256, 0, s>>>(m.V, U, m.Ua, m.FGK, m.fx.rec, edge3_fx(m), ph.g1);
  else                    k3_vertex<false><<<nb, 256, 0, s>>>(m.V, U, m.Ua, m.FGK, m.fx.rec, edge3_fx(m), ph.g1);
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
