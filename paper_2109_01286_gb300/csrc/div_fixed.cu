// The FP64 divergence in fixed point (k_div_fx): R = -div f + div f_vis and the fused stage
// update, with the sums of products on the integer pipe (fixed_point.cuh).
//
// What bounds it.  The plain FP64 kernel issues 24 DFMA per stencil vertex and 12 per stencil edge
// (1010 per row at the mean 20 vertices and 44.2 edges), and the FP64 pipe, 2 lanes per clock
// and SM, takes 505 clocks of an SM for them; the row's coefficients and indices, 2.3 KB, need about
// 120 clocks of the SM's share of the HBM.  In fixed point the row is 3030 integer multiply-adds of
// two issue slots each and about as many other instructions, 110 clocks if every slot were used; at
// 16 warps an SM (128 registers) 41% are.  Four-quadrant 400x400 (160,000 rows, one stage): 168 us, the
// plain kernel 334 us; 256x256: 84 us against 184 us; 24x24 with 8 lanes: 12 us against 45 us.
// Measured slower: coefficients staged in shared memory with the fluxes (50 KB a block leave 8
// warps an SM; 199 us), or streamed through a cp.async ring per lane (204 us); fluxes gathered from
// global memory entry by entry (one L2 latency each; 194 us); two lanes an entry with half the
// components each (183 us).
//
// Layout.  Entries come in chunks of four (padded with zero coefficients): four consecutive lanes
// take one chunk, so each 16-byte coefficient load of a group covers 64 contiguous bytes.  A
// vertex chunk holds [row k = 0, 1, 2][entry] x {F hi, F lo, G hi, G lo}, an edge chunk
// [entry] x {d0 hi, d0 lo, dx hi, dx lo} and [entry] x {dy hi, dy lo}: the bytes of the FP64
// coefficients.  k_vertex and k_edge write the fluxes in the stored form of fixed_point.cuh with
// codes per vertex and per edge; an edge's codes cover its end vertices, so the row's scale is the
// largest over its edges.  Tiles of 16 rows: a tile reads about 60 distinct vertices and 190 edges, a
// quarter of its rows' entries; 8 in meshes of fewer than kFxSmallRows, for more blocks.  The line is not
// sharp: a residual with tiles of 8 and 16 and the better lane count took 35.2 and 33.2 us with 576 rows, 49.7 and
// 49.5 with 10,000, 75.2 and 74.5 with 19,881, 85.2 and 83.2 with 25,600, 226 and 225 with 90,000;
// with 4 and 8 lanes 37 and 35 us with 576 rows, 50 and 52 with 10,000, 76 and 75 with 19,881, 126 and 124
// with 40,000, 225 and 235 with 90,000.
#include <algorithm>

#include "div_common.cuh"
#include "fixed_point.cuh"
#include "mbar.cuh"

namespace hfd {

// G lanes share a row: they take its entries in turn and hold all 12 sums (rows d_0, d_x, d_y by
// components, 48 registers), so that an entry's index, codes and coefficients are read once for its 72
// multiply-adds.

// Four exponent codes, 16 bits each; the larger of each.
__device__ __forceinline__ uint2 max_codes(uint2 a, uint2 b) {
  return make_uint2(__vmaxu2(a.x, b.x), __vmaxu2(a.y, b.y));
}

template <int G>
__device__ __forceinline__ uint2 group_max_codes(uint2 e) {
#pragma unroll
  for (int o = 1; o < G; o <<= 1) {
    const unsigned x = __shfl_xor_sync(0xffffffffu, e.x, o, G), y = __shfl_xor_sync(0xffffffffu, e.y, o, G);
    e = max_codes(e, make_uint2(x, y));
  }
  return e;
}

__device__ __forceinline__ int code_of(uint2 e, int q) {
  return (int)((q & 2 ? e.y : e.x) >> (16 * (q & 1))) & 0xffff;
}

__device__ __forceinline__ bool any_raw(uint2 e) {
  return code_of(e, 0) == kFxRaw || code_of(e, 1) == kFxRaw || code_of(e, 2) == kFxRaw || code_of(e, 3) == kFxRaw;
}

struct FxAcc {
  long long hh[12], x[12];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 12; ++i) { hh[i] = 0; x[i] = 0; }
  }
  __device__ __forceinline__ void carry() {
#pragma unroll
    for (int i = 0; i < 12; ++i) x[i] = fx_carry(hh[i], x[i], kFxBits);
  }
  // the four components of a flux vector (limbs a: components 0, 1; b: 2, 3) times the
  // coefficients (ch, cl) of row d_k
  __device__ __forceinline__ void row(int k, int4 a, int4 b, int ch, int cl) {
    fx_fma(hh[4 * k], x[4 * k], ch, cl, a.x, a.y);
    fx_fma(hh[4 * k + 1], x[4 * k + 1], ch, cl, a.z, a.w);
    fx_fma(hh[4 * k + 2], x[4 * k + 2], ch, cl, b.x, b.y);
    fx_fma(hh[4 * k + 3], x[4 * k + 3], ch, cl, b.z, b.w);
  }
};

// An entry's shifts to the row's scale, from its code word; true if one is 32 or more.
__device__ __forceinline__ bool shifts(uint2 E, uint2 e, int* d) {
  const uint2 t = make_uint2(E.x - e.x, E.y - e.y);
  d[0] = (int)(t.x & 0xffffu);
  d[1] = (int)(t.x >> 16);
  d[2] = (int)(t.y & 0xffffu);
  d[3] = (int)(t.y >> 16);
  return ((t.x | t.y) & 0xffe0ffe0u) != 0u;
}

// Four components' stored pairs to limbs at the row's scale.
__device__ __forceinline__ void limbs4(int4& a, int4& b, const int* d) {
  constexpr int L = kFxBits;
  fx_limbs(a.x, a.y, d[0], L);
  fx_limbs(a.z, a.w, d[1], L);
  fx_limbs(b.x, b.y, d[2], L);
  fx_limbs(b.z, b.w, d[3], L);
}
__device__ __forceinline__ void far4(int4& a, int4& b, int* d) {
  fx_far(a.x, a.y, d[0]);
  fx_far(a.z, a.w, d[1]);
  fx_far(b.x, b.y, d[2]);
  fx_far(b.z, b.w, d[3]);
}

// The vertex entries of one row (Euler fluxes with cv, or viscous fluxes with cvis): lane `lane` of
// G takes the entries first + lane, first + lane + G, ... (first: a multiple of G).  id: the entries' positions in the tile's staged
// vertices (four planes of 16-byte pieces F01, F23, G01, G23, n pieces each; sx: code words), cc:
// the row's coefficient chunks, E: the row's codes.
template <int G>
__device__ __forceinline__ void vertex_entries(FxAcc& A, int first, int entries, int lane, uint2 E, const uint16_t* id,
                                               const int4* cc, const int4* planes, int n, const uint2* sx) {
  cc += 12 * (lane >> 2) + (lane & 3) + 3 * first;
  for (int j = first + lane; j < entries; j += G, cc += 3 * G) {
    const int u = id[j];
    const int4* f = planes + u;
    int4 f0 = f[0], f1 = f[n], g0 = f[2 * n], g1 = f[3 * n];
    const int4 k0 = __ldg(cc), k1 = __ldg(cc + 4), k2 = __ldg(cc + 8);
    int d[4];
    if (shifts(E, sx[u], d)) {
      int df[4] = {d[0], d[1], d[2], d[3]};
      far4(f0, f1, df);
      far4(g0, g1, d);
    }
    limbs4(f0, f1, d);
    A.row(0, f0, f1, k0.x, k0.y);
    A.row(1, f0, f1, k1.x, k1.y);
    A.row(2, f0, f1, k2.x, k2.y);
    limbs4(g0, g1, d);
    A.row(0, g0, g1, k0.z, k0.w);
    A.row(1, g0, g1, k1.z, k1.w);
    A.row(2, g0, g1, k2.z, k2.w);
  }
}

template <int G>
__device__ __forceinline__ void edge_entries(FxAcc& A, int first, int entries, int lane, uint2 E, const uint16_t* id,
                                             const unsigned char* cc, const int4* planes, int n,
                                             const uint2* sx) {
  const unsigned char* c01 = cc + 96 * (lane >> 2) + 16 * (lane & 3) + 24 * first;
  const unsigned char* c2 = cc + 96 * (lane >> 2) + 64 + 8 * (lane & 3) + 24 * first;
  for (int j = first + lane; j < entries; j += G, c01 += 24 * G, c2 += 24 * G) {
    const int u = id[j];
    int4 h0 = planes[u], h1 = planes[n + u];
    const int4 k01 = __ldg(reinterpret_cast<const int4*>(c01));
    const int2 k2 = __ldg(reinterpret_cast<const int2*>(c2));
    int d[4];
    if (shifts(E, sx[u], d)) far4(h0, h1, d);
    limbs4(h0, h1, d);
    A.row(0, h0, h1, k01.x, k01.y);
    A.row(1, h0, h1, k01.z, k01.w);
    A.row(2, h0, h1, k2.x, k2.y);
  }
}

// Calls f(first, end) for all entries of a row: at once, or (CARRY) in spans of at most kFxCarry products of
// a lane, `per` an entry, after each of which the cross sums are carried over (the same sums, so the same
// bits).  One row of more than about 150 products sends its mesh or batch to the kernel with CARRY: 160,000
// rows and a mesh whose largest row has 282 products 400 us a residual (386 us with 28-bit limbs for every
// row, which need no carry but hold 55-bit factors), 582 products 455 us (986 us in FP64); 372 us
// beside rows of ordinary length.  Most of that is the shared memory of the largest tile.
template <int G, bool CARRY, typename F>
__device__ __forceinline__ void in_spans(FxAcc& A, int entries, int per, F f) {
  if (!CARRY) {
    f(0, entries);
    return;
  }
  const int span = G * (kFxCarry / per);
#pragma unroll 1
  for (int first = 0; first < entries; first += span) {
    f(first, min(entries, first + span));
    A.carry();
  }
}

// Adds the lanes' sums (exactly) and leaves each lane its share of the 12 rows (RowShare): value i
// is (hh[i] 2^L + lo[i]) in units of the row's scale.
template <int G>
__device__ __forceinline__ void reduce_rows(FxAcc& A, unsigned* lo, int lane) {
#pragma unroll
  for (int i = 0; i < 12; ++i) lo[i] = fx_carry(A.hh[i], A.x[i], kFxBits);
  reduce_scatter12<G>(A.hh, lane);
  reduce_scatter12<G>(lo, lane);
}

// Exponents of the rows' coefficients: 3 signed 10-bit fields.
__device__ __forceinline__ int coef_exp(int packed, int k) { return (packed << (22 - 10 * k)) >> 22; }

// One sum (row d_k, component q) of a row some of whose fluxes are not finite, in FP64 as the plain
// kernel evaluates it: -div f + div f_vis.  NaN stays NaN, so the first one ends the sum.
__device__ __noinline__ double fallback_sum(const DivFx& m, int r, int k, int q, bool visc) {
  const int half = q >> 1;
  double R = 0.0;
  const unsigned *mex = reinterpret_cast<const unsigned*>(m.ex), *mexv = reinterpret_cast<const unsigned*>(m.exv);
  const unsigned* mee = reinterpret_cast<const unsigned*>(m.ee);
  auto code = [&](unsigned e) { return (int)(e >> (16 * (q & 1))) & 0xffff; };
  auto coef = [&](int hi, int lo, int ke) {
    return scalbn((double)((long long)hi * (1ll << kFxBits) + lo), coef_exp(ke, k) - (2 * kFxBits - 1));
  };
  auto flux = [&](const int4* base, size_t piece, unsigned e) {
    const int4 p = base[piece + half];
    return fx_decode(q & 1 ? make_int2(p.z, p.w) : make_int2(p.x, p.y), code(e), kFxBits);
  };
  auto vertices = [&](const int4* cv, const int4* FG, const unsigned* ex, int ke, double sign) {
    const int n0 = m.nvptr[r], N = m.nvptr[r + 1] - n0;
    for (int j = 0; j < N; ++j) {
      const size_t u = m.nvidx[n0 + j];
      const int4 c = cv[12 * ((size_t)m.vptr[r] + (j >> 2)) + 4 * k + (j & 3)];
      const unsigned e = ex[2 * u + half];
      R = fma(sign * coef(c.x, c.y, ke), flux(FG, 4 * u, e), R);
      R = fma(sign * coef(c.z, c.w, ke), flux(FG, 4 * u + 2, e), R);
      if (isnan(R)) return;
    }
  };
  const int2 ke = m.cexp[r];
  vertices(m.cv, m.FG, mex, ke.x, -1.0);
  if (isnan(R)) return R;
  const int m0 = m.neptr[r], M = m.neptr[r + 1] - m0;
  for (int j = 0; j < M; ++j) {
    const size_t s = m.neidx[m0 + j];
    const unsigned char* ck = m.ce + 96 * ((size_t)m.eptr[r] + (j >> 2));
    const int4 k01 = reinterpret_cast<const int4*>(ck)[j & 3];
    const int2 k2 = reinterpret_cast<const int2*>(ck + 64)[j & 3];
    const double c = k == 0 ? coef(k01.x, k01.y, ke.x) : k == 1 ? coef(k01.z, k01.w, ke.x)
                                                                : coef(k2.x, k2.y, ke.x);
    R = fma(-c, flux(m.h, 2 * s, mee[2 * s + half]), R);
    if (isnan(R)) return R;
  }
  if (visc) vertices(m.cvis, m.FGv, mexv, ke.y, 1.0);
  return R;
}

__device__ __forceinline__ void copy8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

// One block: the rows of tile blockIdx.x, G lanes each.  Three rounds of loads: the tile's record
// (the ids of the vertices and edges its rows read, each once, and the entries' positions in them)
// and its coefficients by bulk copies, contiguous in their arrays; the listed fluxes, all at once; the
// state.  Everything else reads shared memory.
template <int G, bool CARRY, bool VISC>
__global__ void __launch_bounds__(128, 4) k_div_fx(DivFx m, StageArgs sa, const int32_t* __restrict__ vmem,
                                                const unsigned long long* dtbits, double cfl,
                                                double* dt_last, unsigned* err) {
  constexpr int L = kFxBits;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) unsigned long long bar;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int r0 = blockIdx.x * m.rows, r1 = min(r0 + m.rows, m.A);
  const int r = r0 + tid / G, lane = tid % G;
  const bool live = r < m.A;
  const int4 head = __ldg(m.head + blockIdx.x);
  const int cb = __ldg(m.vptr + r0), mb = __ldg(m.eptr + r0);
  const int nvc = __ldg(m.vptr + r1) - cb, nec = __ldg(m.eptr + r1) - mb;
  const int nv = head.z, ne = head.w;
  // shared memory: record | fluxes | codes
  int4* sF = reinterpret_cast<int4*>(smem + 16 * head.y);
  int4* sH = sF + 4 * nv;
  int4* sFv = sH + 2 * ne;
  uint2* sx = reinterpret_cast<uint2*>(sFv + (VISC ? 4 * nv : 0));
  uint2* sxv = sx + nv;
  uint2* sxe = sxv + (VISC ? nv : 0);
  if (tid == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
    mbar_expect_tx(&bar, 16u * (unsigned)head.y);
    bulk_g2s(smem, m.rec + head.x, 16u * head.y, &bar);
    bulk_prefetch(m.ce + 96 * (size_t)mb, 96u * nec);
    bulk_prefetch(m.cv + 12 * (size_t)cb, 192u * nvc);
    if (VISC) bulk_prefetch(m.cvis + 12 * (size_t)cb, 192u * nvc);
  }
  __syncthreads();
  int m0 = 0, mc = 0, c0 = 0, nc = 0;
  int2 ke = make_int2(0, 0);
  if (live) {
    m0 = __ldg(m.eptr + r) - mb;
    mc = __ldg(m.eptr + r + 1) - mb - m0;
    c0 = __ldg(m.vptr + r) - cb;
    nc = __ldg(m.vptr + r + 1) - cb - c0;
    ke = __ldg(m.cexp + r);
  }
  const int32_t* ids = reinterpret_cast<const int32_t*>(smem);
  const uint16_t* vid = reinterpret_cast<const uint16_t*>(ids + ((nv + ne + 3) & ~3)) + 4 * c0;
  const uint16_t* eid = vid - 4 * c0 + 4 * nvc + 4 * m0;
  bool ok = mbar_wait(&bar, 0);
  if (ok) {
    for (int i = tid; i < 4 * nv; i += nt) {
      const size_t u = (size_t)chk_idx(ids[i >> 2], m.V, err);
      const int p = i & 3;
      copy16(sF + p * nv + (i >> 2), m.FG + 4 * u + p);
      if (VISC) copy16(sFv + p * nv + (i >> 2), m.FGv + 4 * u + p);
    }
    for (int i = tid; i < 2 * ne; i += nt)
      copy16(sH + (i & 1) * ne + (i >> 1), m.h + 2 * (size_t)chk_idx(ids[nv + (i >> 1)], m.Ef, err) + (i & 1));
    for (int i = tid; i < nv; i += nt) {
      const size_t u = (size_t)chk_idx(ids[i], m.V, err);
      copy8(sx + i, m.ex + u);
      if (VISC) copy8(sxv + i, m.exv + u);
    }
    for (int i = tid; i < ne; i += nt) copy8(sxe + i, m.ee + (size_t)chk_idx(ids[nv + i], m.Ef, err));
  }
  copies_wait();
  ok = __syncthreads_and(ok);
  // the row's scale
  uint2 E = make_uint2(0x00010001u, 0x00010001u), Ev = E;
  if (ok) {
#pragma unroll 4
    for (int j = lane; j < 4 * mc; j += G) E = max_codes(E, sxe[eid[j]]);
    if (VISC) {
#pragma unroll 4
      for (int j = lane; j < 4 * nc; j += G) Ev = max_codes(Ev, sxv[vid[j]]);
    }
  }
  E = group_max_codes<G>(E);
  if (VISC) Ev = group_max_codes<G>(Ev);
  // rows whose fluxes are all finite are summed in fixed point
  const bool odd = any_raw(E) || (VISC && any_raw(Ev));
  const int base = RowShare<G>::first(lane);
  FxAcc A;
  unsigned lo[12];
  double R[RowShare<G>::kMax];
  A.clear();
  if (!ok && tid == 0) atomicOr(err, ERRBIT_TIMEOUT);
  if (live && !odd && ok) {
    in_spans<G, CARRY>(A, 4 * mc, 1, [&](int first, int end) {
      edge_entries<G>(A, first, end, lane, E, eid, m.ce + 96 * (size_t)(mb + m0), sH, ne, sxe);
    });
    in_spans<G, CARRY>(A, 4 * nc, 2, [&](int first, int end) {
      vertex_entries<G>(A, first, end, lane, E, vid, m.cv + 12 * (size_t)(cb + c0), sF, nv, sx);
    });
  }
  reduce_rows<G>(A, lo, lane);
  // a flux is b 2^(code - 1022 - (2L - 1)) and a coefficient a 2^(e - (2L - 1)); lo counts 2^L of a b
  constexpr int unit = L - 1022 - 2 * (2 * L - 1);
#pragma unroll
  for (int i = 0; i < RowShare<G>::kMax; ++i) {
    const int k = (base + i) >> 2, q = (base + i) & 3;
    R[i] = -fx_to_double(A.hh[i], lo[i], code_of(E, q) + coef_exp(ke.x, k) + unit, L);
  }
  if (VISC) {
    A.clear();
    if (live && !odd && ok)
      in_spans<G, CARRY>(A, 4 * nc, 2, [&](int first, int end) {
        vertex_entries<G>(A, first, end, lane, Ev, vid, m.cvis + 12 * (size_t)(cb + c0), sFv, nv, sxv);
      });
    reduce_rows<G>(A, lo, lane);
#pragma unroll
    for (int i = 0; i < RowShare<G>::kMax; ++i) {
      const int k = (base + i) >> 2, q = (base + i) & 3;
      R[i] += fx_to_double(A.hh[i], lo[i], code_of(Ev, q) + coef_exp(ke.y, k) + unit, L);
    }
  }
  if (!live) return;
#pragma unroll
  for (int i = 0; i < RowShare<G>::kMax; ++i)
    if (odd && i < RowShare<G>::count(lane)) R[i] = fallback_sum(m, r, (base + i) >> 2, (base + i) & 3, VISC);
  finish_rows<G>(r, lane, [&](int i) { return R[i]; }, m.V, sa, vmem, dtbits, cfl, dt_last, err);
}

// ------------------------------------------------------------------ coefficients to fixed point
// One thread per row: packs the row's FP64 coefficients (cv, ce, cvis: structure of arrays over the
// row's entries) into chunks.  Flags a row whose exponents leave 10 bits or one of whose vertices
// is on none of its edges (its exponent word would not cover that vertex).
__global__ void k_pack_fx(int A, int Ef, const int32_t* __restrict__ vp, const int32_t* __restrict__ vi,
                          const int32_t* __restrict__ ep, const int32_t* __restrict__ ei,
                          const double* __restrict__ cv, const double* __restrict__ ce,
                          const double* __restrict__ cvis, const int32_t* __restrict__ sten,
                          const int32_t* __restrict__ cvp, const int32_t* __restrict__ cep, int4* ocv, unsigned char* oce, int4* ocvis, int2* cexp,
                          int* flag) {
  constexpr int L = kFxBits;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= A) return;
  const int n0 = vp[r], N = vp[r + 1] - n0, m0 = ep[r], M = ep[r + 1] - m0;
  const double* c = cv + 6 * (size_t)n0;
  const double* d = ce + 3 * (size_t)m0;
  const double* z = cvis ? cvis + 6 * (size_t)n0 : nullptr;
  int e[3], ez[3] = {0, 0, 0};
  bool bad = false;
  for (int k = 0; k < 3; ++k) {
    int t = -10000, tz = -10000;
    double sum = 0.0, sumz = 0.0;
    for (int j = 0; j < N; ++j) {
      t = max(t, max(exp_above(c[(2 * k) * N + j]), exp_above(c[(2 * k + 1) * N + j])));
      if (z) tz = max(tz, max(exp_above(z[(2 * k) * N + j]), exp_above(z[(2 * k + 1) * N + j])));
      bad |= !isfinite(c[(2 * k) * N + j]) || !isfinite(c[(2 * k + 1) * N + j]);
      if (z) bad |= !isfinite(z[(2 * k) * N + j]) || !isfinite(z[(2 * k + 1) * N + j]);
      sum += fabs(c[(2 * k) * N + j]) + fabs(c[(2 * k + 1) * N + j]);
      if (z) sumz += fabs(z[(2 * k) * N + j]) + fabs(z[(2 * k + 1) * N + j]);
    }
    for (int j = 0; j < M; ++j) {
      t = max(t, exp_above(d[k * M + j]));
      bad |= !isfinite(d[k * M + j]);
      sum += fabs(d[k * M + j]);
    }
    e[k] = t == -10000 ? 0 : t;
    ez[k] = tz == -10000 ? 0 : tz;
    bad |= abs(e[k]) > 500 || abs(ez[k]) > 500;
    if (bad) break;
    while (sum > scalbn((double)kFxCoefSum, e[k])) ++e[k];
    while (sumz > scalbn((double)kFxCoefSum, ez[k])) ++ez[k];
    bad |= e[k] > 500 || ez[k] > 500;
  }
  if (bad) {
    *flag = 1;
    return;
  }
  auto pack = [](const int* x) { return (x[0] & 0x3ff) | ((x[1] & 0x3ff) << 10) | ((x[2] & 0x3ff) << 20); };
  cexp[r] = make_int2(pack(e), pack(ez));
  const int c0 = cvp[r], nc = cvp[r + 1] - c0;
  for (int j = 0; j < 4 * nc; ++j) {
    const bool pad = j >= N;
    for (int k = 0; k < 3; ++k) {
      const size_t o = 12 * ((size_t)c0 + (j >> 2)) + 4 * k + (j & 3);
      const int2 f = pad ? make_int2(0, 0) : coef_limbs(c[(2 * k) * N + j], e[k], L);
      const int2 g = pad ? make_int2(0, 0) : coef_limbs(c[(2 * k + 1) * N + j], e[k], L);
      ocv[o] = make_int4(f.x, f.y, g.x, g.y);
      if (z) {
        const int2 zf = pad ? make_int2(0, 0) : coef_limbs(z[(2 * k) * N + j], ez[k], L);
        const int2 zg = pad ? make_int2(0, 0) : coef_limbs(z[(2 * k + 1) * N + j], ez[k], L);
        ocvis[o] = make_int4(zf.x, zf.y, zg.x, zg.y);
      }
    }
    if (pad) continue;
    const int v = vi[n0 + j];
    bool found = false;
    for (int t = 0; t < M && !found; ++t) {
      const int s = ei[m0 + t];
      found = sten[2 * (size_t)Ef + s] == v || sten[3 * (size_t)Ef + s] == v;
    }
    if (!found) *flag = 1;
  }
  const int q0 = cep[r], mc = cep[r + 1] - q0;
  for (int j = 0; j < 4 * mc; ++j) {
    const bool pad = j >= M;
    int2 t[3];
    for (int k = 0; k < 3; ++k) t[k] = pad ? make_int2(0, 0) : coef_limbs(d[k * M + j], e[k], L);
    unsigned char* ck = oce + 96 * ((size_t)q0 + (j >> 2));
    reinterpret_cast<int4*>(ck)[j & 3] = make_int4(t[0].x, t[0].y, t[1].x, t[1].y);
    reinterpret_cast<int2*>(ck + 64)[j & 3] = t[2];
  }
}

cudaError_t pack_div_fx(const DevMesh& m, int* flag, cudaStream_t s) {
  if (m.A == 0) return cudaSuccess;
  const DivFx& f = m.fx;
  k_pack_fx<<<(m.A + 63) / 64, 64, 0, s>>>(
      m.A, m.Ef, m.vptr, m.vidx, m.eptr, m.eidx, (const double*)m.cv, (const double*)m.ce,
      m.viscous ? (const double*)m.cvis : nullptr, m.sten, f.vptr, f.eptr, f.cv, f.ce,
      f.cvis, f.cexp, flag);
  return cudaGetLastError();
}

// One thread per flux edge: the 30 weights of its sides (side * 15 + node * 3 + {value, x, y}) as limbs.
// Exponents: one per side for the values, and one offset for the derivatives of both sides.
__global__ void k_pack_w5(int Ef, const double* __restrict__ w5, int2* w5f, int2* w5e, int* flag) {
  constexpr int L = kFxBits;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= Ef) return;
  int ev[2] = {-10000, -10000}, off = -10000;
  bool bad = false;
  for (int s = 0; s < 2; ++s) {
    int ed = -10000;
    for (int j = 0; j < 15; ++j) {
      const double w = w5[(size_t)(15 * s + j) * Ef + e];
      bad |= !isfinite(w);
      if (j % 3 == 0) ev[s] = max(ev[s], exp_above(w));
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
    for (int j = 0; j < 15; ++j) {
      const size_t i = (size_t)(15 * s + j) * Ef + e;
      w5f[i] = coef_limbs(w5[i], ev[s] + (j % 3 ? off : 0), L);
    }
  w5e[e] = make_int2((ev[0] & 0xffff) | (int)((unsigned)ev[1] << 16), off);
}

cudaError_t pack_w5_fx(const DevMesh& m, int* flag, cudaStream_t s) {
  if (m.Ef == 0) return cudaSuccess;
  k_pack_w5<<<(m.Ef + 63) / 64, 64, 0, s>>>(m.Ef, (const double*)m.w5, m.fx.w5f, m.fx.w5e, flag);
  return cudaGetLastError();
}

template <int G, bool CARRY>
static const void* fx_kernel(bool visc) {
  return visc ? (const void*)&k_div_fx<G, CARRY, true> : (const void*)&k_div_fx<G, CARRY, false>;
}

static const void* fx_kernel(const DevMesh& m, int lanes) {
  const bool visc = m.viscous != 0;
  if (m.fx.carry) return lanes == 8 ? fx_kernel<8, true>(visc) : fx_kernel<4, true>(visc);
  return lanes == 8 ? fx_kernel<8, false>(visc) : fx_kernel<4, false>(visc);
}

cudaError_t prepare_div_fx(const DevMesh& m) {
  cudaError_t e = cudaSuccess;
  for (int lanes : {4, 8})
    if (e == cudaSuccess)                // one limit for every mesh
      e = cudaFuncSetAttribute(fx_kernel(m, lanes), cudaFuncAttributeMaxDynamicSharedMemorySize, kFxSmemMax);
  return e;
}

cudaError_t launch_div_fx(const DevMesh& m, const StageArgs& sa, const Phys& ph, int lanes, cudaStream_t s) {
  DivFx f = m.fx;
  f.A = m.A;
  f.V = m.V;
  f.Ef = m.Ef;
  f.nvptr = m.vptr;
  f.nvidx = m.vidx;
  f.neptr = m.eptr;
  f.neidx = m.eidx;
  f.FG = (const int4*)m.FG;
  f.FGv = (const int4*)m.FGv;
  f.h = (const int4*)m.h;
  const int G = lanes == 8 ? 8 : 4;
  StageArgs a = sa;
  const int32_t* vmem = m.vmem;
  const unsigned long long* dtbits = m.dtbits;
  double cfl = ph.cfl, *dt_last = m.dt_last;
  unsigned* err = m.err;
  void* args[] = {&f, &a, &vmem, &dtbits, &cfl, &dt_last, &err};
  return cudaLaunchKernel(fx_kernel(m, G), dim3((m.A + f.rows - 1) / f.rows), dim3(G * f.rows), args,
                          (size_t)f.smem, s);
}

}  // namespace hfd
