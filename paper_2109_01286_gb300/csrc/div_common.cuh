// Pieces shared by the 2D kernels (kernels.cu) and the fixed-point divergence (div_fixed.cu).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.hpp"

namespace hfd {

enum : unsigned { ERRBIT_NONFINITE = 1u, ERRBIT_POSITIVITY = 2u, ERRBIT_TIMEOUT = 4u, ERRBIT_INDEX = 8u };

// Bounds-checked build (compiled with -DHFD_CHECK=1, the stand-in for a memory checker): every
// gathered index is tested against its array's extent; one outside [0, n) records ERRBIT_INDEX
// in the mesh's error word and is replaced by 0, so that the access stays in bounds (the result
// is then wrong, and hfd_check reports it).  In the normal build this is the identity.
#ifndef HFD_CHECK
#define HFD_CHECK 0
#endif
__device__ __forceinline__ int chk_idx(int i, int n, unsigned* err) {
#if HFD_CHECK
  if ((unsigned)i >= (unsigned)n) {
    atomicOr(err, ERRBIT_INDEX);
    return 0;
  }
#endif
  return i;
}

// Finite (not inf or NaN) by the exponent field, on the integer pipe (GB300's FP64 pipe is
// the limit of the FP64 divergence).
__device__ __forceinline__ bool finite_bits(double x) {
  return ((unsigned)(__double_as_longlong(x) >> 52) & 0x7ffu) != 0x7ffu;
}

// G lanes per active vertex (G in {1, 2, 4, 8}); lanes stride over the CSR entries; the 12 partial
// sums are combined by a fixed reduce-scatter over the group (each level halves the values a
// lane holds), so the result is deterministic and every add is useful.  acc = div(f) -
// div(f_vis) for the 12 rows; R = -acc.
template <int G, typename T>
__device__ __forceinline__ void reduce_scatter12(T* acc, int lane) {
  // after the loop lane `lane` holds rows base .. base + 12/G - 1 in acc[0 .. 12/G - 1]
  if (G >= 2) {
    const int o = G / 2;
    bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      T keep = hi ? acc[6 + i] : acc[i];
      T send = hi ? acc[i] : acc[6 + i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o, G);
    }
  }
  if (G >= 4) {
    const int o = G / 4;
    bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      T keep = hi ? acc[3 + i] : acc[i];
      T send = hi ? acc[i] : acc[3 + i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o, G);
    }
  }
  if (G >= 8) {
    // three values left: the lane with bit 0 clear keeps rows 0-1, its partner keeps row 2
    bool hi = (lane & 1) != 0;
    T r0 = __shfl_xor_sync(0xffffffffu, acc[0], 1, G);
    T r1 = __shfl_xor_sync(0xffffffffu, acc[1], 1, G);
    T r2 = __shfl_xor_sync(0xffffffffu, acc[2], 1, G);
    if (hi) {
      acc[0] = acc[2] + r2;
    } else {
      acc[0] += r0;
      acc[1] += r1;
    }
  }
}

// The rows of its vertex that a lane of G holds after reduce_scatter12, first() .. first() +
// count() - 1, in its first registers.
template <int G>
struct RowShare {
  static constexpr int kMax = G >= 8 ? 2 : 12 / G;
  static __device__ __forceinline__ int first(int lane) {
    return (G >= 2 && (lane & (G / 2)) ? 6 : 0) + (G >= 4 && (lane & (G / 4)) ? 3 : 0) +
           (G >= 8 && (lane & 1) ? 2 : 0);
  }
  static __device__ __forceinline__ int count(int lane) { return G >= 8 && (lane & 1) ? 1 : kMax; }
};

// Writes R, or the Runge-Kutta stage combination a*Un + b*(Us + dt*R), for the rows of vertex r that
// this lane of G holds, value(i) being R of its i-th; flags non-finite values and non-positive
// densities in the error word.
template <int G, typename F>
__device__ __forceinline__ void finish_rows(int r, int lane, F value, int V, const StageArgs& sa,
                                            const int32_t* __restrict__ vmem,
                                            const unsigned long long* dtbits, double cfl,
                                            double* dt_last, unsigned* err) {
  const double* __restrict__ Us = sa.Us;
  const double* __restrict__ Un = sa.Un;
  double* out = sa.out;
  const int mode = sa.mode;
  const double a = sa.a, b = sa.b, dt_fixed = sa.dt_fixed;
  // time step of this vertex's mesh (a batch holds several meshes, each with its own CFL step)
  const int mem = vmem ? __ldg(vmem + r) : 0;
  double dt = dt_fixed > 0.0 ? dt_fixed
               : sa.dt_member ? __ldg(sa.dt_member + mem)
                              : cfl * __longlong_as_double((long long)dtbits[mem]);
  if (mode == DIV_STAGE && lane == 0 && dt_last && (r == 0 || (vmem && __ldg(vmem + r - 1) != mem)))
    dt_last[mem] = dt;
  // rows held by this lane after the reduce-scatter: base .. base + per - 1
  int per = G == 1 ? 12 : G == 2 ? 6 : 3;
  int base = (G >= 2 && (lane & (G / 2)) ? 6 : 0) + (G >= 4 && (lane & (G / 4)) ? 3 : 0);
  if (G >= 8) {
    if (lane & 1) { base += 2; per = 1; } else { per = 2; }
  }
  unsigned bad = 0;
#pragma unroll
  for (int i = 0; i < 12 / (G >= 8 ? 4 : G); ++i) {
    if (i >= per) break;
    int k = base + i;
    double R = value(i);
    size_t idx = (size_t)k * V + r;
    double o;
    if (mode == DIV_RESIDUAL) {
      o = R;
    } else {
      // explicit roundings, so that every kernel holding this code (four-launch, fixed-point,
      // persistent) gives the same bits: one FMA, one multiply, one FMA
      o = __dmul_rn(b, __fma_rn(dt, R, Us[idx]));
      if (a != 0.0) o = __fma_rn(a, Un[idx], o);   // the first stage does not read the base state
    }
    out[idx] = o;
    if (!finite_bits(o)) bad |= ERRBIT_NONFINITE;
    if (mode == DIV_STAGE && k == 0 && !(o > 0.0)) bad |= ERRBIT_POSITIVITY;
  }
  if (bad) atomicOr(err, bad);
}

}  // namespace hfd
