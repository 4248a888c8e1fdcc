// Flux records of the fixed-point 3D divergence (k3_div_fx), written by k3_vertex and the edge kernels.
#pragma once
#include "fixed_point.cuh"

namespace hfd {

// A 5-vector's record in fixed point: its pairs and the codes of mass, momentum (one for the three: each row
// reads fluxes in all directions, so every momentum sum has pressure-sized terms) and energy.
constexpr int kBits3 = kFxBits;
__device__ __forceinline__ void st_record3(int4* rec, size_t i, const double* f) {
  const int E0 = fx_code(f[0]), E1 = max(fx_code(f[1]), max(fx_code(f[2]), fx_code(f[3]))), E2 = fx_code(f[4]);
  const int2 p0 = fx_encode(f[0], E0, kBits3), p1 = fx_encode(f[1], E1, kBits3), p2 = fx_encode(f[2], E1, kBits3);
  const int2 p3 = fx_encode(f[3], E1, kBits3), p4 = fx_encode(f[4], E2, kBits3);
  int4* o = rec + 3 * i;
  o[0] = make_int4(p0.x, p0.y, p1.x, p1.y);
  o[1] = make_int4(p2.x, p2.y, p3.x, p3.y);
  o[2] = make_int4(p4.x, p4.y, (int)((unsigned)E0 | ((unsigned)E1 << 16)), E2);
}

}  // namespace hfd
