// Launchers of the 3D extension's kernels (kernels3d.cu).
#pragma once
#include <cuda_runtime.h>

#include "mesh3.hpp"

namespace hfd {

// Vertex-major copy of U (20 x V) into m.Ua and the flux vectors F, G, K into m.FGK.
cudaError_t launch3_vertex(const DevMesh3& m, const double* U, const Phys3& ph, cudaStream_t s);
// Edge fluxes h from m.Ua (Alg. 1 in 3D and Roe's flux).
cudaError_t launch3_edge(const DevMesh3& m, const Phys3& ph, cudaStream_t s);
// Divergence gather: mode 0 writes R = -div into out; mode 1 writes b (Us + dt R) + a Un.
cudaError_t launch3_div(const DevMesh3& m, const double* Us, const double* Un, double* out,
                        int mode, double a, double b, double dt, cudaStream_t s);

// Packs m.cv and m.ce into m.fx; *flag (device) is set if a coefficient does not fit.
cudaError_t launch3_pack(const DevMesh3& m, int* flag, cudaStream_t s);
// Packs m.w5 into m.ex (and the frame in FP32); *flag (device) is set if a weight does not fit.
cudaError_t launch3_pack_w5(const DevMesh3& m, int* flag, cudaStream_t s);
// The edges' fixed-point arrays, without nodes and weights (the sums in FP64) where these do not fit.
inline Edge3Fx edge3_fx(const DevMesh3& m) {
  Edge3Fx x = m.ex;
  if (!m.ex_ok) x.uf = nullptr;
  return x;
}
// The lanes of the next launches: 0 the fixed-point divergence, which 4 lanes (the default) stand for where the
// rows have that form, else the FP64 one.
inline int div3_lanes(const DevMesh3& m) { return m.lanes == 4 && m.fx_ok ? 0 : m.lanes; }

}  // namespace hfd
