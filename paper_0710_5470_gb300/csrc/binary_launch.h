// Internal interface between the binary-fluid host code (binary2d.cu) and the
// D3Q19 kernels (binary3d.cu).  Not part of the C ABI.
#pragma once
#include <cuda_runtime.h>

#include "binary_common.cuh"

namespace lbb {

// One D3Q19 step from a.src into a.dst: the phi pass into `phi` (one value
// per site), then the fused step; both launches on `st`.
cudaError_t binary_step3(bool forcing, const StepArgs<float>& a, float* phi, cudaStream_t st, const int4* work, int ctas);
cudaError_t binary_step3(bool forcing, const StepArgs<double>& a, double* phi, cudaStream_t st);

// The marching float32 step (binary3d_march.cu) from a.phi: `ctas` entries (x0, y0,
// z0, z1) of column tiles of 32 x 8 sites and their z chunks.
cudaError_t binary_march3(bool forcing, const StepArgs<float>& a, const int4* work, int ctas, cudaStream_t st);
int binary_march3_ctas(bool forcing, int nx);   // resident CTAs per SM

// f = f^eq, g = g^eq of float64 fields rho [N], phi [N], u [3][N] (NULL: 0) into
// the population set `dst` (float32 if f32, else float64).
cudaError_t binary_init3(bool forcing, bool f32, const double* rho, const double* phi, const double* u, void* dst,
                         unsigned pitch, int nx, int ny, int nz, double A, double B, double kappa, double Gamma,
                         cudaStream_t st);

// Observables of the set `src` into the workspace w (15 N doubles): rho, phi,
// and where needed u [3], v [3], mu, and (forcing, for v) the six M' fields of
// the body force.
cudaError_t binary_fields3(bool forcing, bool f32, const void* src, unsigned pitch, int nx, int ny, int nz, double A,
                           double B, double kappa, double* w, bool need_u, bool need_v, bool need_mu,
                           cudaStream_t st);

}  // namespace lbb
