// The adjoint's dense parts on the tensor-core path, in double-float (adjoint.cu).
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace adjoint {

// FP64 matrices to double-float, element by element.
cudaError_t to_ff(const zc* in, float4* out, size_t n, cudaStream_t st);

// Gam[ws][(k1,a)][(k2,r)] = conj(grad_e)-weighted dE/dGh, k2 = k1 - Q, in FP64:
//   c2 sum_g X[w][-Q][g] LH[Q][k1][g][a][r]   (Coulomb; fp32 sum over g)
// + c1 AhH[k1][a][r] on the diagonal blocks  (one-body)
// - c3 gam32[k1][k2][ws][(a,r)]              (exchange, from the adjoint GEMM)
// with c = conj(grad_e) per walker.
cudaError_t gamma_smem(int G);   // shared-memory opt-in; fails for a G that no block can hold
cudaError_t gamma(const zc* LH, const zc* X, const zc* AhH, const zc* grad_e, const float2* gam32, zc* Gam,
                  const int* kminus, const int* minus, int nk, int G, int M, int n, int Mp, int W, cudaStream_t st);

// grad_phi[ws] = [S^-1 (Gam - (Gam phi S^-1) A^dag)]^H per walker-spin (Gh^T = phi S^-1).  Gam is
// overwritten; Y and P are [WS][N][N] scratch.
// launches: incremented by every kernel launch.
cudaError_t project(const zc* phi, zc* Gam, const float4* Sinv, const zc* A, float4* Y, float4* P,
                    zc* grad_phi, int WS, int nk, int M, int n, int& launches, cudaStream_t st);

// grad_h1[k][p][q] = sum_w g1[w] sum_s sum_a A[k][p][a] conj(Gh[w][s][(k,a)][(k,q)]), Gh^T = phi S^-1.
// ghd: [WS][nk][n][M] scratch, part: scratch of part_cap elements. 
cudaError_t grad_h1(const zc* phi, const float4* Sinv, const zc* A, const zc* grad_e, zc* ghd, zc* part,
                    size_t part_cap, zc* gh1, int W, int nk, int M, int n, int& launches, cudaStream_t st);

}  // namespace adjoint
