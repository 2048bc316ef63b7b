// The adjoint's dense parts on the tensor-core path: dE/dGh from its three pieces (the Coulomb sum in
// fp32, the exchange from the split GEMM's 22 bits), the projection through S^-1 and the walker, and
// dE/dh.  The projection and dE/dh are in double-float (ff.cuh, 48 bits): they multiply by S^-1, whose
// condition number would eat the 22 bits of the split GEMMs.
#include <algorithm>

#include "adjoint.hpp"
#include "attr.hpp"
#include "ff.cuh"

namespace adjoint {
namespace {

__device__ __forceinline__ float4 ff_of(zc v) { return ffa::cfrom(v); }
__device__ __forceinline__ float4 ff_of(float4 v) { return v; }
__device__ __forceinline__ void put(zc* o, float4 v) {
  *o = zmake(ffa::to_double(ffa::re(v)), ffa::to_double(ffa::im(v)));
}
__device__ __forceinline__ void put(float4* o, float4 v) { *o = v; }
__device__ __forceinline__ float4 conj_ff(float4 v) { return make_float4(v.x, v.y, -v.z, -v.w); }

__global__ void to_ff_kernel(const zc* in, float4* out, size_t n) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x)
    out[e] = ffa::cfrom(in[e]);
}

// C = op(A) op(B) per matrix of a batch (op 0: as stored, 2: conjugate transpose), operands FP64 or
// double-float, sums in double-float.
//
// Bound by the FP32 issue rate: 48 instructions per complex multiply-add, its TwoSum and TwoProduct
// errors collected beside the running sum, which is normalised after every k chunk of 32 so that the
// collected part stays small: its own roundings are the largest error of a long sum.  Tile 64 x 32,
// a thread holds rows ty + 16 i, columns tx + 16 j, so a tile's unused rows and columns are skipped in
// steps of 16 (N = 108: 7 % of the work is padding).
// Three products of 128 matrices, 108 x 702 x 108 twice and 108^3 once: 8.6 ms with 4 x 4
// outputs per thread and tiles of 64 x 64, 2.44 + 2.38 + 0.41 = 5.2 ms here (4.9 with Gam in double-float).  (Biased accumulators, 24
// instructions per multiply-add for an error of 2^-47 of a row maximum times a column sum per product,
// took 3.6 ms and made the gradient of E1 alone 25 to 60 times less exact on walkers near the trial.)
constexpr int BM = 64, BN = 32, BK = 32, TI = 4, TJ = 2;
constexpr int LDA = BM + 1, LDB = BN + 1;
constexpr size_t GEMM_SMEM = sizeof(float4) * BK * (LDA + LDB);

struct Dims {
  int m, n, k;
  long lda, ldb, ldc, sa, sb, sc;   // row strides and matrix strides, elements
};

template <int OPA, int OPB, class TA, class TB, class TC>
__global__ void __launch_bounds__(256, 2) gemm_ff_kernel(const TA* Ab, const TB* Bb, TC* Cb, Dims d) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float4* As = reinterpret_cast<float4*>(sm_raw);   // [BK][LDA]
  float4* Bs = As + BK * LDA;                         // [BK][LDB]
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  const int row0 = blockIdx.y * BM, col0 = blockIdx.x * BN;
  const TA* A = Ab + (size_t)blockIdx.z * d.sa;
  const TB* B = Bb + (size_t)blockIdx.z * d.sb;
  TC* C = Cb + (size_t)blockIdx.z * d.sc;
  const int ni = (min(BM, d.m - row0) + 15) >> 4, nj = (min(BN, d.n - col0) + 15) >> 4;   // used steps of 16
  ffa::cacc acc[TI][TJ];
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) acc[i][j] = ffa::cacc_from(ffa::czero());
  for (int p0 = 0; p0 < d.k; p0 += BK) {
    __syncthreads();
    for (int e = t; e < BM * BK; e += 256) {   // along the operand's contiguous index
      const int i = OPA == 0 ? e / BK : e % BM, p = OPA == 0 ? e % BK : e / BM;
      float4 v = ffa::czero();
      if (row0 + i < d.m && p0 + p < d.k) {
        v = ff_of(OPA == 0 ? A[(size_t)(row0 + i) * d.lda + p0 + p] : A[(size_t)(p0 + p) * d.lda + row0 + i]);
        if (OPA == 2) v = conj_ff(v);
      }
      As[p * LDA + i] = v;
    }
    for (int e = t; e < BN * BK; e += 256) {
      const int j = OPB == 0 ? e % BN : e / BK, p = OPB == 0 ? e / BN : e % BK;
      float4 v = ffa::czero();
      if (col0 + j < d.n && p0 + p < d.k) {
        v = ff_of(OPB == 0 ? B[(size_t)(p0 + p) * d.ldb + col0 + j] : B[(size_t)(col0 + j) * d.ldb + p0 + p]);
        if (OPB == 2) v = conj_ff(v);
      }
      Bs[p * LDB + j] = v;
    }
    __syncthreads();
#pragma unroll 1
    for (int p = 0; p < BK; ++p) {
      float4 b[TJ];
#pragma unroll
      for (int j = 0; j < TJ; ++j) b[j] = Bs[p * LDB + tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TI; ++i) {
        if (i >= ni) break;
        const float4 a = As[p * LDA + ty + 16 * i];
#pragma unroll
        for (int j = 0; j < TJ; ++j) {
          if (j >= nj) break;
          ffa::cacc_fma(acc[i][j], a, b[j]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
      for (int j = 0; j < TJ; ++j)
        acc[i][j] = ffa::cacc_from(ffa::cacc_get(acc[i][j]));
  }
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) {
      const int gi = row0 + ty + 16 * i, gj = col0 + tx + 16 * j;
      if (gi < d.m && gj < d.n) put(C + (size_t)gi * d.ldc + gj, ffa::cacc_get(acc[i][j]));
    }
}

template <int OPA, int OPB, class TA, class TB, class TC>
cudaError_t gemm(const TA* A, const TB* B, TC* C, const Dims& d, int batch, int& launches, cudaStream_t st) {
  auto fn = gemm_ff_kernel<OPA, OPB, TA, TB, TC>;
  cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(fn), GEMM_SMEM);
  if (e != cudaSuccess) return e;
  for (int b0 = 0; b0 < batch; b0 += 65535) {
    const dim3 grid((d.n + BN - 1) / BN, (d.m + BM - 1) / BM, std::min(batch - b0, 65535));
    fn<<<grid, 256, GEMM_SMEM, st>>>(A + (size_t)b0 * d.sa, B + (size_t)b0 * d.sb, C + (size_t)b0 * d.sc, d);
    ++launches;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// A block takes one (k1, Q) and GW walkers; a thread one (a, r) for all of them, so that each FP64
// vector element is converted once per GW walkers (the conversions run at the FP64 pipe's two per
// clock); consecutive walkers' X lie side by side in shared memory, two per load.  The weights are
// applied and the parts added in FP64, in which Gam is kept (610 us at 3x3x3, 64 walkers; 515 with
// double-float weights, which left up to four roundings of 2^-48 where FP64 leaves one).
template <int GW>
__global__ void __launch_bounds__(128) gamma_kernel(const zc* LH, const zc* X, const zc* AhH, const zc* grad_e,
                                                    const float2* gam32, zc* Gam, const int* kminus,
                                                    const int* minus, int nk, int G, int M, int n, int Mp, int W) {
  const int k1 = blockIdx.x, Q = blockIdx.y, w0 = blockIdx.z * GW;
  const int k2 = kminus[k1 * nk + Q], mQ = minus[Q];
  const int nw = min(GW, W - w0);
  const int nM = n * M, N = nk * n, NM = nk * M, WS = 2 * W, nMp = n * Mp;
  extern __shared__ __align__(16) float2 xs[];   // [G][GW]
  __shared__ zc cw[GW][3];                        // conj(grad_e)
  for (int e = threadIdx.x; e < GW * G; e += blockDim.x) {
    const int wi = e / G, g = e % G;
    const zc v = wi < nw ? X[((size_t)(w0 + wi) * nk + mQ) * G + g] : zzero();
    xs[g * GW + wi] = make_float2((float)v.x, (float)v.y);
  }
  for (int e = threadIdx.x; e < 3 * nw; e += blockDim.x) cw[e / 3][e % 3] = zconj(grad_e[3 * w0 + e]);
  __syncthreads();
  const zc* lh = LH + ((size_t)Q * nk + k1) * G * nM;
  for (int e = threadIdx.x; e < nM; e += blockDim.x) {
    float2 acc[GW];
#pragma unroll
    for (int i = 0; i < GW; ++i) acc[i] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int g = 0; g < G; ++g) {
      const zc l = lh[(size_t)g * nM + e];
      const float lr = (float)l.x, li = (float)l.y;
      const float4* x4 = reinterpret_cast<const float4*>(xs + g * GW);
#pragma unroll
      for (int i = 0; i < GW / 2; ++i) {
        const float4 x = x4[i];
        acc[2 * i].x = fmaf(x.x, lr, fmaf(-x.y, li, acc[2 * i].x));
        acc[2 * i].y = fmaf(x.x, li, fmaf(x.y, lr, acc[2 * i].y));
        acc[2 * i + 1].x = fmaf(x.z, lr, fmaf(-x.w, li, acc[2 * i + 1].x));
        acc[2 * i + 1].y = fmaf(x.z, li, fmaf(x.w, lr, acc[2 * i + 1].y));
      }
    }
    const int a = e / M, r = e % M;
    const zc ah = Q == 0 ? AhH[(size_t)k1 * nM + e] : zzero();
#pragma unroll
    for (int i = 0; i < GW; ++i) {
      if (i >= nw) break;
      const int w = w0 + i;
      zc base = zmul(cw[i][1], zmake(f2d(acc[i].x), f2d(acc[i].y)));
      if (Q == 0) base = zfma(cw[i][0], ah, base);
      for (int sp = 0; sp < 2; ++sp) {
        const int ws = 2 * w + sp;
        const float2 gx = gam32[(((size_t)k1 * nk + k2) * WS + ws) * nMp + a * Mp + r];
        Gam[((size_t)ws * N + k1 * n + a) * NM + k2 * M + r] =
            zsub(base, zmul(cw[i][2], zmake(f2d(gx.x), f2d(gx.y))));
      }
    }
  }
}

// Gam[ws][i][(k,r)] -= sum_a P[ws][i][(k,a)] conj(A[k][r][a]) ; grid (ws, row chunks of 16).  One pass
// over Gam, which the difference leaves in FP64; P's rows of the chunk and one k block of A at a time in shared memory.
constexpr int PROWS = 16;
__global__ void __launch_bounds__(256) gamma_project_kernel(zc* Gam, const float4* P, const zc* A, int nk, int M,
                                                            int n) {
  const int ws = blockIdx.x, i0 = blockIdx.y * PROWS, N = nk * n, NM = nk * M;
  const int rows = min(PROWS, N - i0);
  extern __shared__ __align__(16) float4 ps[];   // [rows][n] of one k block, then A[k] as [n][M]
  float4* as = ps + PROWS * n;
  for (int k = 0; k < nk; ++k) {
    __syncthreads();
    for (int e = threadIdx.x; e < rows * n; e += blockDim.x)
      ps[e] = P[((size_t)ws * N + i0 + e / n) * N + k * n + e % n];
    for (int e = threadIdx.x; e < M * n; e += blockDim.x)
      as[(e % n) * M + e / n] = conj_ff(ff_of(A[(size_t)k * M * n + e]));
    __syncthreads();
    for (int e = threadIdx.x; e < rows * M; e += blockDim.x) {
      const int i = e / M, r = e % M;
      zc* o = Gam + ((size_t)ws * N + i0 + i) * NM + k * M + r;
      ffa::cacc acc = ffa::cacc_from(ffa::czero());
      for (int a = 0; a < n; ++a) ffa::cacc_fma(acc, ps[i * n + a], as[a * M + r]);
      const float4 v = ffa::cacc_get(acc);
      *o = zsub(*o, zmake(ffa::to_double(ffa::re(v)), ffa::to_double(ffa::im(v))));
    }
  }
}

// The diagonal k blocks of the Green's function, ghd[ws][k][a][q] = sum_j S^-1[j][(k,a)] phi[(k,q)][j]:
// all that dE/dh reads (1 / Nk of Gh).  grid (ws, k), sums in double-float, normalised per chunk of j.
constexpr int GD_J = 32;
__global__ void __launch_bounds__(256) green_diag_kernel(const zc* phi, const float4* Sinv, zc* ghd, int nk, int M,
                                                         int n) {
  const int ws = blockIdx.x, k = blockIdx.y, N = nk * n, NM = nk * M;
  extern __shared__ __align__(16) float4 gd[];   // phi [M][GD_J + 1], S^-1 [GD_J][n]
  float4* sv = gd + M * (GD_J + 1);
  const zc* ph = phi + ((size_t)ws * NM + (size_t)k * M) * N;
  const float4* S = Sinv + (size_t)ws * N * N + k * n;
  for (int e0 = 0; e0 < n * M; e0 += blockDim.x) {
    const int e = e0 + threadIdx.x, a = e / M, q = e % M;
    ffa::cacc acc = ffa::cacc_from(ffa::czero());
    for (int j0 = 0; j0 < N; j0 += GD_J) {
      const int jn = min(GD_J, N - j0);
      __syncthreads();
      for (int u = threadIdx.x; u < M * GD_J; u += blockDim.x) {
        const int p = u / GD_J, j = u % GD_J;
        if (j < jn) gd[p * (GD_J + 1) + j] = ff_of(ph[(size_t)p * N + j0 + j]);
      }
      for (int u = threadIdx.x; u < jn * n; u += blockDim.x) sv[u] = S[(size_t)(j0 + u / n) * N + u % n];
      __syncthreads();
      if (e < n * M)
        for (int j = 0; j < jn; ++j) ffa::cacc_fma(acc, sv[j * n + a], gd[q * (GD_J + 1) + j]);
      acc = ffa::cacc_from(ffa::cacc_get(acc));
    }
    if (e < n * M) put(ghd + ((size_t)ws * nk + k) * n * M + e, ffa::cacc_get(acc));
  }
}

// part[c][k][p][q]: the walkers of chunk c; grid (k, chunks)
__global__ void grad_h1_part_kernel(const zc* A, const zc* ghd, const zc* grad_e, zc* part, int nk, int M, int n,
                                    int W) {
  const int k = blockIdx.x, per = (W + gridDim.y - 1) / gridDim.y;
  const int w0 = blockIdx.y * per, w1 = min(W, w0 + per);
  for (int e = threadIdx.x; e < M * M; e += blockDim.x) {
    const int p = e / M, q = e % M;
    zc s = zzero();
    for (int w = w0; w < w1; ++w) {
      zc t = zzero();
      for (int sp = 0; sp < 2; ++sp)
        for (int a = 0; a < n; ++a)
          t = zfma(A[((size_t)k * M + p) * n + a], zconj(ghd[(((size_t)(w * 2 + sp) * nk + k) * n + a) * M + q]), t);
      s = zfma(grad_e[3 * w + 0], t, s);
    }
    part[((size_t)blockIdx.y * nk + k) * M * M + e] = s;
  }
}
__global__ void grad_h1_sum_kernel(const zc* part, zc* gh1, int chunks, size_t per) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < per; e += (size_t)gridDim.x * blockDim.x) {
    zc s = zzero();
    for (int c = 0; c < chunks; ++c) s = zadd(s, part[(size_t)c * per + e]);
    gh1[e] = s;
  }
}

}  // namespace

cudaError_t to_ff(const zc* in, float4* out, size_t n, cudaStream_t st) {
  to_ff_kernel<<<(int)std::min<size_t>((n + 255) / 256, 4096), 256, 0, st>>>(in, out, n);
  return cudaGetLastError();
}

// 32 walkers per block where their X fits beside a second block, else 16
static bool gamma_wide(int G) { return sizeof(float2) * 32 * (size_t)G <= 100 * 1024; }

cudaError_t gamma_smem(int G) {
  return gamma_wide(G) ? ensure_dyn_smem(reinterpret_cast<const void*>(gamma_kernel<32>), sizeof(float2) * 32 * G)
                       : ensure_dyn_smem(reinterpret_cast<const void*>(gamma_kernel<16>), sizeof(float2) * 16 * G);
}

cudaError_t gamma(const zc* LH, const zc* X, const zc* AhH, const zc* grad_e, const float2* gam32, zc* Gam,
                  const int* kminus, const int* minus, int nk, int G, int M, int n, int Mp, int W, cudaStream_t st) {
  if (gamma_wide(G))
    gamma_kernel<32><<<dim3(nk, nk, (W + 31) / 32), 128, sizeof(float2) * 32 * G, st>>>(
        LH, X, AhH, grad_e, gam32, Gam, kminus, minus, nk, G, M, n, Mp, W);
  else
    gamma_kernel<16><<<dim3(nk, nk, (W + 15) / 16), 128, sizeof(float2) * 16 * G, st>>>(
        LH, X, AhH, grad_e, gam32, Gam, kminus, minus, nk, G, M, n, Mp, W);
  return cudaGetLastError();
}

cudaError_t project(const zc* phi, zc* Gam, const float4* Sinv, const zc* A, float4* Y, float4* P,
                    zc* grad_phi, int WS, int nk, int M, int n, int& launches, cudaStream_t st) {
  const int N = nk * n, NM = nk * M;
  const long NN = (long)N * N, NNM = (long)N * NM;
  cudaError_t e;
  // Y = Gam phi, P = Y S^-1
  if ((e = gemm<0, 0>(Gam, phi, Y, Dims{N, N, NM, NM, N, N, NNM, NNM, NN}, WS, launches, st)) != cudaSuccess) return e;
  if ((e = gemm<0, 0>(Y, Sinv, P, Dims{N, N, N, N, N, N, NN, NN, NN}, WS, launches, st)) != cudaSuccess) return e;
  const size_t smem = sizeof(float4) * ((size_t)PROWS * n + (size_t)M * n);
  if ((e = ensure_dyn_smem(reinterpret_cast<const void*>(gamma_project_kernel), smem)) != cudaSuccess) return e;
  gamma_project_kernel<<<dim3(WS, (N + PROWS - 1) / PROWS), 256, smem, st>>>(Gam, P, A, nk, M, n);
  ++launches;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // grad_phi = Gam^H S^-H
  return gemm<2, 2>(Gam, Sinv, grad_phi, Dims{NM, N, N, NM, N, N, NNM, NN, NNM}, WS, launches, st);
}

cudaError_t grad_h1(const zc* phi, const float4* Sinv, const zc* A, const zc* grad_e, zc* ghd, zc* part,
                    size_t part_cap, zc* gh1, int W, int nk, int M, int n, int& launches, cudaStream_t st) {
  const size_t smem = sizeof(float4) * ((size_t)M * (GD_J + 1) + (size_t)GD_J * n);
  cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(green_diag_kernel), smem);
  if (e != cudaSuccess) return e;
  green_diag_kernel<<<dim3(2 * W, nk), std::min(256, (n * M + 31) / 32 * 32), smem, st>>>(phi, Sinv, ghd, nk, M, n);
  ++launches;
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const size_t per = (size_t)nk * M * M;
  const int chunks = (int)std::max<size_t>(1, std::min<size_t>({(size_t)16, (size_t)W, part_cap / per}));
  zc* dst = chunks == 1 ? gh1 : part;
  grad_h1_part_kernel<<<dim3(nk, chunks), 256, 0, st>>>(A, ghd, grad_e, dst, nk, M, n, W);
  ++launches;
  if ((e = cudaGetLastError()) != cudaSuccess || chunks == 1) return e;
  grad_h1_sum_kernel<<<(int)std::min<size_t>((per + 255) / 256, 4096), 256, 0, st>>>(part, gh1, chunks, per);
  ++launches;
  return cudaGetLastError();
}

}  // namespace adjoint
