// FP64 path of the k-point AFQMC walker step: every contraction in complex128
// on the FP64 pipes.  It is the precision reference on the GPU and the
// baseline the tensor-core path is measured against.
//
// Paper map (arXiv:2003.09468):
//   overlap / Green's function    Sec. 2.2 Eqs. gf, gfhrot
//   Cholesky trace X, force bias  Sec. 2.2 Eq. fb; Sec. 2.3 Eq. kp_vbias
//   vHS                           Sec. 2.2 Eq. vhs; Sec. 2.3 Eq. kp_vhs
//   Taylor exp(V), one-body half  Sec. 2.1 Eq. propagator; Sec. 2.2 (Taylor series)
//   hybrid weight                 Sec. 2.1 (importance function, phase, hybrid form)
//   local energy                  Sec. 2.2 Eq. local_energy; Sec. 2.3 Eq. kp_el;
//                                 Sec. 3.2 energy steps 1-3
#include <math.h>

#include <algorithm>
#include <utility>

#include "attr.hpp"
#include "handle.hpp"

namespace fp64 {

// ---------------------------------------------------------------------------
// Generic strided-batched complex GEMM:  C = alpha op(A) op(B) + beta C
// (optionally also Acc += alpha op(A) op(B)).  op: 0 = N, 1 = T, 2 = C.
// Three batch dimensions with independent strides.
// ---------------------------------------------------------------------------
struct ZGemm {
  int m, n, k;
  int opA, opB;
  const zc* A; long lda; long sA[3];
  const zc* B; long ldb; long sB[3];
  zc* C; long ldc; long sC[3];
  zc* Acc; long ldacc; long sAcc[3];
  int nb[3];
  zc alpha, beta;
};

constexpr int GBM = 32, GBN = 32, GBK = 8;

__global__ void __launch_bounds__(256) zgemm_kernel(ZGemm g) {
  __shared__ zc As[GBK][GBM + 1];
  __shared__ zc Bs[GBK][GBN + 1];
  const int t = threadIdx.x;
  const int ty = t >> 4, tx = t & 15;
  const int row0 = blockIdx.y * GBM, col0 = blockIdx.x * GBN;
  const long nbatch = (long)g.nb[0] * g.nb[1] * g.nb[2];
  for (long z = blockIdx.z; z < nbatch; z += gridDim.z) {
    const int b2 = (int)(z % g.nb[2]);
    const int b1 = (int)((z / g.nb[2]) % g.nb[1]);
    const int b0 = (int)(z / ((long)g.nb[2] * g.nb[1]));
    const zc* A = g.A + b0 * g.sA[0] + b1 * g.sA[1] + b2 * g.sA[2];
    const zc* B = g.B + b0 * g.sB[0] + b1 * g.sB[1] + b2 * g.sB[2];
    zc* C = g.C + b0 * g.sC[0] + b1 * g.sC[1] + b2 * g.sC[2];
    zc acc[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] = zzero();
    for (int p0 = 0; p0 < g.k; p0 += GBK) {
      {  // A tile: op(A)[row0 + i][p0 + p]
        int i, p;
        if (g.opA == 0) { i = t >> 3; p = t & 7; } else { p = t >> 5; i = t & 31; }
        const int gi = row0 + i, gp = p0 + p;
        zc v = zzero();
        if (gi < g.m && gp < g.k) {
          if (g.opA == 0) v = A[(long)gi * g.lda + gp];
          else { v = A[(long)gp * g.lda + gi]; if (g.opA == 2) v = zconj(v); }
        }
        As[p][i] = v;
      }
      {  // B tile: op(B)[p0 + p][col0 + j]
        int j, p;
        if (g.opB == 0) { p = t >> 5; j = t & 31; } else { j = t >> 3; p = t & 7; }
        const int gj = col0 + j, gp = p0 + p;
        zc v = zzero();
        if (gj < g.n && gp < g.k) {
          if (g.opB == 0) v = B[(long)gp * g.ldb + gj];
          else { v = B[(long)gj * g.ldb + gp]; if (g.opB == 2) v = zconj(v); }
        }
        Bs[p][j] = v;
      }
      __syncthreads();
#pragma unroll
      for (int p = 0; p < GBK; ++p) {
        zc a0 = As[p][ty * 2], a1 = As[p][ty * 2 + 1];
        zc c0 = Bs[p][tx * 2], c1 = Bs[p][tx * 2 + 1];
        acc[0][0] = zfma(a0, c0, acc[0][0]);
        acc[0][1] = zfma(a0, c1, acc[0][1]);
        acc[1][0] = zfma(a1, c0, acc[1][0]);
        acc[1][1] = zfma(a1, c1, acc[1][1]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int gi = row0 + ty * 2 + i, gj = col0 + tx * 2 + j;
        if (gi < g.m && gj < g.n) {
          zc r = zmul(g.alpha, acc[i][j]);
          zc* c = C + (long)gi * g.ldc + gj;
          if (g.beta.x != 0.0 || g.beta.y != 0.0) r = zfma(g.beta, *c, r);
          *c = r;
          if (g.Acc) {
            zc* a = g.Acc + b0 * g.sAcc[0] + b1 * g.sAcc[1] + b2 * g.sAcc[2] + (long)gi * g.ldacc + gj;
            *a = zadd(*a, zmul(g.alpha, acc[i][j]));
          }
        }
      }
  }
}

static ZGemm gemm_init(int m, int n, int k, int opA, int opB) {
  ZGemm g;
  memset(&g, 0, sizeof(g));
  g.m = m; g.n = n; g.k = k; g.opA = opA; g.opB = opB;
  g.nb[0] = g.nb[1] = g.nb[2] = 1;
  g.alpha = zmake(1.0, 0.0);
  g.beta = zzero();
  return g;
}

static cudaError_t gemm_launch(afqmc_kp* h, const ZGemm& g, cudaStream_t st) {
  long nb = (long)g.nb[0] * g.nb[1] * g.nb[2];
  dim3 grid((g.n + GBN - 1) / GBN, (g.m + GBM - 1) / GBM, (unsigned)(nb < 65535 ? nb : 65535));
  zgemm_kernel<<<grid, 256, 0, st>>>(g);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Set-up kernels
// ---------------------------------------------------------------------------

// v0[k][p][q] = -1/2 sum_{Q,g,r} L[Q][k][g][p][r] conj(L[Q][k][g][q][r])
// v0[k] = -1/2 sum_{Q,g} L[Q,k,g] L[Q,k,g]^dagger in two passes: one block per (k, Q) sums
// its g's into part[k][Q] (the block reads its own slab of L once; the M x M products run
// from L1), then the Q partials are added in a fixed order.
__global__ void v0_partial_kernel(const zc* L, zc* part, int nk, int G, int M) {
  const int k = blockIdx.x, Q = blockIdx.y;
  const int MM = M * M;
  const zc* slab = L + ((size_t)Q * nk + k) * G * MM;
  zc* out = part + ((size_t)k * nk + Q) * MM;
  for (int o = threadIdx.x; o < MM; o += blockDim.x) {
    const int p = o / M, q = o % M;
    zc s = zzero();
    for (int g = 0; g < G; ++g) {
      const zc* blk = slab + (size_t)g * MM;
      for (int r = 0; r < M; ++r) s = zfma(blk[p * M + r], zconj(blk[q * M + r]), s);
    }
    out[o] = s;
  }
}
__global__ void v0_reduce_kernel(const zc* part, zc* v0, int nk, int M) {
  const int k = blockIdx.x, MM = M * M;
  for (int o = threadIdx.x; o < MM; o += blockDim.x) {
    zc s = zzero();
    for (int Q = 0; Q < nk; ++Q) s = zadd(s, part[((size_t)k * nk + Q) * MM + o]);
    v0[(size_t)k * MM + o] = zscale(s, -0.5);
  }
}

// Ehalf[k] = exp(-dt/2 (h[k] + v0[k])) by scaling, 24-term Taylor series and squaring.
// Three launches: X = -dt/2 (h + v0) scaled by 2^-sq to a norm of at most 1/4, the Taylor series by
// groups of rows (row i of X^j / j! needs only itself and X, so the rows spread over the GPU: one
// block per k ran 24 dependent M^3 products at one SM's FP64 rate, 517 us at M = 26, 27 k-points),
// and sq squarings (none at the time steps in use).  tmp: [k][3][M][M] = X, (sq in its first element), scratch.
__global__ void expm_scale_kernel(const zc* h1, const zc* v0, zc* tmp, int M, double dt) {
  const int k = blockIdx.x;
  const long MM = (long)M * M;
  zc* Xm = tmp + (long)k * 3 * MM;
  __shared__ double red[32];
  __shared__ int s_sq;
  double rowmax = 0.0;
  for (int i = threadIdx.x; i < M; i += blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < M; ++j) {
      zc v = zscale(zadd(h1[k * MM + i * M + j], v0[k * MM + i * M + j]), -0.5 * dt);
      s += sqrt(zabs2(v));
    }
    rowmax = fmax(rowmax, s);
  }
  double v = rowmax;
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int i = 0; i < (int)((blockDim.x + 31) >> 5); ++i) m = fmax(m, red[i]);
    int sq = 0;
    while (m > 0.25 && sq < 60) { m *= 0.5; ++sq; }
    s_sq = sq;
    tmp[((long)k * 3 + 1) * MM] = zmake((double)sq, 0.0);
  }
  __syncthreads();
  const double scl = ldexp(1.0, -s_sq);
  for (long e = threadIdx.x; e < MM; e += blockDim.x)
    Xm[e] = zscale(zscale(zadd(h1[k * MM + e], v0[k * MM + e]), -0.5 * dt), scl);
}
constexpr int EXPM_ROWS = 4;
// out rows of sum_{j<=24} X^j / j! ; grid (k, groups of EXPM_ROWS rows), dynamic shared memory
// 2 EXPM_ROWS M elements
__global__ void expm_rows_kernel(const zc* tmp, zc* out, int M) {
  const int k = blockIdx.x, i0 = blockIdx.y * EXPM_ROWS, rows = min(EXPM_ROWS, M - i0);
  const long MM = (long)M * M;
  const zc* Xm = tmp + (long)k * 3 * MM;
  zc* E = out + k * MM + (long)i0 * M;
  extern __shared__ zc er[];   // [EXPM_ROWS][M] the term's rows, [EXPM_ROWS][M] the next term's
  zc* Tm = er;
  zc* Rm = er + EXPM_ROWS * M;
  for (int e = threadIdx.x; e < rows * M; e += blockDim.x) {
    Tm[e] = zmake(i0 + e / M == e % M ? 1.0 : 0.0, 0.0);
    E[e] = Tm[e];
  }
  __syncthreads();
  for (int term = 1; term <= 24; ++term) {
    for (int e = threadIdx.x; e < rows * M; e += blockDim.x) {
      const int i = e / M, j = e % M;
      zc s = zzero();
      for (int l = 0; l < M; ++l) s = zfma(Tm[i * M + l], Xm[(long)l * M + j], s);
      Rm[e] = zscale(s, 1.0 / term);
      E[e] = zadd(E[e], Rm[e]);
    }
    __syncthreads();
    zc* t = Tm;
    Tm = Rm;
    Rm = t;
  }
}
__global__ void expm_square_kernel(zc* out, zc* tmp, int M) {
  const int k = blockIdx.x;
  const long MM = (long)M * M;
  zc* E = out + k * MM;
  zc* Rm = tmp + ((long)k * 3 + 2) * MM;
  const int sq = (int)tmp[((long)k * 3 + 1) * MM].x;
  for (int s = 0; s < sq; ++s) {
    for (long e = threadIdx.x; e < MM; e += blockDim.x) {
      const int i = (int)(e / M), j = (int)(e % M);
      zc acc = zzero();
      for (int l = 0; l < M; ++l) acc = zfma(E[i * M + l], E[l * M + j], acc);
      Rm[e] = acc;
    }
    __syncthreads();
    for (long e = threadIdx.x; e < MM; e += blockDim.x) E[e] = Rm[e];
    __syncthreads();
  }
}

static cudaError_t configure_smem(afqmc_kp* h);

cudaError_t setup_static(afqmc_kp* h, cudaStream_t st) {
  const int nk = h->nk, M = h->M, n = h->n, G = h->G;
  {
    cudaError_t e = configure_smem(h);
    if (e != cudaSuccess) return e;
  }
  // LH[Q][k][g] = A[k]^dagger L[Q][k][g]
  {
    ZGemm g = gemm_init(n, M, M, 2, 0);
    g.A = h->A; g.lda = n; g.sA[0] = 0; g.sA[1] = (long)M * n; g.sA[2] = 0;
    g.B = h->L; g.ldb = M; g.sB[0] = (long)nk * G * M * M; g.sB[1] = (long)G * M * M; g.sB[2] = (long)M * M;
    g.C = h->LH; g.ldc = M; g.sC[0] = (long)nk * G * n * M; g.sC[1] = (long)G * n * M; g.sC[2] = (long)n * M;
    g.nb[0] = nk; g.nb[1] = nk; g.nb[2] = G;
    cudaError_t e = gemm_launch(h, g, st);
    if (e != cudaSuccess) return e;
  }
  {
    // the Q partials of v0 live in a temporary buffer (create time: allocation is allowed)
    zc* part = nullptr;
    cudaError_t e = cudaMalloc(&part, sizeof(zc) * (size_t)nk * nk * M * M);
    if (e != cudaSuccess) return e;
    v0_partial_kernel<<<dim3(nk, nk), 256, 0, st>>>(h->L, part, nk, G, M);
    AFQMC_LAUNCHED(h);
    v0_reduce_kernel<<<nk, 256, 0, st>>>(part, h->v0, nk, M);
    AFQMC_LAUNCHED(h);
    e = cudaGetLastError();
    const cudaError_t e2 = cudaStreamSynchronize(st);
    cudaFree(part);
    if (e != cudaSuccess) return e;
    if (e2 != cudaSuccess) return e2;
  }
  return set_one_body(h, st);
}

cudaError_t set_one_body(afqmc_kp* h, cudaStream_t st) {
  const int nk = h->nk, M = h->M, n = h->n;
  ZGemm g = gemm_init(n, M, M, 2, 0);  // AhH[k] = A[k]^dagger h[k]
  g.A = h->A; g.lda = n; g.sA[0] = (long)M * n;
  g.B = h->h1; g.ldb = M; g.sB[0] = (long)M * M;
  g.C = h->AhH; g.ldc = M; g.sC[0] = (long)n * M;
  g.nb[0] = nk;
  cudaError_t e = gemm_launch(h, g, st);
  if (e != cudaSuccess) return e;
  expm_scale_kernel<<<nk, 256, 0, st>>>(h->h1, h->v0, h->expm_tmp, M, h->dt);
  AFQMC_LAUNCHED(h);
  expm_rows_kernel<<<dim3(nk, (M + EXPM_ROWS - 1) / EXPM_ROWS), 128, sizeof(zc) * 2 * EXPM_ROWS * M, st>>>(
      h->expm_tmp, h->Ehalf, M);
  AFQMC_LAUNCHED(h);
  expm_square_kernel<<<nk, 256, 0, st>>>(h->Ehalf, h->expm_tmp, M);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Overlap, LU with partial pivoting, log det and inverse (one block per matrix)
// ---------------------------------------------------------------------------

// S[ws][(k,a)][j] = sum_p conj(A[k][p][a]) phi[ws][(k,p)][j]
// Block (ws, k); threads over j, eight rows a at a time held in registers.
constexpr int OVA = 8;
__global__ void __launch_bounds__(256) overlap_kernel(const zc* A, const zc* phi, zc* S, int nk, int M, int n,
                                                      int N) {
  const int ws = blockIdx.x, k = blockIdx.y;
  const zc* Ak = A + (size_t)k * M * n;
  const zc* ph = phi + ((size_t)ws * nk * M + (size_t)k * M) * N;
  zc* Sk = S + ((size_t)ws * N + (size_t)k * n) * N;
  for (int a0 = 0; a0 < n; a0 += OVA) {
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      zc acc[OVA];
#pragma unroll
      for (int i = 0; i < OVA; ++i) acc[i] = zzero();
      for (int p = 0; p < M; ++p) {
        const zc v = ph[(size_t)p * N + j];
#pragma unroll
        for (int i = 0; i < OVA; ++i)
          if (a0 + i < n) acc[i] = zfma(zconj(Ak[p * n + a0 + i]), v, acc[i]);
      }
#pragma unroll
      for (int i = 0; i < OVA; ++i)
        if (a0 + i < n) Sk[(size_t)(a0 + i) * N + j] = acc[i];
    }
  }
}

static cudaError_t overlap(afqmc_kp* h, const zc* phi, cudaStream_t st) {
  overlap_kernel<<<dim3(2 * h->W, h->nk), 256, 0, st>>>(h->A, phi, h->S, h->nk, h->M, h->n, h->N);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// In-place LU of S (row pivoting), log det, optional inverse.  sing[b] = 1 if a
// pivot is zero or not finite; then Sinv = 0 and logdet = (-inf, 0).
// A chain of short steps: SA keeps the matrix in shared memory while it is factored, SX the
// inverse too (from global memory every step waited for L2); the pivot search is a warp maximum and
// one pass over the warps; the logarithms of the pivots and the reciprocals of U's diagonal, which
// one thread formed column by column while the others waited, are formed for all columns at once.
// N = 16, 32 matrices: 146 us before.
template <bool SA, bool SX>
__global__ void __launch_bounds__(256) lu_kernel(zc* S, zc* Sinv, zc* logdet, int* sing, int* flags,
                                                 int N, int want_inv, int* perm_ws) {
  const int b = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  extern __shared__ __align__(16) unsigned char lu_smem[];
  zc* g = S + (long)b * N * N;
  zc* a = SA ? reinterpret_cast<zc*>(lu_smem) : g;
  int* perm = perm_ws + (long)b * N;
  __shared__ unsigned long long s_val[8];
  __shared__ int s_idx[8];
  __shared__ zc s_red[8];
  int swaps = 0;   // the same in every thread
  bool singular = false;
  if (SA)
    for (long e = threadIdx.x; e < (long)N * N; e += blockDim.x) a[e] = g[e];
  for (int i = threadIdx.x; i < N; i += blockDim.x) perm[i] = i;
  __syncthreads();
  for (int j = 0; j < N; ++j) {
    // largest |a_ij|^2, the smallest row among equals, compared by bits (ordered as the values,
    // NaN left out): 64-bit compares would go through the FP64 pipe
    unsigned long long best = 0;
    int bi = N;
    for (int i = j + threadIdx.x; i < N; i += blockDim.x) {
      const unsigned long long v = (unsigned long long)__double_as_longlong(zabs2(a[(long)i * N + j]));
      if (v <= 0x7ff0000000000000ull && (v > best || bi == N)) { best = v; bi = i; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long v2 = __shfl_xor_sync(0xffffffffu, best, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
      if (v2 > best || (v2 == best && i2 < bi)) { best = v2; bi = i2; }
    }
    if (lane == 0) { s_val[wid] = best; s_idx[wid] = bi; }
    __syncthreads();
    unsigned long long pv = s_val[0];
    int p = s_idx[0];
    for (int w = 1; w < nw; ++w) {
      const unsigned long long v2 = s_val[w];
      const int i2 = s_idx[w];
      if (v2 > pv || (v2 == pv && i2 < p)) { pv = v2; p = i2; }
    }
    if (pv == 0 || pv >= 0x7ff0000000000000ull) {   // zero, infinite or all NaN; the same in every thread
      singular = true;
      break;
    }
    if (p != j) {
      for (int c = threadIdx.x; c < N; c += blockDim.x) {
        zc t = a[(long)j * N + c];
        a[(long)j * N + c] = a[(long)p * N + c];
        a[(long)p * N + c] = t;
      }
      if (threadIdx.x == 0) { int t = perm[j]; perm[j] = perm[p]; perm[p] = t; }
      ++swaps;
    }
    __syncthreads();
    if (j + 1 + (int)threadIdx.x < N) {   // only the warps that use it: an FP64 division of 8 warps is a column's longest step
      const zc inv = zinv(a[(long)j * N + j]);
      for (int i = j + 1 + threadIdx.x; i < N; i += blockDim.x) a[(long)i * N + j] = zmul(a[(long)i * N + j], inv);
    }
    __syncthreads();
    const int rem = N - j - 1;
    for (long e = threadIdx.x; e < (long)rem * rem; e += blockDim.x) {
      const int i = j + 1 + (int)(e / rem), c = j + 1 + (int)(e % rem);
      a[(long)i * N + c] = zfma(zmake(-a[(long)i * N + j].x, -a[(long)i * N + j].y), a[(long)j * N + c],
                                a[(long)i * N + c]);
    }
    __syncthreads();
  }
  zc la = zzero();   // (log |pivot|, arg pivot) sums
  if (!singular)
    for (int j = threadIdx.x; j < N; j += blockDim.x) {
      const zc piv = a[(long)j * N + j];
      la = zadd(la, zmake(0.5 * log(zabs2(piv)), atan2(piv.y, piv.x)));
    }
  la = block_zsum(la, s_red);
  if (threadIdx.x == 0) {
    if (singular) {
      logdet[b] = zmake(-INFINITY, 0.0);
      sing[b] = 1;
      atomicAdd(&flags[0], 1);
    } else {
      double ang = la.y + (swaps & 1 ? M_PI : 0.0);
      ang = remainder(ang, 2.0 * M_PI);
      logdet[b] = zmake(la.x, ang);
      sing[b] = 0;
    }
  }
  if (SA)   // the factors, as callers of the in-place form find them
    for (long e = threadIdx.x; e < (long)N * N; e += blockDim.x) g[e] = a[e];
  if (!want_inv) return;
  zc* out = Sinv + (long)b * N * N;
  if (singular) {
    for (long e = threadIdx.x; e < (long)N * N; e += blockDim.x) out[e] = zzero();
    return;
  }
  // U's diagonal by its reciprocals: the solves below read nothing else of it, and nothing reads the
  // factors after them
  __syncthreads();
  for (int j = threadIdx.x; j < N; j += blockDim.x) a[(long)j * N + j] = zinv(a[(long)j * N + j]);
  __syncthreads();
  zc* x = SX ? a + (long)N * N : out;
  if (SX) {
    // L U X = P by rows: once row l of X is known, every thread takes its share of the rows still to
    // come (a column per thread, as below, is one dependent chain of N^2 multiply-adds)
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) x[e] = zmake(perm[e / N] == e % N ? 1.0 : 0.0, 0.0);
    __syncthreads();
    for (int l = 0; l < N; ++l) {
      for (int e = threadIdx.x; e < (N - 1 - l) * N; e += blockDim.x) {
        const int i = l + 1 + e / N, c = e % N;
        const zc f = a[i * N + l];
        x[i * N + c] = zfma(zmake(-f.x, -f.y), x[l * N + c], x[i * N + c]);
      }
      __syncthreads();
    }
    for (int l = N - 1; l >= 0; --l) {
      for (int c = threadIdx.x; c < N; c += blockDim.x) x[l * N + c] = zmul(x[l * N + c], a[l * N + l]);
      __syncthreads();
      for (int e = threadIdx.x; e < l * N; e += blockDim.x) {
        const int i = e / N, c = e % N;
        const zc f = a[i * N + l];
        x[i * N + c] = zfma(zmake(-f.x, -f.y), x[l * N + c], x[i * N + c]);
      }
      __syncthreads();
    }
    for (int e = threadIdx.x; e < N * N; e += blockDim.x) out[e] = x[e];
    return;
  }
  // Column c of S^-1 solves L U x = P e_c: forward (unit lower), then backward.
  for (int c = threadIdx.x; c < N; c += blockDim.x) {
    for (int i = 0; i < N; ++i) {
      zc s = zmake(perm[i] == c ? 1.0 : 0.0, 0.0);
      for (int l = 0; l < i; ++l) s = zfma(zmake(-a[(long)i * N + l].x, -a[(long)i * N + l].y), x[(long)l * N + c], s);
      x[(long)i * N + c] = s;
    }
    for (int i = N - 1; i >= 0; --i) {
      zc s = x[(long)i * N + c];
      for (int l = i + 1; l < N; ++l) s = zfma(zmake(-a[(long)i * N + l].x, -a[(long)i * N + l].y), x[(long)l * N + c], s);
      x[(long)i * N + c] = zmul(s, a[(long)i * N + i]);
    }
  }
}

static cudaError_t lu_launch(afqmc_kp* h, zc* ld, int* sing, int want_inv, cudaStream_t st) {
  // pivot scratch lives in the P buffer (used otherwise only by the backward pass)
  int* perm = reinterpret_cast<int*>(h->P);
  const size_t one = sizeof(zc) * (size_t)h->N * h->N, cap = 200 * 1024;
  const bool sx = want_inv && 2 * one <= cap, sa = one <= cap;
  auto fn = sx ? lu_kernel<true, true> : sa ? lu_kernel<true, false> : lu_kernel<false, false>;
  const size_t bytes = sx ? 2 * one : sa ? one : 0;
  cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void*>(fn), bytes);
  if (e != cudaSuccess) return e;
  fn<<<2 * h->W, 256, bytes, st>>>(h->S, h->Sinv, ld, sing, h->flags, h->N, want_inv, perm);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// Gh[w][s] = (phi S^-1)^T = S^-T phi^T  (N x NM)
static cudaError_t green_impl(afqmc_kp* h, const zc* phi, zc* ld, int* sing, cudaStream_t st) {
  cudaError_t e = overlap(h, phi, st);
  if (e != cudaSuccess) return e;
  if ((e = lu_launch(h, ld, sing, 1, st)) != cudaSuccess) return e;
  const int N = h->N, NM = h->NM;
  ZGemm g = gemm_init(N, NM, N, 1, 1);
  g.A = h->Sinv; g.lda = N; g.sA[0] = (long)N * N;
  g.B = phi; g.ldb = N; g.sB[0] = (long)NM * N;
  g.C = h->Gh; g.ldc = NM; g.sC[0] = (long)N * NM;
  g.nb[0] = 2 * h->W;
  return gemm_launch(h, g, st);
}

cudaError_t green(afqmc_kp* h, const zc* phi, cudaStream_t st) {
  prof_begin(h, AFQMC_STAGE_GREEN, st);
  cudaError_t e = green_impl(h, phi, h->ld_old, h->sing_old, st);
  prof_end(h, st);
  return e;
}

// ---------------------------------------------------------------------------
// Cholesky trace X[w][Q][g] = sum_k sum_{a,r} LH[Q][k][g][a][r] (Gh_up + Gh_dn)[(k,a)][(k-Q,r)]
// Block (Q, walker chunk, vectors); one warp per g at a time, lanes over (a, r).  The vectors are
// spread over as many blocks as fill the GPU (with all of them in one block the 2x2x2 system of 16
// walkers ran on 16 SMs, 168 us).
// ---------------------------------------------------------------------------
constexpr int XWC = 8;  // walkers per block

__global__ void __launch_bounds__(256) xtrace_kernel(const zc* LH, const zc* Gh, zc* X, const int* kminus,
                                                     int nk, int G, int M, int n, int W) {
  extern __shared__ zc sm[];  // [XWC][n*M]
  const int Q = blockIdx.x, w0 = blockIdx.y * XWC;
  const int N = nk * n, NM = nk * M, nM = n * M;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int g0 = blockIdx.z * nwarp; g0 < G; g0 += nwarp * gridDim.z) {
    const int g = g0 + wid;
    zc acc[XWC];
#pragma unroll
    for (int i = 0; i < XWC; ++i) acc[i] = zzero();
    for (int k = 0; k < nk; ++k) {
      const int kq = kminus[k * nk + Q];
      __syncthreads();
      for (int e = threadIdx.x; e < XWC * nM; e += blockDim.x) {
        const int wi = e / nM, ar = e % nM, a = ar / M, r = ar % M;
        const int w = w0 + wi;
        zc v = zzero();
        if (w < W) {
          const zc* g0p = Gh + ((long)(w * 2 + 0) * N + k * n + a) * NM + kq * M + r;
          const zc* g1p = Gh + ((long)(w * 2 + 1) * N + k * n + a) * NM + kq * M + r;
          v = zadd(*g0p, *g1p);
        }
        sm[e] = v;
      }
      __syncthreads();
      if (g < G) {
        const zc* lh = LH + (((long)Q * nk + k) * G + g) * nM;
        for (int ar = lane; ar < nM; ar += 32) {
          const zc l = lh[ar];
#pragma unroll
          for (int i = 0; i < XWC; ++i) acc[i] = zfma(l, sm[i * nM + ar], acc[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < XWC; ++i) {
      zc v = warp_zsum(acc[i]);
      if (lane == 0 && g < G && w0 + i < W) X[((long)(w0 + i) * nk + Q) * G + g] = v;
    }
  }
}

cudaError_t cholesky_trace(afqmc_kp* h, cudaStream_t st) {
  const int wc = (h->W + XWC - 1) / XWC, groups = (h->G + 7) / 8;   // 8 warps, one vector each
  const long filled = (long)h->nk * wc;
  dim3 grid(h->nk, wc, (unsigned)std::max(1L, std::min((long)groups, (912 + filled - 1) / filled)));   // 6 blocks per SM
  size_t smem = sizeof(zc) * XWC * h->n * h->M;
  xtrace_kernel<<<grid, 256, smem, st>>>(h->LH, h->Gh, h->X, h->kminus, h->nk, h->G, h->M, h->n, h->W);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// xbar from X; y = sqrt(dt) * vHS coefficients (needs x; skipped when x == NULL).
__global__ void xbar_kernel(const zc* X, const double* x, zc* xbar, zc* y, const int* minus, int nk, int G,
                            long total, double sqdt) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < total; e += (long)gridDim.x * blockDim.x) {
    const int g = (int)(e % G);
    const int Q = (int)((e / G) % nk);
    const long w = e / ((long)G * nk);
    const int mQ = minus[Q];
    const zc XQ = X[(w * nk + Q) * G + g], XmQ = X[(w * nk + mQ) * G + g];
    // <v+> = i (X_Q + X_-Q)/2, <v-> = -(X_Q - X_-Q)/2, xbar = -sqrt(dt) <v>
    const zc s = zadd(XQ, XmQ), d = zsub(XQ, XmQ);
    const zc xbp = zmake(0.5 * sqdt * s.y, -0.5 * sqdt * s.x);   // -sqdt * i s / 2
    const zc xbm = zscale(d, 0.5 * sqdt);                         //  sqdt * d / 2
    xbar[((w * 2 + 0) * nk + Q) * G + g] = xbp;
    xbar[((w * 2 + 1) * nk + Q) * G + g] = xbm;
    if (x) {
      // xbar at -Q: s is symmetric, d flips sign
      const zc xbp_m = xbp, xbm_m = zscale(d, -0.5 * sqdt);
      const zc tpQ = zsub(zmake(x[((w * 2 + 0) * nk + Q) * G + g], 0.0), xbp);
      const zc tmQ = zsub(zmake(x[((w * 2 + 1) * nk + Q) * G + g], 0.0), xbm);
      const zc tpM = zsub(zmake(x[((w * 2 + 0) * nk + mQ) * G + g], 0.0), xbp_m);
      const zc tmM = zsub(zmake(x[((w * 2 + 1) * nk + mQ) * G + g], 0.0), xbm_m);
      // y = (i tp_Q - tm_Q)/2 + (i tp_-Q + tm_-Q)/2
      zc v = zmake(-tpQ.y - tmQ.x - tpM.y + tmM.x, tpQ.x - tmQ.y + tpM.x + tmM.y);
      y[(w * nk + Q) * G + g] = zscale(v, 0.5 * sqdt);
    }
  }
}

cudaError_t force_bias(afqmc_kp* h, const double* x, zc* xbar_out, cudaStream_t st) {
  long total = (long)h->W * h->nk * h->G;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  xbar_kernel<<<blocks, 256, 0, st>>>(h->X, x, xbar_out, h->y, h->minus, h->nk, h->G, total, h->sqdt);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// vHS: V[w][(k,p)][(k-Q,r)] = sum_g L[Q][k][g][p][r] y[w][Q][g]   (y carries sqrt(dt))
// Block (Q*nk + k, walker chunk); threads over (p, r).
// ---------------------------------------------------------------------------
constexpr int VWC = 8;

__global__ void __launch_bounds__(256) vhs_kernel(const zc* L, const zc* y, zc* V, const int* kminus, int nk,
                                                  int G, int M, int W) {
  extern __shared__ zc ys[];  // [VWC][G]
  const int Q = blockIdx.x / nk, k = blockIdx.x % nk, w0 = blockIdx.y * VWC;
  const int kq = kminus[k * nk + Q];
  const int NM = nk * M, MM = M * M;
  for (int e = threadIdx.x; e < VWC * G; e += blockDim.x) {
    const int wi = e / G, g = e % G;
    ys[e] = (w0 + wi < W) ? y[((long)(w0 + wi) * nk + Q) * G + g] : zzero();
  }
  __syncthreads();
  const zc* blk = L + ((long)Q * nk + k) * G * MM;
  for (int pr = threadIdx.x; pr < MM; pr += blockDim.x) {
    zc acc[VWC];
#pragma unroll
    for (int i = 0; i < VWC; ++i) acc[i] = zzero();
    for (int g = 0; g < G; ++g) {
      const zc l = blk[(long)g * MM + pr];
#pragma unroll
      for (int i = 0; i < VWC; ++i) acc[i] = zfma(l, ys[i * G + g], acc[i]);
    }
    const int p = pr / M, r = pr % M;
#pragma unroll
    for (int i = 0; i < VWC; ++i)
      if (w0 + i < W) V[(long)(w0 + i) * NM * NM + (long)(k * M + p) * NM + kq * M + r] = acc[i];
  }
}

// ---------------------------------------------------------------------------
// Hybrid weight: one block per walker.
// ---------------------------------------------------------------------------
__global__ void weight_kernel(const double* x, const zc* xbar, const zc* ld_old, const zc* ld_new,
                              const int* sing_old, const int* sing_new, double* weight, zc* logdet_out,
                              int nf) {
  const int w = blockIdx.x;
  __shared__ double red[32];
  double s = 0.0;
  // Re(x xbar - xbar^2 / 2) = xr (x - xr / 2) + xi^2 / 2: the weight needs no imaginary part, and the
  // FP64 pipe's two operations per clock are what this kernel waits for
  for (int f = threadIdx.x; f < nf; f += blockDim.x) {
    const zc xb = xbar[(long)w * nf + f];
    s = fma(xb.x, fma(-0.5, xb.x, x[(long)w * nf + f]), s);
    s = fma(0.5 * xb.y, xb.y, s);
  }
  s = block_dsum(s, red);
  if (threadIdx.x == 0) {
    const bool dead = sing_old[2 * w] || sing_old[2 * w + 1] || sing_new[2 * w] || sing_new[2 * w + 1];
    double wn = 0.0;
    if (!dead) {
      const zc dlog = zadd(zsub(ld_new[2 * w], ld_old[2 * w]), zsub(ld_new[2 * w + 1], ld_old[2 * w + 1]));
      const double c = cos(dlog.y);
      wn = weight[w] * exp(dlog.x + s) * (c > 0.0 ? c : 0.0);
    }
    weight[w] = wn;
    if (logdet_out) {
      logdet_out[2 * w] = ld_new[2 * w];
      logdet_out[2 * w + 1] = ld_new[2 * w + 1];
    }
  }
}

// ---------------------------------------------------------------------------
// Householder QR of each walker spin block (NM x N), Q factor with diag(R) > 0.
// One block per (w, s); phi overwritten; Qm is NM x N scratch.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) qr_kernel(zc* phi, zc* Qm_ws, int NM, int N) {
  const int b = blockIdx.x;
  zc* a = phi + (long)b * NM * N;
  zc* Qm = Qm_ws + (long)b * NM * N;
  extern __shared__ unsigned char qsm[];
  zc* alpha = reinterpret_cast<zc*>(qsm);          // [N]  R_jj
  zc* vhead = alpha + N;                           // [N]  first entry of v_j
  double* vn2 = reinterpret_cast<double*>(vhead + N);  // [N] |v_j|^2
  __shared__ double redd[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  for (int j = 0; j < N; ++j) {
    double ss = 0.0;
    for (int i = j + threadIdx.x; i < NM; i += blockDim.x) ss += zabs2(a[(long)i * N + j]);
    ss = block_dsum(ss, redd);
    const zc x0 = a[(long)j * N + j];
    const double nx = sqrt(ss);
    const double ax0 = sqrt(zabs2(x0));
    const zc ph = ax0 > 0.0 ? zscale(x0, 1.0 / ax0) : zmake(1.0, 0.0);
    const zc al = zscale(ph, -nx);                 // alpha = -e^{i arg x0} |x|
    const zc v0 = zsub(x0, al);                    // v = x - alpha e_0
    const double v2 = ss - zabs2(x0) + zabs2(v0);  // |v|^2
    if (threadIdx.x == 0) { alpha[j] = al; vhead[j] = v0; vn2[j] = v2; }
    __syncthreads();
    // apply H = I - 2 v v^H / |v|^2 to columns c > j ; v_i = a[i][j] for i > j, v_j = v0
    for (int c = j + 1 + wid; c < N; c += nwarp) {
      zc d = zzero();
      for (int i = j + lane; i < NM; i += 32) {
        const zc vi = (i == j) ? v0 : a[(long)i * N + j];
        d = zfma(zconj(vi), a[(long)i * N + c], d);
      }
      d = warp_zsum(d);
      const zc f = v2 > 0.0 ? zscale(d, -2.0 / v2) : zzero();
      for (int i = j + lane; i < NM; i += 32) {
        const zc vi = (i == j) ? v0 : a[(long)i * N + j];
        a[(long)i * N + c] = zfma(vi, f, a[(long)i * N + c]);
      }
    }
    __syncthreads();
  }
  // Q = H_0 ... H_{N-1} [I; 0], built backwards into Qm
  for (long e = threadIdx.x; e < (long)NM * N; e += blockDim.x) {
    const int i = (int)(e / N), c = (int)(e % N);
    Qm[e] = zmake(i == c ? 1.0 : 0.0, 0.0);
  }
  __syncthreads();
  for (int j = N - 1; j >= 0; --j) {
    const zc v0 = vhead[j];
    const double v2 = vn2[j];
    for (int c = wid; c < N; c += nwarp) {
      zc d = zzero();
      for (int i = j + lane; i < NM; i += 32) {
        const zc vi = (i == j) ? v0 : a[(long)i * N + j];
        d = zfma(zconj(vi), Qm[(long)i * N + c], d);
      }
      d = warp_zsum(d);
      const zc f = v2 > 0.0 ? zscale(d, -2.0 / v2) : zzero();
      for (int i = j + lane; i < NM; i += 32) {
        const zc vi = (i == j) ? v0 : a[(long)i * N + j];
        Qm[(long)i * N + c] = zfma(vi, f, Qm[(long)i * N + c]);
      }
    }
    __syncthreads();
  }
  // phi = Qm diag(alpha_j / |alpha_j|)  (makes diag(R) real positive)
  for (long e = threadIdx.x; e < (long)NM * N; e += blockDim.x) {
    const int c = (int)(e % N);
    const zc al = alpha[c];
    const double aa = sqrt(zabs2(al));
    const zc ph = aa > 0.0 ? zscale(al, 1.0 / aa) : zmake(1.0, 0.0);
    a[e] = zmul(Qm[e], ph);
  }
}

cudaError_t qr_with(afqmc_kp* h, zc* phi, zc* scratch, cudaStream_t st) {
  size_t smem = (size_t)h->N * (2 * sizeof(zc) + sizeof(double));
  qr_kernel<<<2 * h->W, 256, smem, st>>>(phi, scratch, h->NM, h->N);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// Same kernel, without a handle: nmat matrices of rows x cols, scratch of the same size.
// Launched through cudaLaunchKernel, whose return value is this launch's own status: an
// earlier, unrelated error stays pending for the code that caused it.
cudaError_t qr_launch(zc* phi, zc* scratch, int rows, int cols, int nmat, cudaStream_t st) {
  size_t smem = (size_t)cols * (2 * sizeof(zc) + sizeof(double));
  void* args[] = {&phi, &scratch, &rows, &cols};
  return cudaLaunchKernel(reinterpret_cast<const void*>(qr_kernel), dim3(nmat), dim3(256), args, smem, st);
}

static cudaError_t qr(afqmc_kp* h, zc* phi, cudaStream_t st) {
  size_t smem = (size_t)h->N * (2 * sizeof(zc) + sizeof(double));
  qr_kernel<<<2 * h->W, 256, smem, st>>>(phi, h->T1, h->NM, h->N);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// phi_out[w][s][(k,p)][j] = sum_q Ehalf[k][p][q] phi_in[w][s][(k,q)][j]
static cudaError_t one_body(afqmc_kp* h, const zc* in, zc* out, cudaStream_t st) {
  const int M = h->M, N = h->N, NM = h->NM;
  ZGemm g = gemm_init(M, N, M, 0, 0);
  g.A = h->Ehalf; g.lda = M; g.sA[0] = 0; g.sA[1] = (long)M * M;
  g.B = in; g.ldb = N; g.sB[0] = (long)NM * N; g.sB[1] = (long)M * N;
  g.C = out; g.ldc = N; g.sC[0] = (long)NM * N; g.sC[1] = (long)M * N;
  g.nb[0] = 2 * h->W; g.nb[1] = h->nk;
  return gemm_launch(h, g, st);
}

cudaError_t overlap_lu(afqmc_kp* h, const zc* phi, zc* ld, int* sing, int want_inv, cudaStream_t st) {
  cudaError_t e = overlap(h, phi, st);
  if (e != cudaSuccess) return e;
  return lu_launch(h, ld, sing, want_inv, st);
}

static cudaError_t logdet_only(afqmc_kp* h, const zc* phi, zc* ld, int* sing, cudaStream_t st) {
  return overlap_lu(h, phi, ld, sing, 0, st);
}

#define STAGE(stage, body)          \
  do {                              \
    prof_begin(h, stage, st);       \
    cudaError_t e_ = (body);        \
    prof_end(h, st);                \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

static cudaError_t vhs_build(afqmc_kp* h, cudaStream_t st) {
  dim3 grid(h->nk * h->nk, (h->W + VWC - 1) / VWC);
  vhs_kernel<<<grid, 256, sizeof(zc) * VWC * h->G, st>>>(h->L, h->y, h->V, h->kminus, h->nk, h->G, h->M, h->W);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// T0 = E phi ; acc = T0 ; T_j = V T_{j-1} / j ; acc += T_j ; phi = E acc
static cudaError_t taylor(afqmc_kp* h, zc* phi, cudaStream_t st) {
  cudaError_t e;
  const int NM = h->NM, N = h->N, W = h->W;
  if ((e = one_body(h, phi, h->T0, st)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(h->acc, h->T0, sizeof(zc) * (size_t)W * 2 * NM * N, cudaMemcpyDeviceToDevice, st)) !=
      cudaSuccess)
    return e;
  zc* cur = h->T0;
  zc* nxt = h->T1;
  for (int j = 1; j <= h->order; ++j) {
    ZGemm g = gemm_init(NM, N, NM, 0, 0);
    g.A = h->V; g.lda = NM; g.sA[0] = (long)NM * NM; g.sA[1] = 0;
    g.B = cur; g.ldb = N; g.sB[0] = 2L * NM * N; g.sB[1] = (long)NM * N;
    g.C = nxt; g.ldc = N; g.sC[0] = 2L * NM * N; g.sC[1] = (long)NM * N;
    g.Acc = h->acc; g.ldacc = N; g.sAcc[0] = 2L * NM * N; g.sAcc[1] = (long)NM * N;
    g.nb[0] = W; g.nb[1] = 2;
    g.alpha = zmake(1.0 / j, 0.0);
    if ((e = gemm_launch(h, g, st)) != cudaSuccess) return e;
    zc* t = cur; cur = nxt; nxt = t;
  }
  return one_body(h, h->acc, phi, st);
}

cudaError_t weights(afqmc_kp* h, const zc* phi, const double* x, double* w, zc* logdet, cudaStream_t st) {
  cudaError_t e;
  if ((e = logdet_only(h, phi, h->ld_new, h->sing_new, st)) != cudaSuccess) return e;
  weight_kernel<<<h->W, 512, 0, st>>>(x, h->xbar, h->ld_old, h->ld_new, h->sing_old, h->sing_new, w, logdet,
                                      2 * h->nk * h->G);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// Hybrid weight from the log dets already in ld_old / ld_new.
cudaError_t weight_only(afqmc_kp* h, const double* x, double* w, zc* logdet, cudaStream_t st) {
  weight_kernel<<<h->W, 512, 0, st>>>(x, h->xbar, h->ld_old, h->ld_new, h->sing_old, h->sing_new, w, logdet,
                                      2 * h->nk * h->G);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

static cudaError_t trace_and_bias(afqmc_kp* h, const double* x, zc* xbar, cudaStream_t st) {
  cudaError_t e = cholesky_trace(h, st);
  if (e != cudaSuccess) return e;
  return force_bias(h, x, xbar, st);
}

cudaError_t propagate(afqmc_kp* h, zc* phi, const double* x, double* w, zc* logdet, int do_qr,
                      cudaStream_t st) {
  cudaError_t e;
  if ((e = green(h, phi, st)) != cudaSuccess) return e;
  STAGE(AFQMC_STAGE_FORCE_BIAS, trace_and_bias(h, x, h->xbar, st));
  STAGE(AFQMC_STAGE_VHS, vhs_build(h, st));
  STAGE(AFQMC_STAGE_TAYLOR, taylor(h, phi, st));
  STAGE(AFQMC_STAGE_WEIGHT, weights(h, phi, x, w, do_qr ? nullptr : logdet, st));
  if (do_qr) return orthonormalise(h, phi, logdet, st);
  return cudaSuccess;
}

static cudaError_t qr_and_logdet(afqmc_kp* h, zc* phi, zc* logdet, cudaStream_t st) {
  cudaError_t e = qr(h, phi, st);
  if (e != cudaSuccess) return e;
  if (logdet) return logdet_only(h, phi, logdet, h->sing_new, st);
  return cudaSuccess;
}

cudaError_t orthonormalise(afqmc_kp* h, zc* phi, zc* logdet, cudaStream_t st) {
  STAGE(AFQMC_STAGE_QR, qr_and_logdet(h, phi, logdet, st));
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Local energy
// ---------------------------------------------------------------------------

// E1[w] = sum_s sum_k sum_{a,q} AhH[k][a][q] Gh[w][s][(k,a)][(k,q)];  EC[w] = 1/2 sum X_Q X_-Q
__global__ void e1_ec_kernel(const zc* AhH, const zc* Gh, const zc* X, const int* minus, zc* eloc, int nk,
                             int M, int n, int G) {
  const int w = blockIdx.x;
  const int N = nk * n, NM = nk * M;
  __shared__ zc red[32];
  zc s = zzero();
  for (long e = threadIdx.x; e < 2L * nk * n * M; e += blockDim.x) {
    const int q = (int)(e % M), a = (int)((e / M) % n), k = (int)((e / ((long)M * n)) % nk);
    const int sp = (int)(e / ((long)M * n * nk));
    s = zfma(AhH[((long)k * n + a) * M + q], Gh[((long)(w * 2 + sp) * N + k * n + a) * NM + k * M + q], s);
  }
  const zc e1 = block_zsum(s, red);
  zc c = zzero();
  for (long e = threadIdx.x; e < (long)nk * G; e += blockDim.x) {
    const int g = (int)(e % G), Q = (int)(e / G);
    c = zfma(X[((long)w * nk + Q) * G + g], X[((long)w * nk + minus[Q]) * G + g], c);
  }
  const zc ec = block_zsum(c, red);
  if (threadIdx.x == 0) {
    eloc[3 * w + 0] = e1;
    eloc[3 * w + 1] = zscale(ec, 0.5);
  }
}

// Exchange partial per (w, s, Q, k): sum over k' of the canonical (Q,k,k') terms.
// The term of (Q,k,k') equals that of its partner (-Q, k'-Q, k... ) under the
// involution (Q, k, kx) -> (-Q, kx, k) with kx = k' - Q, so only the
// lexicographically smaller member of each pair is evaluated, with weight 2.
__global__ void __launch_bounds__(256) exchange_fp64_kernel(const zc* LH, const zc* Gh, const int* kminus,
                                                            const int* minus, zc* epart, int nk, int G, int M,
                                                            int n) {
  const int ws = blockIdx.x, Q = blockIdx.y, k = blockIdx.z;
  const int N = nk * n, NM = nk * M, nM = n * M;
  const int mQ = minus[Q], kq = kminus[k * nk + Q];
  extern __shared__ zc sm[];
  zc* g1 = sm;         // Gh[(kx,b)][(k-Q, r)]  n x M
  zc* g2 = sm + nM;    // Gh[(k,a)][(kx+Q, s)]  n x M
  __shared__ zc red[32];
  const zc* Gw = Gh + (long)ws * N * NM;
  zc acc = zzero();
  for (int kx = 0; kx < nk; ++kx) {
    // partner of (Q, k, kx) is (mQ, kx, k)
    const bool self = (mQ == Q) && (kx == k);
    const bool canon = (Q < mQ) || (Q == mQ && k <= kx);
    if (!canon) continue;
    const double wt = self ? 1.0 : 2.0;
    const int kxq = kminus[kx * nk + mQ];  // kx + Q
    __syncthreads();
    for (int e = threadIdx.x; e < nM; e += blockDim.x) {
      const int a = e / M, r = e % M;
      g1[e] = Gw[(long)(kx * n + a) * NM + kq * M + r];
      g2[e] = Gw[(long)(k * n + a) * NM + kxq * M + r];
    }
    __syncthreads();
    const zc* L1 = LH + ((long)Q * nk + k) * G * nM;    // LH[Q][k]
    const zc* L2 = LH + ((long)mQ * nk + kx) * G * nM;  // LH[-Q][kx]
    for (int e = threadIdx.x; e < G * n * n; e += blockDim.x) {
      const int g = e / (n * n), a = (e / n) % n, b = e % n;
      // T1[g,a,b] = sum_r LH[Q,k,g,a,r] Gh[(kx,b),(k-Q,r)]
      // T2[g,b,a] = sum_s LH[-Q,kx,g,b,s] Gh[(k,a),(kx+Q,s)]
      zc t1 = zzero(), t2 = zzero();
      const zc* l1 = L1 + ((long)g * n + a) * M;
      const zc* l2 = L2 + ((long)g * n + b) * M;
      for (int r = 0; r < M; ++r) {
        t1 = zfma(l1[r], g1[b * M + r], t1);
        t2 = zfma(l2[r], g2[a * M + r], t2);
      }
      acc = zadd(acc, zscale(zmul(t1, t2), wt));
    }
  }
  acc = block_zsum(acc, red);
  if (threadIdx.x == 0) epart[((long)ws * nk + Q) * nk + k] = zscale(acc, -0.5);
}

__global__ void ex_reduce_kernel(const zc* epart, zc* eloc, int per_walker) {
  const int w = blockIdx.x;
  __shared__ zc red[32];
  zc s = zzero();
  for (int i = threadIdx.x; i < per_walker; i += blockDim.x) s = zadd(s, epart[(long)w * per_walker + i]);
  s = block_zsum(s, red);
  if (threadIdx.x == 0) eloc[3 * w + 2] = s;
}

static cudaError_t e1_ec(afqmc_kp* h, zc* eloc, cudaStream_t st) {
  e1_ec_kernel<<<h->W, 256, 0, st>>>(h->AhH, h->Gh, h->X, h->minus, eloc, h->nk, h->M, h->n, h->G);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

static cudaError_t exchange(afqmc_kp* h, cudaStream_t st) {
  dim3 grid(2 * h->W, h->nk, h->nk);
  exchange_fp64_kernel<<<grid, 256, sizeof(zc) * 2 * h->n * h->M, st>>>(h->LH, h->Gh, h->kminus, h->minus,
                                                                        h->epart, h->nk, h->G, h->M, h->n);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

static cudaError_t ex_reduce(afqmc_kp* h, zc* eloc, cudaStream_t st) {
  ex_reduce_kernel<<<h->W, 256, 0, st>>>(h->epart, eloc, 2 * h->nk * h->nk);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

cudaError_t local_energy(afqmc_kp* h, const zc* phi, zc* eloc, cudaStream_t st) {
  cudaError_t e;
  if ((e = green(h, phi, st)) != cudaSuccess) return e;
  STAGE(AFQMC_STAGE_FORCE_BIAS, cholesky_trace(h, st));
  STAGE(AFQMC_STAGE_ENERGY, e1_ec(h, eloc, st));
  STAGE(AFQMC_STAGE_EXCHANGE, exchange(h, st));
  STAGE(AFQMC_STAGE_ENERGY, ex_reduce(h, eloc, st));
  return cudaSuccess;
}

// One fused walker step: propagate every walker and evaluate the local energy of
// the propagated walkers.  The Green's function of the new walkers serves the
// new log det (weights), the energy, and the next step's force bias.
cudaError_t step(afqmc_kp* h, zc* phi, const double* x, double* w, zc* eloc, zc* logdet, int do_qr, int reuse,
                 cudaStream_t st) {
  cudaError_t e;
  if (!reuse) {
    STAGE(AFQMC_STAGE_GREEN, green_impl(h, phi, h->ld_old, h->sing_old, st));
    STAGE(AFQMC_STAGE_FORCE_BIAS, cholesky_trace(h, st));
  }
  STAGE(AFQMC_STAGE_FORCE_BIAS, force_bias(h, x, h->xbar, st));
  STAGE(AFQMC_STAGE_VHS, vhs_build(h, st));
  STAGE(AFQMC_STAGE_TAYLOR, taylor(h, phi, st));
  STAGE(AFQMC_STAGE_GREEN, green_impl(h, phi, h->ld_new, h->sing_new, st));
  STAGE(AFQMC_STAGE_FORCE_BIAS, cholesky_trace(h, st));
  STAGE(AFQMC_STAGE_WEIGHT, weight_only(h, x, w, do_qr ? nullptr : logdet, st));
  if (eloc) {   // NULL: a propagation-only step of a block (the energy is measured less often)
    STAGE(AFQMC_STAGE_ENERGY, e1_ec(h, eloc, st));
    STAGE(AFQMC_STAGE_EXCHANGE, exchange(h, st));
    STAGE(AFQMC_STAGE_ENERGY, ex_reduce(h, eloc, st));
  }
  if (do_qr) {
    // the Green's function is invariant under phi -> phi R^-1; only the log det moves
    STAGE(AFQMC_STAGE_QR, qr(h, phi, st));
    STAGE(AFQMC_STAGE_QR, overlap_lu(h, phi, h->ld_new, h->sing_new, 0, st));
    if (logdet &&
        (e = cudaMemcpyAsync(logdet, h->ld_new, sizeof(zc) * 2 * h->W, cudaMemcpyDeviceToDevice, st)) != cudaSuccess)
      return e;
  }
  std::swap(h->ld_old, h->ld_new);
  std::swap(h->sing_old, h->sing_new);
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Adjoint of the local energy
// ---------------------------------------------------------------------------

// Gam[w][s][(k,a)][(k-Q,r)] = c2 sum_g X[w][-Q][g] LH[Q][k][g][a][r] + (Q == 0 ? c1 AhH[k][a][r] : 0)
// with c = conj(grad_e).  Every (k, k') block is written exactly once.
__global__ void gamma_init_kernel(const zc* LH, const zc* X, const zc* AhH, const zc* grad_e, zc* Gam,
                                  const int* kminus, const int* minus, int nk, int G, int M, int n) {
  const int ws = blockIdx.x, k = blockIdx.y, Q = blockIdx.z;
  const int w = ws >> 1;
  const int N = nk * n, NM = nk * M, nM = n * M;
  const int kq = kminus[k * nk + Q], mQ = minus[Q];
  const zc c1 = zconj(grad_e[3 * w + 0]), c2 = zconj(grad_e[3 * w + 1]);
  const zc* xm = X + ((long)w * nk + mQ) * G;
  const zc* lh = LH + ((long)Q * nk + k) * G * nM;
  for (int e = threadIdx.x; e < nM; e += blockDim.x) {
    zc s = zzero();
    for (int g = 0; g < G; ++g) s = zfma(xm[g], lh[(long)g * nM + e], s);
    s = zmul(c2, s);
    if (Q == 0) s = zfma(c1, AhH[(long)k * nM + e], s);
    const int a = e / M, r = e % M;
    Gam[((long)ws * N + k * n + a) * NM + kq * M + r] = s;
  }
}

// Gam[(kx,b)][(c,r)] += -c3 sum_Q sum_{g,a} T2[g,b,a] LH[Q][c+Q][g][a][r],
// T2[g,b,a] = sum_s LH[-Q][kx][g][b][s] Gh[(c+Q,a)][(kx+Q,s)].  Block (w s, kx, c).
__global__ void __launch_bounds__(256) gamma_exchange_kernel(const zc* LH, const zc* Gh, const zc* grad_e,
                                                             zc* Gam, const int* kminus, const int* minus,
                                                             int nk, int G, int M, int n) {
  const int ws = blockIdx.x, kx = blockIdx.y, c = blockIdx.z;
  const int w = ws >> 1;
  const int N = nk * n, NM = nk * M, nM = n * M;
  const zc c3 = zconj(grad_e[3 * w + 2]);
  extern __shared__ zc sm[];
  zc* gblk = sm;            // n x M : Gh[(k,a)][(kx+Q, s)]
  zc* T2 = sm + nM;         // G x n x n
  const zc* Gw = Gh + (long)ws * N * NM;
  // each thread owns outputs e = (b, r) over n*M entries
  zc outv[4];
  const int per = (nM + blockDim.x - 1) / blockDim.x;
  for (int i = 0; i < 4; ++i) outv[i] = zzero();
  for (int Q = 0; Q < nk; ++Q) {
    const int mQ = minus[Q];
    const int k = kminus[c * nk + mQ];      // k = c + Q
    const int kxq = kminus[kx * nk + mQ];   // kx + Q
    __syncthreads();
    for (int e = threadIdx.x; e < nM; e += blockDim.x) {
      const int a = e / M, s = e % M;
      gblk[e] = Gw[(long)(k * n + a) * NM + kxq * M + s];
    }
    __syncthreads();
    const zc* L2 = LH + ((long)mQ * nk + kx) * G * nM;
    for (int e = threadIdx.x; e < G * n * n; e += blockDim.x) {
      const int g = e / (n * n), b = (e / n) % n, a = e % n;
      zc t = zzero();
      const zc* l2 = L2 + ((long)g * n + b) * M;
      for (int s = 0; s < M; ++s) t = zfma(l2[s], gblk[a * M + s], t);
      T2[e] = t;
    }
    __syncthreads();
    const zc* L1 = LH + ((long)Q * nk + k) * G * nM;
    for (int i = 0; i < per && i < 4; ++i) {
      const int e = threadIdx.x + i * blockDim.x;
      if (e >= nM) break;
      const int b = e / M, r = e % M;
      zc s = outv[i];
      for (int g = 0; g < G; ++g)
        for (int a = 0; a < n; ++a) s = zfma(T2[((long)g * n + b) * n + a], L1[((long)g * n + a) * M + r], s);
      outv[i] = s;
    }
  }
  for (int i = 0; i < per && i < 4; ++i) {
    const int e = threadIdx.x + i * blockDim.x;
    if (e >= nM) break;
    const int b = e / M, r = e % M;
    zc* o = Gam + ((long)ws * N + kx * n + b) * NM + c * M + r;
    *o = zsub(*o, zmul(c3, outv[i]));
  }
}

// grad_h1[k][p][q] = sum_w g1[w] sum_s sum_a A[k][p][a] conj(Gh[w][s][(k,a)][(k,q)])
__global__ void grad_h1_kernel(const zc* A, const zc* Gh, const zc* grad_e, zc* gh1, int nk, int M, int n,
                               int W) {
  const int k = blockIdx.x;
  const int N = nk * n, NM = nk * M;
  for (int e = threadIdx.x; e < M * M; e += blockDim.x) {
    const int p = e / M, q = e % M;
    zc s = zzero();
    for (int w = 0; w < W; ++w) {
      zc t = zzero();
      for (int sp = 0; sp < 2; ++sp)
        for (int a = 0; a < n; ++a)
          t = zfma(A[((long)k * M + p) * n + a], zconj(Gh[((long)(w * 2 + sp) * N + k * n + a) * NM + k * M + q]), t);
      s = zfma(grad_e[3 * w + 0], t, s);
    }
    gh1[(long)k * M * M + e] = s;
  }
}

static cudaError_t grad_h1(afqmc_kp* h, const zc* grad_e, zc* gh1, cudaStream_t st) {
  grad_h1_kernel<<<h->nk, 256, 0, st>>>(h->A, h->Gh, grad_e, gh1, h->nk, h->M, h->n, h->W);
  AFQMC_LAUNCHED(h);
  return cudaGetLastError();
}

// dE/dphi from Gam = conj(grad_e)-weighted dE/dGh: with Gh = S^-T phi^T and S = A^dag phi,
// dGh = S^-T dphi^T (I - A* Gh), so grad_phi = [S^-1 (Gam - (Gam Gh^T) A^dag)]^H in the
// conjugate convention of the binding.
static cudaError_t project_gamma(afqmc_kp* h, zc* grad_phi, cudaStream_t st) {
  cudaError_t e;
  const int nk = h->nk, M = h->M, n = h->n, N = h->N, NM = h->NM, W = h->W;
  {  // P = Gam Gh^T  (N x N)
    ZGemm g = gemm_init(N, N, NM, 0, 1);
    g.A = h->Gam; g.lda = NM; g.sA[0] = (long)N * NM;
    g.B = h->Gh; g.ldb = NM; g.sB[0] = (long)N * NM;
    g.C = h->P; g.ldc = N; g.sC[0] = (long)N * N;
    g.nb[0] = 2 * W;
    if ((e = gemm_launch(h, g, st)) != cudaSuccess) return e;
  }
  {  // Gam[:, k-block] -= P[:, k-block of n] A[k]^dagger
    ZGemm g = gemm_init(N, M, n, 0, 2);
    g.A = h->P; g.lda = N; g.sA[0] = (long)N * N; g.sA[1] = n;
    g.B = h->A; g.ldb = n; g.sB[0] = 0; g.sB[1] = (long)M * n;
    g.C = h->Gam; g.ldc = NM; g.sC[0] = (long)N * NM; g.sC[1] = M;
    g.nb[0] = 2 * W; g.nb[1] = nk;
    g.alpha = zmake(-1.0, 0.0);
    g.beta = zmake(1.0, 0.0);
    if ((e = gemm_launch(h, g, st)) != cudaSuccess) return e;
  }
  {  // grad_phi = Gam^H Sinv^H  (NM x N)
    ZGemm g = gemm_init(NM, N, N, 2, 2);
    g.A = h->Gam; g.lda = NM; g.sA[0] = (long)N * NM;
    g.B = h->Sinv; g.ldb = N; g.sB[0] = (long)N * N;
    g.C = grad_phi; g.ldc = N; g.sC[0] = (long)NM * N;
    g.nb[0] = 2 * W;
    if ((e = gemm_launch(h, g, st)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

static cudaError_t backward_impl(afqmc_kp* h, const zc* grad_e, zc* grad_phi, zc* gh1, cudaStream_t st) {
  cudaError_t e;
  const int nk = h->nk, M = h->M, n = h->n, W = h->W;
  if (gh1 && (e = grad_h1(h, grad_e, gh1, st)) != cudaSuccess) return e;
  if (!grad_phi) return cudaSuccess;
  if ((e = cholesky_trace(h, st)) != cudaSuccess) return e;
  gamma_init_kernel<<<dim3(2 * W, nk, nk), 128, 0, st>>>(h->LH, h->X, h->AhH, grad_e, h->Gam, h->kminus, h->minus,
                                                          nk, h->G, M, n);
  AFQMC_LAUNCHED(h);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  gamma_exchange_kernel<<<dim3(2 * W, nk, nk), 256, sizeof(zc) * (n * M + h->G * n * n), st>>>(
      h->LH, h->Gh, grad_e, h->Gam, h->kminus, h->minus, nk, h->G, M, n);
  AFQMC_LAUNCHED(h);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return project_gamma(h, grad_phi, st);
}

cudaError_t local_energy_backward(afqmc_kp* h, const zc* phi, const zc* grad_e, zc* grad_phi, zc* grad_h1,
                                  cudaStream_t st) {
  cudaError_t e;
  if ((e = green(h, phi, st)) != cudaSuccess) return e;
  STAGE(AFQMC_STAGE_BACKWARD, backward_impl(h, grad_e, grad_phi, grad_h1, st));
  return cudaSuccess;
}

static cudaError_t set_smem(const void* fn, size_t bytes) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  if (bytes > 227 * 1024) return cudaErrorNotSupported;   // larger than one CTA may hold
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Opt in to the dynamic shared memory each kernel needs at this system size.  A tensor-core
// (mixed) handle runs none of these kernels (its own take their place), so it needs none.
static cudaError_t configure_smem(afqmc_kp* h) {
  if (h->d.prec == AFQMC_MIXED) return cudaSuccess;
  cudaError_t e = set_smem((const void*)vhs_kernel, sizeof(zc) * VWC * h->G);
  if (e == cudaSuccess)
    e = set_smem((const void*)gamma_exchange_kernel, sizeof(zc) * (h->n * h->M + (size_t)h->G * h->n * h->n));
  if (e == cudaSuccess) e = set_smem((const void*)xtrace_kernel, sizeof(zc) * XWC * h->n * h->M);
  if (e == cudaSuccess) e = set_smem((const void*)qr_kernel, (size_t)h->N * (2 * sizeof(zc) + sizeof(double)));
  if (e == cudaSuccess) e = set_smem((const void*)exchange_fp64_kernel, sizeof(zc) * 2 * h->n * h->M);
  return e;
}

}  // namespace fp64
