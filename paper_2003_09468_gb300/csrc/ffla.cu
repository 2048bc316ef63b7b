// Double-float dense kernels of the tensor-core path (ff.cuh): the overlap matrix,
// the trial-subspace projection of the walker, and the inverse / log-determinant
// of the overlap matrix.
//
// These are the steps of Sec. 3.2 (step 1, the Green's function of Eq. kp_gf) whose
// results need more than the 22 bits of the split GEMM: S = A^dag phi enters the
// log-determinant (the weight, Eq. hybrid) and its inverse; phi_perp = phi - B S is a
// cancelling difference.  FP64 would serve, but this GPU's FP64 pipe is two fused
// multiply-adds per clock per SM; double-float arithmetic on the FP32 pipe keeps 48
// bits at several times the speed.
#include <cuda_fp16.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>
#include <cmath>

#include "attr.hpp"
#include "ff.cuh"
#include "ffla.hpp"
#include "split.cuh"

namespace ffla {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int OV_THREADS = 256;
constexpr int GJ_THREADS = 512;
constexpr int GJ_WARPS = GJ_THREADS / 32;
constexpr size_t OV_SMEM_TARGET = 96 * 1024;
constexpr size_t SMEM_LIMIT = 220 * 1024;

__device__ __forceinline__ float block_max_f(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(FULL, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float m = 0.f;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = fmaxf(m, red[i]);
  return m;
}
__device__ __forceinline__ double block_sum_d(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += red[i];
  return s;
}

// S[ws][(k,a)][j] = sum_p conj(A[k][p][a]) phi[ws][(k,p)][j]                       (Eq. kp_gf)
// PROJECT: phi_perp[ws][(k,p)][j] = phi[ws][(k,p)][j] - sum_a B[k][p][a] S[ws][(k,a)][j]
// (rounded to fp32) and mx[ws] = max |phi_perp| (atomic max on the bits of a
// non-negative double).  Grid (WS, nk, column chunks of JC).
template <bool PROJECT>
__global__ void __launch_bounds__(OV_THREADS)
    overlap_ff_kernel(const zc* A, const zc* phi, const zc* B, float4* Sff, float2* phi_perp,
                      unsigned long long* mx, int nk, int M, int n, int N, int JC) {
  extern __shared__ __align__(16) unsigned char ov_smem[];
  __shared__ float red[OV_THREADS / 32];
  const int ws = blockIdx.x, k = blockIdx.y, j0 = blockIdx.z * JC, tid = threadIdx.x;
  const int jc = min(JC, N - j0);
  float4* ph = reinterpret_cast<float4*>(ov_smem);   // [M][JC]
  float4* Ak = ph + (size_t)M * JC;                    // [M][n]
  float4* Bk = Ak + (size_t)M * n;                     // [M][n]
  float4* Sk = Bk + (size_t)M * n;                     // [n][JC]
  const size_t row0 = (size_t)ws * nk * M + (size_t)k * M;   // first row (k, 0) of this walker-spin
  for (int e = tid; e < M * jc; e += OV_THREADS) {
    const int p = e / jc, jj = e % jc;
    ph[p * JC + jj] = ffa::cfrom(phi[(row0 + p) * N + j0 + jj]);
  }
  for (int e = tid; e < M * n; e += OV_THREADS) {
    Ak[e] = ffa::cfrom(A[(size_t)k * M * n + e]);
    if (PROJECT) Bk[e] = ffa::cfrom(B[(size_t)k * M * n + e]);
  }
  __syncthreads();
  for (int e = tid; e < n * jc; e += OV_THREADS) {
    const int a = e / jc, jj = e % jc;
    ffa::cacc acc = ffa::cacc_from(ffa::czero());
    for (int p = 0; p < M; ++p) ffa::cacc_fma_conj(acc, Ak[p * n + a], ph[p * JC + jj]);
    const float4 v = ffa::cacc_get(acc);
    Sk[a * JC + jj] = v;
    Sff[((size_t)ws * N + (size_t)k * n + a) * N + j0 + jj] = v;
  }
  if (!PROJECT) return;
  __syncthreads();
  float m = 0.f;
  for (int e = tid; e < M * jc; e += OV_THREADS) {
    const int p = e / jc, jj = e % jc;
    ffa::cacc pa = ffa::cacc_from(ph[p * JC + jj]);
    for (int a = 0; a < n; ++a) ffa::cacc_fms(pa, Bk[p * n + a], Sk[a * JC + jj]);
    const float4 v = ffa::cacc_get(pa);
    const float2 o = make_float2(__fadd_rn(v.x, v.y), __fadd_rn(v.z, v.w));
    phi_perp[(row0 + p) * N + j0 + jj] = o;
    m = fmaxf(m, fmaxf(fabsf(o.x), fabsf(o.y)));
  }
  m = block_max_f(m, red);
  if (tid == 0) atomicMax(mx + ws, static_cast<unsigned long long>(__double_as_longlong((double)m)));
}

// log det of one N x N matrix per CTA, by an in-place LU factorisation with partial (row)
// pivoting in double-float.  Step j: pick the row p >= j with the largest |re| + |im| in column j,
// swap rows j and p, eliminate below the diagonal.  The pivots are the diagonal of U in P S = L U, so
//   log det S = sum_j log a_jj + i pi (number of swaps mod 2).
// A zero or non-finite pivot marks the matrix singular: logdet = (-inf, 0), sing = 1,
// flags[0] counts it.
// For matrices that the cluster form below does not take; the matrix stays in global memory (L2).
__global__ void __launch_bounds__(GJ_THREADS) gj_ff_kernel(float4* Sff, int N, zc* logdet, int* sing, int* flags) {
  extern __shared__ __align__(16) unsigned char gj_smem[];
  __shared__ int s_p, s_sing, s_swaps;
  __shared__ float4 s_pv, s_ajj;
  __shared__ double s_red[GJ_WARPS];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float4* a = Sff + (size_t)b * N * N;
  float4* f = reinterpret_cast<float4*>(gj_smem);
  double2* piv = reinterpret_cast<double2*>(f + N);
  if (tid == 0) {
    s_sing = 0;
    s_swaps = 0;
  }
  __syncthreads();
  for (int j = 0; j < N; ++j) {
    if (warp == 0) {
      float best = -1.f;
      int bi = j;
      for (int i = j + lane; i < N; i += 32) {
        const float4 v = a[(size_t)i * N + j];
        const float m = fabsf(v.x) + fabsf(v.z);
        if (m > best) {
          best = m;
          bi = i;
        }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const float b2 = __shfl_xor_sync(FULL, best, o);
        const int i2 = __shfl_xor_sync(FULL, bi, o);
        if (b2 > best || (b2 == best && i2 < bi)) {
          best = b2;
          bi = i2;
        }
      }
      if (lane == 0) {
        s_p = bi;
        s_pv = a[(size_t)bi * N + j];
        s_ajj = a[(size_t)j * N + j];
        if (!(best > 0.f) || !isfinite(best)) {
          s_sing = 1;
        } else if (bi != j) {
          ++s_swaps;
        }
      }
    }
    __syncthreads();
    if (s_sing) break;   // the same shared value for every thread after the barrier
    const int p = s_p;
    const float4 pv = s_pv, ajj = s_ajj;
    const float4 inv = ffa::crecip(pv);
    if (tid == 0) piv[j] = make_double2(ffa::to_double(ffa::re(pv)), ffa::to_double(ffa::im(pv)));
    // swap rows j and p (each thread owns whole columns)
    for (int c = tid; c < N; c += GJ_THREADS) {
      const float4 tj = a[(size_t)j * N + c];
      const float4 tp = (p == j) ? tj : a[(size_t)p * N + c];
      a[(size_t)j * N + c] = tp;
      if (p != j) a[(size_t)p * N + c] = tj;
    }
    // multipliers: column j after the swap (rows j and p are the only ones moved)
    for (int i = tid; i < N; i += GJ_THREADS) {
      float4 fi;
      if (i == j)
        fi = ffa::czero();
      else
        fi = (i == p) ? ajj : a[(size_t)i * N + j];
      f[i] = ffa::cmul(fi, inv);
    }
    __syncthreads();
    const float4* aj = a + (size_t)j * N;
    for (int i = j + 1 + warp; i < N; i += GJ_WARPS) {
      const float4 fi = f[i];
      float4* ai = a + (size_t)i * N;
      for (int c = j + 1 + lane; c < N; c += 32) ai[c] = ffa::cfms(ai[c], fi, aj[c]);
    }
    __syncthreads();
  }
  const int singular = s_sing;
  double lg = 0.0, an = 0.0;
  if (!singular)
    for (int i = tid; i < N; i += GJ_THREADS) {
      const double2 v = piv[i];
      lg += 0.5 * log(v.x * v.x + v.y * v.y);
      an += atan2(v.y, v.x);
    }
  lg = block_sum_d(lg, s_red);
  an = block_sum_d(an, s_red);
  if (tid == 0) {
    if (singular) {
      logdet[b] = make_double2(-INFINITY, 0.0);
      sing[b] = 1;
      atomicAdd(&flags[0], 1);
    } else {
      double ang = an + ((s_swaps & 1) ? M_PI : 0.0);
      ang = remainder(ang, 2.0 * M_PI);
      logdet[b] = make_double2(lg, ang);
      sing[b] = 0;
    }
  }
}

// The inverse of one matrix per CTA by Gauss-Jordan elimination with partial (row) pivoting, in place.
// An unblocked step j picks and swaps rows as above, scales row j by 1/a_jj (a_jj itself becomes 1/a_jj)
// and eliminates column j from every other row (a_ij becomes -a_ij / a_jj): after N steps the
// array holds (P S)^-1, P the row permutation, so S^-1[:, perm[i]] = column i.  A singular matrix's
// inverse is written as zero.  Output: the split planes of S^-T, out[b][N][Np] (split.cuh) with scale
// s_out[b].
//
// Pivots are taken in panels of GJB columns:
// within a panel every step updates only the panel's columns (all rows), so that afterwards
// those columns hold the panel's accumulated transform T (T - I has non-zeros only there); every
// other column c then receives the panel's row swaps and one rank-GJB update
// c <- T c = c + (T - I)[:, panel] c[panel rows].  The matrix lives in place in global memory
// (the overlap buffer, L2-resident while the CTA works on it): each panel reads and writes the
// matrix once, where the unblocked kernel does so once per pivot.
constexpr int GJB = 8;
static_assert(GJB == 8, "the panel's index arithmetic uses shifts by 3");
constexpr int GJB_THREADS = 512;
constexpr int GJB_WARPS = GJB_THREADS / 32;
constexpr int GJB_GLOBAL_MAXN = 1024;   // a handle's largest N; GJB N float4 + per-row arrays are within SMEM_LIMIT

// Pivot candidate key: larger |value| first, then the smaller row (m >= 0 and not NaN, so its
// bits order as the values do).
__device__ __forceinline__ unsigned long long pivot_key(float m, int i) {
  return ((unsigned long long)__float_as_uint(m) << 32) | (unsigned long long)(0xffffffffu - (unsigned)i);
}

__global__ void __launch_bounds__(GJB_THREADS)
    gjb_ff_kernel(float4* Sff, int N, zc* logdet, int* sing, int* flags, __half* out, int Np, float* s_out) {
  extern __shared__ __align__(16) unsigned char gj_smem[];
  __shared__ int s_swaps;
  __shared__ unsigned long long s_key[2];   // the next pivot's (|value|, row) key, two in turn
  __shared__ double s_red[GJB_WARPS];
  __shared__ float s_redf[GJB_WARPS];
  __shared__ int s_prow[GJB];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float4* a = Sff + (size_t)b * N * N;                    // [N][N]
  float4* tmp = reinterpret_cast<float4*>(gj_smem);       // [GJB][N] panel rows
  float4* f = tmp + (size_t)GJB * N;                      // [N] multipliers
  double2* piv = reinterpret_cast<double2*>(f + N);
  int* perm = reinterpret_cast<int*>(piv + N);
  int* iperm = perm + N;
  for (int i = tid; i < N; i += GJB_THREADS) perm[i] = i;
  if (tid == 0) s_swaps = 0;
  __syncthreads();
  // Every thread reads the same shared pivot keys after the same barriers, so it takes the
  // singular exit at the same step as the others.
  bool singular_l = false;
  for (int j0 = 0; j0 < N && !singular_l; j0 += GJB) {
    const int jb = min(GJB, N - j0);
    // ---- panel: columns [j0, j0 + jb), every row
    // The pivot of column j is the row i >= j of largest |re.hi| + |im.hi| (the smallest i
    // among equals).  The panel's first column was last written by the rank update and is
    // searched by warp 0; every later column j + 1 is searched while the elimination of
    // column j writes it (a warp maximum of the (|value|, row) keys, then one shared atomic
    // maximum per warp), which saves the search's serial pass and a barrier per pivot.
    for (int jj = 0; jj < jb; ++jj) {
      const int j = j0 + jj;
      if (jj == 0) {
        if (warp == 0) {
          float best = -1.f;
          int bi = j;
          for (int i = j + lane; i < N; i += 32) {
            const float4 v = a[(size_t)i * N + j];
            const float m = fabsf(v.x) + fabsf(v.z);
            if (m > best) {
              best = m;
              bi = i;
            }
          }
          for (int o = 16; o > 0; o >>= 1) {
            const float b2 = __shfl_xor_sync(FULL, best, o);
            const int i2 = __shfl_xor_sync(FULL, bi, o);
            if (b2 > best || (b2 == best && i2 < bi)) {
              best = b2;
              bi = i2;
            }
          }
          if (lane == 0) s_key[0] = best >= 0.f ? pivot_key(best, bi) : 0ull;
        }
        __syncthreads();
      }
      const unsigned long long key = s_key[jj & 1];
      const float best = __uint_as_float((unsigned)(key >> 32));
      if (!(best > 0.f) || !isfinite(best)) {
        singular_l = true;
        break;
      }
      const int p = (int)(0xffffffffu - (unsigned)(key & 0xffffffffull));
      const float4 pv = a[(size_t)p * N + j], ajj = a[(size_t)j * N + j];
      const float4 inv = ffa::crecip(pv);
      if (tid == 0) {
        s_prow[jj] = p;
        if (p != j) {
          const int t = perm[j];
          perm[j] = perm[p];
          perm[p] = t;
          ++s_swaps;
        }
        piv[j] = make_double2(ffa::to_double(ffa::re(pv)), ffa::to_double(ffa::im(pv)));
        s_key[(jj + 1) & 1] = 0ull;   // read last before the previous step's barriers
      }
      // swap rows j and p and scale row j, panel columns other than j (the elimination below
      // writes column j whole: inv in row j, -f inv elsewhere)
      for (int cc = tid; cc < jb; cc += GJB_THREADS) {
        const int c = j0 + cc;
        if (c == j) continue;
        const float4 tj = a[(size_t)j * N + c];
        const float4 tp = (p == j) ? tj : a[(size_t)p * N + c];
        a[(size_t)j * N + c] = ffa::cmul(tp, inv);
        if (p != j) a[(size_t)p * N + c] = tj;
      }
      for (int i = tid; i < N; i += GJB_THREADS) {
        if (i == j)
          f[i] = ffa::czero();
        else
          f[i] = (i == p) ? ajj : a[(size_t)i * N + j];
      }
      __syncthreads();
      // eliminate column j from every other row, panel columns only: one thread per
      // (row, panel column)
      unsigned long long cand = 0ull;
      for (int e = tid; e < N * jb; e += GJB_THREADS) {
        const int i = (jb == GJB) ? (e >> 3) : e / jb, c = j0 + ((jb == GJB) ? (e & 7) : e % jb);
        if (c == j) {
          a[(size_t)i * N + c] = (i == j) ? inv : ffa::cneg(ffa::cmul(f[i], inv));
          continue;
        }
        if (i == j) continue;
        const float4 v = ffa::cfms(a[(size_t)i * N + c], f[i], a[(size_t)j * N + c]);
        a[(size_t)i * N + c] = v;
        if (c == j + 1 && i > j) {
          const float m = fabsf(v.x) + fabsf(v.z);
          if (!isnan(m)) cand = max(cand, pivot_key(m, i));
        }
      }
      if (jj + 1 < jb) {
        for (int o = 16; o > 0; o >>= 1) {
          const unsigned long long other = __shfl_xor_sync(FULL, cand, o);
          cand = other > cand ? other : cand;
        }
        if (lane == 0 && cand) atomicMax(&s_key[(jj + 1) & 1], cand);
      }
      __syncthreads();
    }
    if (singular_l) break;
    // ---- every other column: the panel's row swaps in order, a copy of the panel rows
    const int R = N - jb;   // rest column r -> c = r < j0 ? r : r + jb
    for (int r = tid; r < R; r += GJB_THREADS) {
      const int c = (r < j0) ? r : r + jb;
      for (int jj = 0; jj < jb; ++jj) {
        const int j = j0 + jj, p = s_prow[jj];
        if (p != j) {
          const float4 t = a[(size_t)j * N + c];
          a[(size_t)j * N + c] = a[(size_t)p * N + c];
          a[(size_t)p * N + c] = t;
        }
      }
      for (int jj = 0; jj < jb; ++jj) tmp[(size_t)jj * N + r] = a[(size_t)(j0 + jj) * N + c];
    }
    __syncthreads();
    // ---- rank-jb update a[i][c] += sum_l (T - I)[i][j0 + l] tmp[l][c]: a thread takes one
    // row and two rest columns r and r + H (H = ceil(R / 2)), consecutive threads consecutive
    // r, so a warp reads tmp in one conflict-free run and (mostly) one row's multipliers;
    // N H tasks spread evenly over the threads
    {
      const int H = (R + 1) / 2;
      for (int u = tid; u < N * H; u += GJB_THREADS) {
        const int i = u / H, rA = u % H, rB = rA + H;
        const bool okB = rB < R;
        const int cA = (rA < j0) ? rA : rA + jb, cB = (rB < j0) ? rB : rB + jb;
        ffa::cacc xA = ffa::cacc_from(a[(size_t)i * N + cA]);
        ffa::cacc xB = ffa::cacc_from(okB ? a[(size_t)i * N + cB] : ffa::czero());
        for (int l = 0; l < jb; ++l) {
          float4 d = a[(size_t)i * N + j0 + l];
          if (i == j0 + l) d = ffa::pack(ffa::add(ffa::re(d), ffa::make(-1.f, 0.f)), ffa::im(d));
          const float4 tA = tmp[(size_t)l * N + rA];
          const float4 tB = okB ? tmp[(size_t)l * N + rB] : ffa::czero();
          ffa::cacc_fma(xA, d, tA);
          ffa::cacc_fma(xB, d, tB);
        }
        a[(size_t)i * N + cA] = ffa::cacc_get(xA);
        if (okB) a[(size_t)i * N + cB] = ffa::cacc_get(xB);
      }
    }
    __syncthreads();
  }
  const int singular = singular_l;
  double lg = 0.0, an = 0.0;
  if (!singular)
    for (int i = tid; i < N; i += GJB_THREADS) {
      const double2 v = piv[i];
      lg += 0.5 * log(v.x * v.x + v.y * v.y);
      an += atan2(v.y, v.x);
    }
  lg = block_sum_d(lg, s_red);
  an = block_sum_d(an, s_red);
  if (tid == 0) {
    if (singular) {
      logdet[b] = make_double2(-INFINITY, 0.0);
      sing[b] = 1;
      atomicAdd(&flags[0], 1);
    } else {
      double ang = an + ((s_swaps & 1) ? M_PI : 0.0);
      ang = remainder(ang, 2.0 * M_PI);
      logdet[b] = make_double2(lg, ang);
      sing[b] = 0;
    }
  }
  __half* o = out + (size_t)b * 4 * N * Np;
  if (singular) {
    for (int e = tid; e < N * N; e += GJB_THREADS) mixed::put4f(o + mixed::sp_at(e / N, Np, e % N), 0.f, 0.f);
    if (tid == 0) s_out[b] = 1.f;
    return;
  }
  for (int c = tid; c < N; c += GJB_THREADS) iperm[perm[c]] = c;
  float m = 0.f;
  for (int e = tid; e < N * N; e += GJB_THREADS) {
    const float4 v = a[e];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.z)));
  }
  m = block_max_f(m, s_redf);   // its barriers also publish iperm
  const float sc = mixed::pow2_scale((double)m);
  if (tid == 0) s_out[b] = sc;
  for (int e = tid; e < N * N; e += GJB_THREADS) {
    const int i = e / N, c = e % N;
    const float4 v = a[(size_t)c * N + iperm[i]];
    mixed::put4f(o + mixed::sp_at(i, Np, c), v.x * sc, v.z * sc);
  }
}

// The same inverse (or log det alone) with the matrix in shared memory, its columns spread over
// a cluster of C CTAs (C = 1 up to N = 110 here).  Per panel of GJB = 8 pivots:
//   1. the CTA that owns the panel's columns eliminates them in registers, LPR lanes per row with
//      8 / LPR of the row's entries each: per pivot a warp maximum and one more over the warps'
//      candidates pick the row, the pivot row and the row it displaces go through shared memory,
//      and every lane eliminates its own entries (INV: all rows by Gauss-Jordan; else the rows below the
//      pivot, whose multipliers stay in the eliminated column), two barriers a pivot.  A pivot is a
//      chain of about 250 dependent instructions (reciprocal, scaled row, update); several lanes per row
//      keep the loop body short enough for the instruction cache (one lane with all eight entries took 3200
//      clocks a pivot);
//   2. T - I (INV: T the panel's accumulated transform; else the multipliers, L) goes to every CTA of the
//      cluster through L2: each fetches it with all its threads, where the owner's 256 row threads storing
//      it eight times into the others' shared memory lengthened the chain that everybody waits for (N = 256,
//      64 matrices: 6.3 ms; 4.75 ms this way);
//   3. each CTA moves the affected rows of its other columns (the log det also solves the panel's 8 x 8
//      triangle for its rows of U, a column per thread) and updates the rest, c += (T - I)[:, panel]
//      c[panel rows]: a thread takes four rows of one column (Rows), consecutive threads consecutive
//      columns, so that T is a broadcast and tmp is read once per four rows (2 / 4 rows: inverse N = 256
//      4.75 / 4.65 ms, N = 108 459 / 451 us; N = 54 114 us with 2, 117 with 4; the log det is faster with
//      two: N = 256 3.19 / 3.32 ms, N = 108 261 / 263 us).
// Both are element by element, in one order, the arithmetic of the global form: INV that of gjb_ff_kernel, the
// log det that of gj_ff_kernel (one normalised multiply-add per pivot), so that both forms give the same
// bits, whichever the number of matrices selects.  (Biased accumulators, with an error of 2^-47 of a row
// maximum times a column sum instead of 2^-48 of the terms, took 217 us for the log det at N = 108 where
// these take 261, and lost one to two decimal digits on walkers near the trial, three on rows graded over six
// decades: 1e-13 became 1e-10.)
// The INV update is N^3 complex multiply-adds of 48 FP32 instructions, the panels 8 N^2 of 60: 230 us
// at 128 instructions per clock and SM for one matrix of N = 108 per SM; the log det N^3 / 3 of 60, 95 us.
constexpr size_t GC_SMEM_LIMIT = 228000;   // dynamic, beside 3.4 KB of static

struct GcLayout {
  int nloc, lda;   // columns per CTA (a multiple of GJB for C > 1), row stride in float4 (odd: columns and rows both conflict-free)
  size_t T, tmp, piv, perm, bytes;   // byte offsets
};
__host__ __device__ inline GcLayout gc_layout(int N, int C) {
  GcLayout L;
  L.nloc = C == 1 ? N : ((N + C - 1) / C + GJB - 1) / GJB * GJB;
  L.lda = L.nloc | 1;
  L.T = (size_t)N * L.lda * sizeof(float4);
  L.tmp = L.T + (size_t)N * GJB * sizeof(float4);
  L.piv = L.tmp + (size_t)GJB * L.nloc * sizeof(float4);
  L.perm = L.piv + (size_t)L.nloc * sizeof(float4);
  L.bytes = L.perm + (size_t)N * sizeof(int);
  return L;
}

struct GcPanel {          // what the owner tells every CTA about one panel
  int prow[GJB];          // pivot row of each step
  int srcp[GJB];          // row (before the panel) that ends at pivot position j0 + l
  int srcd[GJB];          // row that ends at position prow[l], where that lies below the panel
  int singular;
};

template <int C, bool INV, int GC_THREADS, int LPR>
__global__ void __launch_bounds__(GC_THREADS, 512 / GC_THREADS)
    gjc_ff_kernel(float4* Sff, int N, zc* logdet, int* sing, int* flags, __half* out, int Np, float* s_out) {
  namespace cg = cooperative_groups;
  // rows of a column that a thread updates together; in the next panel's eight columns, which everybody
  // waits for, two up to N = 128 (LPR 2), where four would leave half of the threads without any
  using Rows = std::integral_constant<int, INV && GC_THREADS == 512 ? 4 : 2>;
  using RowsNext = std::integral_constant<int, LPR == 1 ? Rows::value : 2>;
  constexpr int GC_WARPS = GC_THREADS / 32, SLOTS = GJB / LPR;   // a lane's entries: columns sub + LPR k
  extern __shared__ __align__(16) unsigned char gj_smem[];
  __shared__ GcPanel s_panel[2];
  __shared__ uint2 s_cand[2][GC_WARPS];   // a warp's pivot candidate: |value| bits, row
  __shared__ float4 s_prow[2][GJB], s_jrow[2][GJB], s_scaled[GC_WARPS][GJB];
  __shared__ int s_porig[2], s_jorig[2], s_next;
  __shared__ double2 s_red[GC_WARPS];
  __shared__ float s_redf[GC_WARPS];
  __shared__ float s_max[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = C == 1 ? 0 : (int)(blockIdx.x % C), b = blockIdx.x / C;
  const GcLayout L = gc_layout(N, C);
  const int lda = L.lda, nloc = L.nloc, c0 = rank * nloc, nc = max(0, min(nloc, N - c0));
  float4* a = reinterpret_cast<float4*>(gj_smem);
  float4* T = reinterpret_cast<float4*>(gj_smem + L.T);
  float4* tmp = reinterpret_cast<float4*>(gj_smem + L.tmp);
  float4* piv = reinterpret_cast<float4*>(gj_smem + L.piv);
  int* perm = reinterpret_cast<int*>(gj_smem + L.perm);
  const float4* g = Sff + (size_t)b * N * N + c0;
  if (nc > 0)
    for (int e = tid; e < N * nc; e += GC_THREADS) {
      const int i = e / nc, c = e - i * nc;
      a[i * lda + c] = g[(size_t)i * N + c];
    }
  for (int i = tid; i < N; i += GC_THREADS) perm[i] = i;
  int swaps = 0;   // the last thread's count
  bool singular = false;
  // the panel's row threads: LPR lanes per row
  const int rows_threads = (N * LPR + 31) & ~31, row_warps = rows_threads >> 5;
  const int ri = tid / LPR, sub = tid % LPR, group = lane & ~(LPR - 1);
  const bool row_thread = tid < rows_threads;
  float4 v[SLOTS];   // this lane's entries of the panel, kept until T may be written
  if (C > 1) cg::this_cluster().sync();   // every CTA of the cluster runs before the first remote store
  else __syncthreads();

  // ---- 1. the panel at column j0 (local column jl), by the row threads of the CTA that owns it
  auto factor = [&](int j0, int jl, int par) {
    const int jb = min(GJB, N - j0), i = ri;
    const bool active = i < N && (INV || i >= j0);
#pragma unroll
    for (int k = 0; k < SLOTS; ++k) {
      const int l = sub + LPR * k;
      v[k] = (active && l < jb) ? a[i * lda + jl + l] : ffa::czero();
    }
    int orig = i;
    bool bad = false;   // the same for all row threads
#pragma unroll 1
    for (int jj = 0; jj < jb; ++jj) {
      const int j = j0 + jj, q = jj & 1, slot = jj / LPR;
      const bool holds = sub == jj % LPR;   // this lane has the row's entry of column j
      float4 vj = v[0];
#pragma unroll
      for (int k = 1; k < SLOTS; ++k)
        if (slot == k) vj = v[k];
      const float m = fabsf(vj.x) + fabsf(vj.z);
      const bool elig = holds && active && i >= j;
      const unsigned key = (elig && !isnan(m)) ? __float_as_uint(m) : 0u;
      const unsigned wk = __reduce_max_sync(FULL, key);
      const unsigned who = __ballot_sync(FULL, elig && key == wk);   // the smallest row among equals
      if (lane == 0) s_cand[q][warp] = make_uint2(wk, (unsigned)(tid + (who ? __ffs(who) - 1 : 0)) / LPR);
      asm volatile("bar.sync 1, %0;" ::"r"(rows_threads) : "memory");
      const uint2 cand = lane < row_warps ? s_cand[q][lane] : make_uint2(0u, 0u);
      const unsigned best = __reduce_max_sync(FULL, cand.x);
      const int p = (int)__shfl_sync(FULL, cand.y, __ffs(__ballot_sync(FULL, cand.x == best)) - 1);
      if (best == 0u || best >= 0x7f800000u) {
        bad = true;
        break;
      }
      if (i == p) {
#pragma unroll
        for (int k = 0; k < SLOTS; ++k) s_prow[q][sub + LPR * k] = v[k];
        s_porig[q] = orig;
        if (holds) piv[jl + jj] = vj;
      }
      if (i == j && p != j) {
#pragma unroll
        for (int k = 0; k < SLOTS; ++k) s_jrow[q][sub + LPR * k] = v[k];
        s_jorig[q] = orig;
      }
      if (tid == 0) s_panel[par].prow[jj] = p;
      asm volatile("bar.sync 1, %0;" ::"r"(rows_threads) : "memory");
      const float4 inv = ffa::crecip(s_prow[q][jj]);
      // INV: every warp scales the pivot row for itself, one entry per lane
      if (INV && lane < GJB) s_scaled[warp][lane] = lane == jj ? inv : ffa::cmul(s_prow[q][lane], inv);
      if (p != j) {   // rows j and p trade places
        if (i == p) {
#pragma unroll
          for (int k = 0; k < SLOTS; ++k) v[k] = s_jrow[q][sub + LPR * k];
          orig = s_jorig[q];
        }
        if (i == j) {
          orig = s_porig[q];
          if (!INV) {   // its multipliers move with it (INV: the scaled row, below)
#pragma unroll
            for (int k = 0; k < SLOTS; ++k) v[k] = s_prow[q][sub + LPR * k];
          }
        }
      }
      vj = v[0];
#pragma unroll
      for (int k = 1; k < SLOTS; ++k)
        if (slot == k) vj = v[k];
      const int from = group + jj % LPR;
      float4 f = vj;
      if (LPR > 1)
        f = make_float4(__shfl_sync(FULL, vj.x, from), __shfl_sync(FULL, vj.y, from), __shfl_sync(FULL, vj.z, from),
                        __shfl_sync(FULL, vj.w, from));
      if constexpr (INV) {
        __syncwarp();
        // row i -= f (row j / pivot); column j, whose entry of the scaled row is 1 / pivot, starts
        // from zero (bit for bit -(f / pivot)), and the pivot row becomes the scaled row
#pragma unroll
        for (int k = 0; k < SLOTS; ++k) {
          const float4 t = s_scaled[warp][sub + LPR * k];
          const float4 from0 = (holds && slot == k) ? ffa::czero() : v[k];
          const float4 e = ffa::cfms(from0, f, t);
          v[k] = i == j ? t : e;
        }
        __syncwarp();
      } else if (i > j) {
        // row i -= (f / pivot) row j; the multiplier takes the place of the entry it eliminates
        const float4 mult = ffa::cmul(f, inv);
#pragma unroll
        for (int k = 0; k < SLOTS; ++k) {
          const int l = sub + LPR * k;
          if (l > jj) v[k] = ffa::cfms(v[k], mult, s_prow[q][l]);
          if (l == jj) v[k] = mult;
        }
      }
    }
    if (tid == 0) s_panel[par].singular = bad;
    if (!bad && i < N) {
#pragma unroll
      for (int k = 0; k < SLOTS; ++k) {
        const int l = sub + LPR * k;
        if constexpr (INV) {
          if (l < jb) a[i * lda + jl + l] = v[k];
          if (l >= jb) v[k] = ffa::czero();
          else if (i == j0 + l) v[k] = ffa::pack(ffa::add(ffa::re(v[k]), ffa::make(-1.f, 0.f)), ffa::im(v[k]));
        } else if (l >= jb || i <= j0 + l) {   // rows above the panel (i < j0) among them
          v[k] = ffa::czero();
        }
      }
      if (sub == 0) {
        if (i >= j0 && i < j0 + jb) s_panel[par].srcp[i - j0] = orig;
        for (int l = 0; l < jb; ++l)
          if (s_panel[par].prow[l] == i) s_panel[par].srcd[l] = orig;
      }
    }
  };
  // ---- T - I (v): into shared memory, or (C > 1) through the matrix's global copy, which nobody
  // reads after the start: eight CTAs fetch it from L2 sooner than one can store it to all of them.  Two
  // slots in turn; the row moves and the verdict go into the other CTAs' shared memory.
  auto put_T = [&](float4* dst) {
    if (ri < N) {
#pragma unroll
      for (int k = 0; k < SLOTS; ++k) dst[ri * GJB + sub + LPR * k] = v[k];
    }
  };
  float4* Tg = Sff + (size_t)b * N * N;   // [2][N][GJB], C > 1 (N > 64, so it fits)
  auto publish = [&](int par) {
    if (!s_panel[par].singular) put_T(Tg + (size_t)par * N * GJB);
    if (tid < (int)(sizeof(GcPanel) / sizeof(int))) {
      const int val = reinterpret_cast<const int*>(&s_panel[par])[tid];
      for (int r = 0; r < C; ++r)
        if (r != rank) reinterpret_cast<int*>(cg::this_cluster().map_shared_rank(&s_panel[par], r))[tid] = val;
    }
  };
  // ---- 3. rows i0 .. of local column c: += (T - I) tmp
  auto update = [&](auto rows, int j0, int ip, int c) {
    constexpr int GC_ROWS = decltype(rows)::value;
    const int jb = min(GJB, N - j0), i0 = (INV ? 0 : j0 + jb) + GC_ROWS * ip;
    float4 v[GC_ROWS];
    const float4* d[GC_ROWS];   // rows past the last repeat it and are not stored
#pragma unroll
    for (int r = 0; r < GC_ROWS; ++r) {
      const int i = min(i0 + r, N - 1);
      v[r] = a[i * lda + c];
      d[r] = T + i * GJB;
    }
    if constexpr (INV) {
      ffa::cacc x[GC_ROWS];
#pragma unroll
      for (int r = 0; r < GC_ROWS; ++r) x[r] = ffa::cacc_from(v[r]);
#pragma unroll 4
      for (int l = 0; l < jb; ++l) {
        const float4 t = tmp[l * nloc + c];
#pragma unroll
        for (int r = 0; r < GC_ROWS; ++r) ffa::cacc_fma(x[r], d[r][l], t);
      }
#pragma unroll
      for (int r = 0; r < GC_ROWS; ++r) v[r] = ffa::cacc_get(x[r]);
    } else {
#pragma unroll 4
      for (int l = 0; l < GJB; ++l) {
        const float4 t = tmp[l * nloc + c];
#pragma unroll
        for (int r = 0; r < GC_ROWS; ++r) v[r] = ffa::cfms(v[r], d[r][l], t);
      }
    }
#pragma unroll
    for (int r = 0; r < GC_ROWS; ++r)
      if (i0 + r < N) a[(i0 + r) * lda + c] = v[r];
  };

  if (rank == 0 && row_thread) {
    factor(0, 0, 0);
    asm volatile("bar.sync 1, %0;" ::"r"(rows_threads) : "memory");
    if (C > 1) publish(0);
  }
  for (int j0 = 0, pan = 0; j0 < N; j0 += GJB, ++pan) {
    const int jb = min(GJB, N - j0), par = pan & 1;
    const int owner = C == 1 ? 0 : j0 / nloc, jl = j0 - owner * nloc;   // the panel's first local column
    if (C > 1)
      cg::this_cluster().sync();
    else
      __syncthreads();   // the previous panel's T has been read for the last time
    if (s_panel[par].singular) {
      singular = true;
      break;
    }
    if (C == 1) {
      if (row_thread) put_T(T);
    } else {
      const float4* src = Tg + (size_t)par * N * GJB;
      for (int e = tid; e < N * GJB; e += GC_THREADS) T[e] = __ldcg(src + e);
    }
    if (tid == 0) s_next = 0;
    // ---- 2. the affected rows of the other columns (LU: those right of the panel): thread
    // (column, half), half 0 the panel's rows (also kept in tmp), half 1 the rows they displaced
    {
      const int first = INV ? 0 : (rank < owner ? nc : (rank == owner ? jl + jb : 0));
      const int x0 = INV && rank == owner ? jl : nc, own = INV && rank == owner ? jb : 0;
      const int half = INV ? tid & 1 : tid / (GC_THREADS / 2), c1 = first + (INV ? tid >> 1 : tid % (GC_THREADS / 2));
      const int c = c1 + (c1 >= x0 ? own : 0);
      const bool has = c < nc;
      float4 x[GJB];
#pragma unroll
      for (int l = 0; l < GJB; ++l) {
        const int src = half ? s_panel[par].srcd[l < jb ? l : 0] : s_panel[par].srcp[l < jb ? l : 0];
        const bool need = has && l < jb && (!half || s_panel[par].prow[l] >= j0 + jb);
        x[l] = need ? a[src * lda + c] : ffa::czero();
      }
      __syncthreads();   // T is complete too
      if (has && !half) {
        if (!INV) {   // the panel's rows of U (jb = GJB: only the last panel is narrower, and no column is right of it)
#pragma unroll
          for (int l = 0; l < GJB; ++l)
#pragma unroll
            for (int i = 1; i < GJB; ++i)
              if (i > l) x[i] = ffa::cfms(x[i], T[(j0 + i) * GJB + l], x[l]);
        }
#pragma unroll
        for (int l = 0; l < GJB; ++l) {
          tmp[l * nloc + c] = x[l];
          if (INV && l < jb) a[(j0 + l) * lda + c] = x[l];
        }
      } else if (has) {
#pragma unroll
        for (int l = 0; l < GJB; ++l)
          if (l < jb && s_panel[par].prow[l] >= j0 + jb) a[s_panel[par].prow[l] * lda + c] = x[l];
      }
      __syncthreads();
    }
    // ---- 3. the rank-GJB update.  The next panel's columns first; then its row threads factor it
    // while the other warps update the rest, and join them.
    const int jn = j0 + GJB, jbn = min(GJB, N - jn);
    const int nowner = jn >= N ? -1 : (C == 1 ? 0 : jn / nloc), nl = jn - nowner * nloc;
    const int below = N - (INV ? 0 : j0 + jb), np = (below + Rows::value - 1) / Rows::value;
    const bool mine = rank == nowner;
    if (mine) {
      for (int u = tid; u < (below + RowsNext::value - 1) / RowsNext::value * GJB; u += GC_THREADS)
        if ((u & (GJB - 1)) < jbn) update(RowsNext(), j0, u / GJB, nl + (u & (GJB - 1)));
      __syncthreads();
      if (row_thread) {
        const int parn = par ^ 1;
        factor(jn, nl, parn);
        if (C > 1) {
          asm volatile("bar.sync 1, %0;" ::"r"(rows_threads) : "memory");
          publish(parn);
        }
      }
      __syncwarp();
    }
    if (tid == GC_THREADS - 1)   // beside the panel's factorisation
      for (int l = 0; l < jb; ++l) {
        const int p = s_panel[par].prow[l];
        if (p != j0 + l) {
          const int t = perm[j0 + l];
          perm[j0 + l] = perm[p];
          perm[p] = t;
          ++swaps;
        }
      }
    __syncwarp();
    // the rest: columns [first, nc) without [x0, x1)
    const int first = INV ? 0 : (rank < owner ? nc : (rank == owner ? jl + jb + (mine ? jbn : 0) : (mine ? jbn : 0)));
    const int x0 = !INV ? nc : (rank == owner ? jl : (mine ? nl : nc));
    const int xn = !INV ? 0 : (rank == owner ? jb : 0) + (mine ? jbn : 0);
    const int R = max(0, nc - first - xn), total = np * R;
    for (;;) {
      int u = 0;
      if (lane == 0) u = atomicAdd(&s_next, 32);
      u = __shfl_sync(FULL, u, 0) + lane;
      if (u - lane >= total) break;
      if (u < total) {
        const int ip = u / R, c1 = first + u - ip * R;
        update(Rows(), j0, ip, c1 + (c1 >= x0 ? xn : 0));
      }
      __syncwarp();
    }
  }
  __syncthreads();
  // ---- log det from the pivots: each CTA the logarithms (one half of its threads) and the arguments (the
  // other, so that the two long FP64 sequences run side by side) of its own columns' pivots, in their place
  if (!singular) {   // the same in every thread of the cluster
    constexpr int HALF = GC_THREADS / 2;   // at least a CTA's columns
    const int c = tid % HALF;
    double z = 0.0;
    if (c < nc) {
      const double2 v = make_double2(ffa::to_double(ffa::re(piv[c])), ffa::to_double(ffa::im(piv[c])));
      z = tid < HALF ? 0.5 * log(v.x * v.x + v.y * v.y) : atan2(v.y, v.x);
    }
    __syncthreads();
    if (c < nc) reinterpret_cast<double*>(piv + c)[tid / HALF] = z;
    __syncthreads();
  }
  float m = 0.f;
  if (INV && !singular) {
    for (int e = tid; e < N * nc; e += GC_THREADS) {
      const int i = e / nc, c = e - i * nc;
      const float4 v = a[i * lda + c];
      m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.z)));
    }
    m = block_max_f(m, s_redf);
  }
  if (C > 1) {
    if (tid < C) cg::this_cluster().map_shared_rank(s_max, tid)[rank] = m;
    cg::this_cluster().sync();
    m = 0.f;
    for (int r = 0; r < C; ++r) m = fmaxf(m, s_max[r]);
  }
  // Summed by the first CTA, 32 pivots per warp, then the warps in order: the order depends on N alone, so that
  // neither the size of the cluster nor the choice of the global form (block_sum_d) shows in the result.
  double lg = 0.0, an = 0.0;
  if (rank == 0 && !singular) {
    if (tid < ((N + 31) & ~31)) {
      double2 z = make_double2(0.0, 0.0);
      if (tid < N) {
        const float4* pr = piv;
        if (C > 1) pr = cg::this_cluster().map_shared_rank(piv, tid / nloc);
        z = reinterpret_cast<const double2*>(pr)[C > 1 ? tid % nloc : tid];
      }
      for (int o = 16; o > 0; o >>= 1) {
        z.x += __shfl_xor_sync(FULL, z.x, o);
        z.y += __shfl_xor_sync(FULL, z.y, o);
      }
      if (lane == 0) s_red[warp] = z;
    }
    __syncthreads();
    for (int w = 0; w < (N + 31) / 32; ++w) {
      lg += s_red[w].x;
      an += s_red[w].y;
    }
  }
  if (rank == 0 && tid == GC_THREADS - 1) {
    if (singular) {
      logdet[b] = make_double2(-INFINITY, 0.0);
      sing[b] = 1;
      atomicAdd(&flags[0], 1);
    } else {
      const double ang = remainder(an + ((swaps & 1) ? M_PI : 0.0), 2.0 * M_PI);
      logdet[b] = make_double2(lg, ang);
      sing[b] = 0;
    }
  }
  if (C > 1 && !INV) cg::this_cluster().sync();   // the first CTA has read the others' pivots
  if (!INV) return;
  __half* o = out + (size_t)b * 4 * N * Np;
  const float sc = singular ? 1.f : mixed::pow2_scale((double)m);
  if (rank == 0 && tid == 0) s_out[b] = sc;
  // out row i, column r = S^-T[i][r] = S^-1[r][i] = a[r][iperm[i]]: local column c is row perm[c0 + c]
  for (int e = tid; e < N * nc; e += GC_THREADS) {
    const int c = e / N, r = e - c * N;
    const float4 v = singular ? ffa::czero() : a[r * lda + c];
    const int i = singular ? c0 + c : perm[c0 + c];
    mixed::put4f(o + mixed::sp_at(i, Np, r), v.x * sc, v.z * sc);
  }
  if (C > 1) cg::this_cluster().sync();
}

template <class K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return ensure_dyn_smem(reinterpret_cast<const void*>(kernel), bytes);
}

size_t gj_smem_bytes(int N) { return (size_t)N * (sizeof(float4) + sizeof(double2) + 2 * sizeof(int)); }

struct GjcArgs {
  float4* Sff;
  int WS, N;
  zc* logdet;
  int *sing, *flags;
  __half* out;
  int Np;
  float* s_out;
};

template <int C, bool INV, int THREADS, int LPR>
cudaError_t gjc_launch(const GjcArgs& g, cudaStream_t st) {
  const size_t bytes = gc_layout(g.N, C).bytes;
  auto fn = gjc_ff_kernel<C, INV, THREADS, LPR>;
  cudaError_t e = set_smem(fn, bytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)g.WS * C);
  cfg.blockDim = dim3(THREADS);
  cfg.dynamicSmemBytes = bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = C > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, fn, g.Sff, g.N, g.logdet, g.sing, g.flags, g.out, g.Np, g.s_out);
}

// CTAs per matrix: the fewest whose shared memory holds it (0: none up to 8), doubled while every
// matrix still gets its CTAs at once and a CTA keeps 32 columns.
int gjc_cluster(int WS, int N) {
  if (N > 256) return 0;
  if (N <= 64) return 1;
  int C = 1;
  while (C <= 8 && gc_layout(N, C).bytes > GC_SMEM_LIMIT) C *= 2;
  if (C > 8) return 0;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return C;
  while (C < (N <= 128 ? 4 : 8) && (long)WS * 2 * C <= sms && N >= 64 * C) C *= 2;
  return C;
}

// Whether a cluster of C CTAs per matrix beats one CTA per matrix in the global form.  Of the clusters
// only 76 / 36 / 15 (C = 2 / 4 / 8) run at once on 152 SMs, so many matrices take many waves; `gain` is
// what one wave of the global form costs in waves of clusters (a little less beyond one wave, when its
// CTAs no longer move in step).  It takes the GPU to be free; members of a group on their own streams share it, and
// then either form may be the slower one, with the same bits.  Measured, cluster | global, ms:
//   inverse  N = 256: 64 matrices 4.63 | 6.55, 128 8.33 | 7.08, 304 19.4 | 12.7, 512 32.3 | 24.2
//            N = 160: 64 1.05 | 1.84, 128 2.09 | 1.85, 512 7.80 | 6.46;  N = 120: 128 0.73 | 0.89, 512 2.58 | 2.99
//   log det  N = 256: 64 3.19 | 4.81, 128 5.75 | 7.09, 304 13.4 | 11.4, 512 22.3 | 20.4
//            N = 160: 64 0.71 | 1.30, 128 1.40 | 1.29, 512 5.22 | 4.04;  N = 120: 64 0.26 | 0.48, 128 0.50 | 0.48
bool cluster_pays(int WS, int C, bool inv, int sms) {
  const int at_once = std::max(1, sms * (C == 8 ? 15 : C == 4 ? 36 : 76) / 152);
  const int waves = (WS + at_once - 1) / at_once;
  const double gain = C == 8 ? (inv ? 7.0 : 10.0) : C == 4 ? 3.45 : (inv ? 2.3 : 1.9);
  return waves <= gain * (WS <= sms ? 1.0 : 0.97 * WS / sms);
}

// Small matrices take fewer threads, so that several share an SM (the panels are latency).
// cudaErrorNotSupported: too large for this form, or faster in the global one.
template <bool INV>
cudaError_t gjc_invert(const GjcArgs& g, cudaStream_t st) {
  const int N = g.N;
  int C = gjc_cluster(g.WS, N);
  if (C == 0) return cudaErrorNotSupported;
  if (N > 128) C = C <= 4 ? 4 : 8;
  int dev = 0, sms = 0;
  if (C > 1 && cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      !cluster_pays(g.WS, C, INV, sms))
    return cudaErrorNotSupported;
  if (N <= 32) return gjc_launch<1, INV, 128, 4>(g, st);
  if (N <= 64) return gjc_launch<1, INV, 256, 2>(g, st);
  if (N <= 128) return C == 1   ? gjc_launch<1, INV, 512, 2>(g, st)
                       : C == 2 ? gjc_launch<2, INV, 512, 2>(g, st)
                                : gjc_launch<4, INV, 512, 2>(g, st);
  return C == 4 ? gjc_launch<4, INV, 512, 1>(g, st) : gjc_launch<8, INV, 512, 1>(g, st);
}

}  // namespace

size_t overlap_scratch_bytes(int WS, int N) { return (size_t)WS * N * N * sizeof(float4); }

cudaError_t overlap(const zc* A, const zc* phi, const zc* B, float4* Sff, float2* phi_perp, unsigned long long* mx,
                    int WS, int nk, int M, int n, int N, cudaStream_t st) {
  const size_t fixed = (size_t)2 * M * n * sizeof(float4);
  size_t JC = (OV_SMEM_TARGET > fixed) ? (OV_SMEM_TARGET - fixed) / ((size_t)(M + n) * sizeof(float4)) : 1;
  JC = std::max<size_t>(1, std::min<size_t>(JC, (size_t)N));
  const size_t bytes = fixed + JC * (size_t)(M + n) * sizeof(float4);
  if (bytes > SMEM_LIMIT) return cudaErrorInvalidValue;
  const dim3 grid(WS, nk, (unsigned)((N + JC - 1) / JC));
  cudaError_t e;
  if (B) {
    if ((e = set_smem(overlap_ff_kernel<true>, bytes)) != cudaSuccess) return e;
    overlap_ff_kernel<true><<<grid, OV_THREADS, bytes, st>>>(A, phi, B, Sff, phi_perp, mx, nk, M, n, N, (int)JC);
  } else {
    if ((e = set_smem(overlap_ff_kernel<false>, bytes)) != cudaSuccess) return e;
    overlap_ff_kernel<false><<<grid, OV_THREADS, bytes, st>>>(A, phi, B, Sff, phi_perp, mx, nk, M, n, N, (int)JC);
  }
  return cudaGetLastError();
}

cudaError_t invert(float4* Sff, int WS, int N, zc* logdet, int* sing, int* flags, __half* out, int Np, float* s_out,
                   cudaStream_t st) {
  const GjcArgs g = {Sff, WS, N, logdet, sing, flags, out, Np, s_out};
  const cudaError_t ec = out ? gjc_invert<true>(g, st) : gjc_invert<false>(g, st);
  if (ec != cudaErrorNotSupported) return ec;
  cudaError_t e;
  if (out) {
    const size_t bytes = (size_t)GJB * N * sizeof(float4) + gj_smem_bytes(N);
    if (N > GJB_GLOBAL_MAXN || bytes > SMEM_LIMIT) return cudaErrorInvalidValue;
    if ((e = set_smem(gjb_ff_kernel, bytes)) != cudaSuccess) return e;
    gjb_ff_kernel<<<WS, GJB_THREADS, bytes, st>>>(Sff, N, logdet, sing, flags, out, Np, s_out);
    return cudaGetLastError();
  }
  const size_t bytes = gj_smem_bytes(N);
  if ((e = set_smem(gj_ff_kernel, bytes)) != cudaSuccess) return e;
  gj_ff_kernel<<<WS, GJ_THREADS, bytes, st>>>(Sff, N, logdet, sing, flags);
  return cudaGetLastError();
}

}  // namespace ffla
