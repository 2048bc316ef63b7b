// fp16 hi/lo operand split shared by the tensor-core GEMM operands (tc_gemm.cuh).
//
// A matrix enters a GEMM as four fp16 planes (hi and lo of the real and imaginary parts) of x*s, with
// s a power of two chosen per matrix so that the largest |x*s| sits near SCALE_TARGET: far from the
// fp16 overflow, and high enough that lo keeps its full 11 bits.
#pragma once

#include <cuda_fp16.h>


namespace mixed {

constexpr float SCALE_TARGET = 4096.f;

// The largest power of two s with maxabs * s <= SCALE_TARGET, its exponent kept within +-100; 1 for
// zero, infinities and NaN.  From the bits: a division per thread would run on the FP64 pipe.
__device__ __forceinline__ float pow2_scale(double maxabs) {
  constexpr int TARGET_EXP = 12;
  static_assert(SCALE_TARGET == (float)(1 << TARGET_EXP), "a power of two");
  const unsigned hi = (unsigned)__double2hiint(maxabs), lo = (unsigned)__double2loint(maxabs);
  const int eb = (int)(hi >> 20);   // sign and exponent
  if (eb >= 0x7ff || !(hi | lo)) return 1.f;   // negative values do not occur
  int e = TARGET_EXP - (eb - 1023) - (((hi & 0xfffffu) | lo) ? 1 : 0);
  e = max(-100, min(100, e));
  return __uint_as_float((unsigned)(e + 127) << 23);
}

// x*s split into hi = fp16(x*s) and lo = fp16(x*s - hi), in fp32 (s is a power of two, so
// x*s is exact; x*s - hi is exact in fp32).  FP64 arithmetic is avoided on purpose: the
// FP64 pipe of this GPU is about 60x slower than FP32.
__device__ __forceinline__ void split_val(float xs, __half& hi, __half& lo) {
  hi = __float2half_rn(xs);
  lo = __float2half_rn(xs - __half2float(hi));
}
// Layout of a split matrix of `rows` rows (all matrices of a batch one after another) and `ld`
// columns, ld a multiple of 32: every row in blocks of 32 columns, a block holding its four
// planes one after another (re hi, im hi, re lo, im lo; 64 bytes each), so that the four planes
// of an element lie in one 256-byte block: a producer's stores of a run of columns and a TMA
// box's rows stay in neighbouring lines and in one memory page, where planes of whole matrices
// would be scattered over four.
constexpr int SP_PLANE = 32;
enum : int { SP_RE_HI = 0, SP_IM_HI = SP_PLANE, SP_RE_LO = 2 * SP_PLANE, SP_IM_LO = 3 * SP_PLANE };
// index of (row, col) in the re hi plane
__host__ __device__ __forceinline__ size_t sp_at(size_t row, int ld, int col) {
  return row * (size_t)(4 * ld) + (size_t)((col >> 5) * 128 + (col & 31));
}
// one element at `o` = base + sp_at(row, ld, col), already scaled
__device__ __forceinline__ void put4f(__half* o, float re, float im) {
  __half h, l;
  split_val(re, h, l);
  o[SP_RE_HI] = h;
  o[SP_RE_LO] = l;
  split_val(im, h, l);
  o[SP_IM_HI] = h;
  o[SP_IM_LO] = l;
}
// x * s of two neighbours as fp16 hi and lo pairs (split_val on both, packed conversions)
__device__ __forceinline__ void split_pair(float x0, float x1, __half2& hi, __half2& lo) {
  hi = __floats2half2_rn(x0, x1);
  const float2 h = __half22float2(hi);
  lo = __floats2half2_rn(x0 - h.x, x1 - h.y);
}
// two elements of one row at even column: one 32-bit store per plane
__device__ __forceinline__ void put4f_pair(__half* o, float re0, float im0, float re1, float im1) {
  __half2 hi, lo;
  split_pair(re0, re1, hi, lo);
  *reinterpret_cast<__half2*>(o + SP_RE_HI) = hi;
  *reinterpret_cast<__half2*>(o + SP_RE_LO) = lo;
  split_pair(im0, im1, hi, lo);
  *reinterpret_cast<__half2*>(o + SP_IM_HI) = hi;
  *reinterpret_cast<__half2*>(o + SP_IM_LO) = lo;
}
}  // namespace mixed
