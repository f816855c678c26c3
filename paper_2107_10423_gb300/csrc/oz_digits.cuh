// Digits of FP64 values (oz_gemm.cu): scales, fixed-point integers and their balanced base-256 digits.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cstdint>

#include "oz_gemm.cuh"

namespace gw {
namespace oz {

constexpr int S = OZ_S;

__device__ __forceinline__ unsigned long long mag(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}

// Power of two from the largest magnitude's bits: 2^e with |x| <= 2^e (the next power), exponents kept inside
// [-900, 900] so that products of scales stay finite; NaN if the row holds a NaN or an infinity.
__device__ __forceinline__ double scale_of(unsigned long long mx) {
  if (mx >= 0x7ff0000000000000ull) return __longlong_as_double(0x7ff8000000000000ll);
  int e = (int)(mx >> 52) - 1022;                 // 2^e > |x|
  if (mx == 0) e = 0;
  if (e < -900) e = -900;
  if (e > 900) return __longlong_as_double(0x7ff8000000000000ll);
  return __longlong_as_double((long long)(1023 + e) << 52);
}

// 63-bit integer of x scaled by 2^(62 - e), rounded to nearest (ties away), for |x| <= 2^e; pure integer arithmetic
// (the FP64 pipe runs at 1/64 of the integer one).
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = bits & 0xfffffffffffffull;
  if (be) m |= 1ull << 52;
  const int sh = (be ? be : 1) - 1075 + 62 - e;        // value = m 2^(be - 1075)
  unsigned long long v;
  if (sh >= 0) v = sh < 11 ? m << sh : 0ull;           // |x| <= 2^e keeps sh <= 10
  else v = sh > -55 ? (m + (1ull << (-sh - 1))) >> (-sh) : 0ull;
  return (bits >> 63) ? -(long long)v : (long long)v;
}

__device__ __forceinline__ int scale_exp(double sc) {   // sc is a power of two (or NaN: any exponent will do)
  return (int)((__double_as_longlong(sc) >> 52) & 0x7ff) - 1023;
}

// Digits of eight consecutive elements: out[i] = the eight BF16 of digit i.
__device__ __forceinline__ void digits8(const long long (&x)[8], uint4 (&out)[S]) {
  uint32_t w[S][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    unsigned long long y[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) y[t] = (unsigned long long)x[2 * p + t] + 0x0080808080808080ull;
#pragma unroll
    for (int i = 0; i < S; ++i) {                      // digit 0 is the top byte (signed), the others byte - 128
      float f[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const uint32_t byte = (uint32_t)(y[t] >> (8 * (S - 1 - i))) & 0xffu;
        f[t] = i == 0 ? __uint_as_float(0x4b000000u | (byte ^ 0x80u)) - 8388736.f
                      : __uint_as_float(0x4b000000u | byte) - 8388736.f;
      }
      __nv_bfloat162 v = __floats2bfloat162_rn(f[0], f[1]);
      w[i][p] = *reinterpret_cast<uint32_t*>(&v);
    }
  }
#pragma unroll
  for (int i = 0; i < S; ++i) out[i] = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
}

// Digits of eight values at the scale sc: digit i to out + i * dstride (16 bytes each).
__device__ __forceinline__ void store8(const double (&v)[8], double sc, __nv_bfloat16* out, long dstride) {
  const int e = scale_exp(sc);
  long long f[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) f[t] = to_fixed(v[t], e);
  uint4 d[S];
  digits8(f, d);
#pragma unroll
  for (int i = 0; i < S; ++i) *reinterpret_cast<uint4*>(out + i * dstride) = d[i];
}

}  // namespace oz
}  // namespace gw
