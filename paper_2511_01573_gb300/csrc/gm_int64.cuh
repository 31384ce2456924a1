// gm_int64.cuh -- 64-bit fixed-point arithmetic on the integer pipes, used in
// place of FP64 instructions: on GB300 an FP64 instruction takes ~76 cycles of
// an SM quarter (1.68 lanes per clock and SM, measured), a 32 x 32 -> 64 bit
// multiply-add 4 and an integer add or shift 1 to 2.
#pragma once

#include <cuda_runtime.h>

namespace gmq {

typedef unsigned long long u64;
typedef long long i64;

__device__ __forceinline__ u64 wide_mul(unsigned a, unsigned b) { return (u64)a * b; }

// acc + a b in one instruction.  Where the compiler knows more about a or b than
// that they are 32-bit integers it makes more of (i64)a * b: with it, the
// Gauss-Kronrod rows went from 427 to 156 multiply-add instructions, the class-5
// products above d = 8 (d = 12, Gaussian) from 289 to 227 us.
__device__ __forceinline__ void mad_wide(i64& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// round(x 2^q) for |x| < 2^(63 - q), modulo 2^64 for |x| < 2^(68 - q), by integer
// operations
__device__ __forceinline__ i64 to_fixed(double x, int q) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  const i64 m = ((i64)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  const int sh = e - 1075 + q;
  const i64 v = sh >= 0 ? m << (sh & 15) : (sh > -56 ? ((m >> (-sh - 1)) + 1) >> 1 : 0);
  return hi < 0 ? -v : v;
}

// Upper 64 bits of a^2 and a b, up to two units below the exact ones.
__device__ __forceinline__ u64 fixed_sqr(u64 a) {
  const unsigned h = (unsigned)(a >> 32), l = (unsigned)a;
  return wide_mul(h, h) + (wide_mul(h, l) >> 31);
}
__device__ __forceinline__ u64 fixed_mul(u64 a, u64 b) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
  return wide_mul(ah, bh) + (wide_mul(ah, bl) >> 32) + (wide_mul(al, bh) >> 32);
}

// The same for a signed a and 0 <= b < 2^63.
__device__ __forceinline__ i64 fixed_mul_signed(i64 a, u64 b) {
  const int ah = (int)(a >> 32), bh = (int)(b >> 32);
  const unsigned al = (unsigned)a, bl = (unsigned)b;
  return (i64)ah * bh + (((i64)ah * (int)(bl >> 1)) >> 31) + (i64)(wide_mul(al, (unsigned)bh) >> 32);
}

// |x| in FP32 by integer operations, rounded towards zero; 0 below 2^-126, infinity
// above FP32's range and for NaN.
__device__ __forceinline__ float abs_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, e = hi >> 20;
  const unsigned b = ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) |
                     ((unsigned)__double2loint(x) >> 29);
  return __uint_as_float(e < 897u ? 0u : (e < 1151u ? b : 0x7f800000u));
}

// v 2^-q rounded to nearest (ties away from zero), for q < 1000
__device__ __forceinline__ double fixed_to_double(i64 v, int q) {
  if (v == 0) return 0.0;
  const u64 a = (u64)(v < 0 ? -v : v);
  const int lz = __clzll((i64)a);
  const u64 m = (a << lz) >> 10;  // 54 bits, the leading one at 2^53
  const u64 bits = ((u64)(1023 + 62 - lz - q) << 52) + ((m + 1) >> 1);  // the leading one adds 1
  return __longlong_as_double((i64)(bits | ((u64)v & 0x8000000000000000ull)));
}

}  // namespace gmq
