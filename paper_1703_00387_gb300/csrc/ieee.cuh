// Float conversions by integer operations on the IEEE-754 bit layouts.
//
// GB300's float64 pipe issues two lanes per clock per SM, and widening a
// float to double runs there: converting every element of a 128 x 256 tile
// in a GEMM epilogue measured ~8 us per launch. (Narrowing by integer fields
// measured slower than the hardware conversion inside the fused W-step, so
// that kernel keeps the hardware one.) These helpers build the result from the
// sign, exponent and fraction fields with integer operations (the integer
// pipe is 32 times wider) for normal numbers, and leave zeros, subnormals,
// infinities, NaNs and out-of-range exponents to the hardware conversion
// (both return signed zeros themselves: they are common as padding).
// Both are exact restatements of the format's definition: widening copies
// the fraction; narrowing rounds the fraction to nearest, ties to even.
#pragma once
#include <stdint.h>

#include <cuda_bf16.h>

namespace osmps {

// (double)x, exactly.
__device__ __forceinline__ double f32_to_f64(float x) {
  const uint32_t u = __float_as_uint(x), mag = u & 0x7FFFFFFFu;
  if (mag - 0x00800000u >= 0x7F000000u && mag != 0u) return (double)x;  // subnormal, inf, nan
  const uint32_t hi = mag == 0u ? 0u : (mag >> 3) + 0x38000000u;  // exponent + 896
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(u << 29));
}

// (float)x, rounded to nearest with ties to even.
__device__ __forceinline__ float f64_to_f32_rn(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  if ((b << 1) == 0) return __uint_as_float((uint32_t)(b >> 63) << 31);  // +-0
  const int E = (int)((b >> 52) & 0x7FFu);
  const int ef = E - 896;  // float biased exponent
  if (ef < 1 || ef > 253) return (float)x;  // float subnormals, overflow, zero, inf, nan
  const uint64_t frac = b & 0xFFFFFFFFFFFFFull;
  const uint32_t keep = (uint32_t)(frac >> 29);            // 23 fraction bits kept
  const uint32_t rest = (uint32_t)(frac & 0x1FFFFFFFu);    // 29 bits dropped
  const uint32_t half = 0x10000000u;
  uint32_t mag = ((uint32_t)ef << 23) | keep;
  mag += (rest > half || (rest == half && (keep & 1u))) ? 1u : 0u;  // a carry moves into the exponent
  return __uint_as_float((uint32_t)(b >> 63) << 31 | mag);
}

// The rounded magnitude a (a > 0, leading bit p) at 2^n kept bits, n = 8 or
// 24: a 2^(n - 1 - p) to nearest-even, in [2^(n-1), 2^n].
template <int N>
__device__ __forceinline__ uint32_t round_bits(uint64_t a, int p) {
  if (p < N) return (uint32_t)(a << (N - 1 - p));
  const int s = p - (N - 1);
  return (uint32_t)((a + ((1ull << (s - 1)) - 1) + ((a >> s) & 1)) >> s);
}

// x as a bf16 pair, hi = x and lo = x - hi rounded to nearest-even, with
// integer operations: the rounded mantissa of hi, the exact difference of the
// 53-bit mantissas and its rounding. The raw bits come back as hi | lo << 16.
// Through the float64 pipe (two conversions and a subtraction per value) this
// split was what bound the operand passes: 5.2M values 41 us. Values whose hi
// or lo is not a normal bf16 number go through the hardware conversions.
__device__ __forceinline__ uint32_t f64_to_bf16_pair(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  if ((b << 1) == 0) return (uint32_t)(b >> 48) & 0x8000u;  // +-0, lo = +0
  const int E = (int)((b >> 52) & 0x7FFu);
  const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const uint32_t sign = (uint32_t)(b >> 48) & 0x8000u;
  const int ef = E - 896;  // bf16 biased exponent of hi
  const uint32_t hm = round_bits<8>(m, 52);
  const int64_t R = (int64_t)(m - ((uint64_t)hm << 45));
  const uint64_t a = (uint64_t)(R < 0 ? -R : R);
  const int p = a ? 63 - __clzll((long long)a) : 0;
  const int el = p + E - 948;  // bf16 biased exponent of lo
  if (ef < 1 || ef > 253 || (a != 0 && el < 1)) {
    const __nv_bfloat16 h = __double2bfloat16(x);
    const __nv_bfloat16 l = __double2bfloat16(x - (double)__bfloat162float(h));
    return (uint32_t)__bfloat16_as_ushort(h) | (uint32_t)__bfloat16_as_ushort(l) << 16;
  }
  const uint32_t hi = sign | (((uint32_t)ef << 7) + hm - 128u);
  if (a == 0) return hi;  // lo = +0
  const uint32_t lo = (R < 0 ? sign ^ 0x8000u : sign) | (((uint32_t)el << 7) + round_bits<8>(a, p) - 128u);
  return hi | lo << 16;
}

__device__ __forceinline__ uint32_t cvt_rna_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

// x as a tf32 pair: hi = x and lo = x - hi, each rounded to float32 (nearest
// even) and then to tf32 (ties away), the difference exact as above.
__device__ __forceinline__ uint2 f64_to_tf32_pair(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FFu);
  const uint32_t h = cvt_rna_tf32(f64_to_f32_rn(x));
  const int eh = (int)((h >> 23) & 0xFFu);  // E - 896, or one more after a carry
  const uint64_t m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const uint64_t hm = (uint64_t)((h & 0x7FFFFFu) | 0x800000u);
  const int up = eh - (E - 896);
  const int64_t R = (int64_t)(m - (hm << (29 + (up & 1))));
  const uint64_t a = (uint64_t)(R < 0 ? -R : R);
  const int p = a ? 63 - __clzll((long long)a) : 0;
  const int el = p + E - 948;  // float biased exponent of x - hi
  if ((b << 1) == 0 || E < 897 || E > 1149 || (unsigned)up > 1u || (a != 0 && el < 1))
    return make_uint2(h, cvt_rna_tf32((float)(x - (double)__uint_as_float(h))));
  if (a == 0) return make_uint2(h, 0u);
  const uint32_t sign = (uint32_t)(b >> 63) << 31;
  const uint32_t lf = (R < 0 ? sign ^ 0x80000000u : sign) | (((uint32_t)el << 23) + round_bits<24>(a, p) - 0x800000u);
  return make_uint2(h, cvt_rna_tf32(__uint_as_float(lf)));
}

}  // namespace osmps
