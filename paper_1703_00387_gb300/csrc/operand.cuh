// Split operands of the tcgen05 GEMM: hi and lo of a value, and the stores of
// eight neighbouring columns of an operand row [hi(0..Kp) | lo(0..Kp)].
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "ieee.cuh"

namespace osmps {

__device__ __forceinline__ uint32_t to_tf32(float x) { return cvt_rna_tf32(x); }

// hi and lo of one value as the two halves of a word (bf16) or a pair of
// words (tf32), from float64 (integer operations, ieee.cuh) or float32.
template <int KIND>
struct SplitWord {
  using T = uint32_t;
};
template <>
struct SplitWord<TC_TF32> {
  using T = uint2;
};
template <int KIND, typename S>
__device__ __forceinline__ typename SplitWord<KIND>::T split_word(S x) {
  if constexpr (KIND == TC_BF16) {
    if constexpr (sizeof(S) == 8) return f64_to_bf16_pair(x);
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
    return (uint32_t)__bfloat16_as_ushort(h) | (uint32_t)__bfloat16_as_ushort(l) << 16;
  } else {
    if constexpr (sizeof(S) == 8) return f64_to_tf32_pair(x);
    const uint32_t h = to_tf32((float)x);
    return make_uint2(h, to_tf32((float)x - __uint_as_float(h)));
  }
}

// Eight consecutive values from a 16-byte boundary, in 16-byte loads.
__device__ __forceinline__ void load_eight(const double* p, double (&x)[8]) {
#pragma unroll
  for (int i = 0; i < 8; i += 2) {
    const double2 q = *reinterpret_cast<const double2*>(p + i);
    x[i] = q.x;
    x[i + 1] = q.y;
  }
}
__device__ __forceinline__ void load_eight(const float* p, float (&x)[8]) {
#pragma unroll
  for (int i = 0; i < 8; i += 4) {
    const float4 q = *reinterpret_cast<const float4*>(p + i);
    x[i] = q.x;
    x[i + 1] = q.y;
    x[i + 2] = q.z;
    x[i + 3] = q.w;
  }
}

// Eight consecutive columns of an operand row (off_hi a multiple of 8) in
// 16-byte stores.
__device__ __forceinline__ void store_words(void* dst, int64_t off_hi, int64_t Kp, const uint32_t (&w)[8]) {
  uint4 h, l;
  uint32_t* hp = &h.x;
  uint32_t* lp = &l.x;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    hp[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);
    lp[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
  }
  __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(dst) + off_hi;
  *reinterpret_cast<uint4*>(d) = h;
  *reinterpret_cast<uint4*>(d + Kp) = l;
}
__device__ __forceinline__ void store_words(void* dst, int64_t off_hi, int64_t Kp, const uint2 (&w)[8]) {
  uint32_t* d = reinterpret_cast<uint32_t*>(dst) + off_hi;
#pragma unroll
  for (int i = 0; i < 8; i += 4) {
    *reinterpret_cast<uint4*>(d + i) = make_uint4(w[i].x, w[i + 1].x, w[i + 2].x, w[i + 3].x);
    *reinterpret_cast<uint4*>(d + Kp + i) = make_uint4(w[i].y, w[i + 1].y, w[i + 2].y, w[i + 3].y);
  }
}

}  // namespace osmps
