// Numbers exchanged between the blocks of one launch (all co-resident) without
// a barrier: a 16-byte word holds a float64 value and a 64-bit tag, written
// and read by single 128-bit accesses, and a reader polls until the word
// carries the tag it waits for. The value needs no other ordering. Polls give
// up after limit_ns of wall time (%globaltimer).
#pragma once
#include <stdint.h>

namespace osmps {

constexpr uint64_t TAGGED_LIMIT_NS = 2000000000ull;

__device__ __forceinline__ uint64_t global_timer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void put_word(ulonglong2* p, double v, uint64_t tag) {
  asm volatile("{\n .reg .b128 w;\n mov.b128 w, {%1, %2};\n st.relaxed.gpu.global.b128 [%0], w;\n}\n" ::"l"(p),
               "l"((unsigned long long)__double_as_longlong(v)), "l"((unsigned long long)tag)
               : "memory");
}

__device__ __forceinline__ ulonglong2 look_word(const ulonglong2* p) {
  ulonglong2 w;
  asm volatile("{\n .reg .b128 w;\n ld.relaxed.gpu.global.b128 w, [%2];\n mov.b128 {%0, %1}, w;\n}\n"
               : "=l"(w.x), "=l"(w.y)
               : "l"(p)
               : "memory");
  return w;
}

// v[i] = the value of word p[i] once it carries the tag (0 where p[i] is null),
// all words in flight together; false when the wait ran out.
template <int N>
__device__ __forceinline__ bool get_words(const ulonglong2* const (&p)[N], uint64_t tag, double (&v)[N],
                                          uint64_t limit_ns = TAGGED_LIMIT_NS) {
  unsigned need = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    v[i] = 0.0;
    if (p[i]) need |= 1u << i;
  }
  uint64_t t0 = 0;
  for (unsigned it = 0; need != 0; ++it) {
    ulonglong2 w[N];
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (need & (1u << i)) w[i] = look_word(p[i]);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if ((need & (1u << i)) && w[i].y == tag) {
        v[i] = __longlong_as_double((long long)w[i].x);
        need &= ~(1u << i);
      }
    if ((it & 63u) == 63u && need != 0) {
      const uint64_t now = global_timer();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return false;
    }
  }
  return true;
}

}  // namespace osmps
