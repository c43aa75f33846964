// Operand preparation and MPO contraction steps.
//
// * split_operand: float64/float32 -> [hi | lo] rows in bf16 or tf32 for the
//   tensor-core GEMM (x = hi + lo + O(2^-17 |x|) for bf16, O(2^-22 |x|) for tf32).
//   Rows are written K-major; a source whose K index is not contiguous is read
//   through a shared-memory transpose so both sides stay coalesced.
// * fiber contractions: the W-steps of Sec. 3.4, where the MPO tensors
//   M^[k] (few entries, Eq. MPOdef) act on the small (w, s) index pair of an
//   intermediate, for every (outer, inner) fiber. These are bandwidth-bound:
//   one coalesced pass over the input and the output, summing only over the
//   nonzero MPO entries while every input is finite.
#include <cuda_bf16.h>

#include "common.cuh"
#include "operand.cuh"

namespace osmps {

namespace {

// The hi / lo split of a float32 value (x - hi is exact in float32: hi keeps
// the leading bits of x), equal bit for bit to that of the same value as
// float64.
template <int KIND>
__device__ __forceinline__ void split_store_f32(void* dst, int64_t off_hi, int64_t Kp, float x) {
  if (KIND == TC_BF16) {
    const __nv_bfloat16 h = __float2bfloat16_rn(x);
    const __nv_bfloat16 l = __float2bfloat16_rn(x - __bfloat162float(h));
    reinterpret_cast<__nv_bfloat16*>(dst)[off_hi] = h;
    reinterpret_cast<__nv_bfloat16*>(dst)[off_hi + Kp] = l;
  } else {
    const uint32_t h = to_tf32(x);
    const uint32_t l = to_tf32(x - __uint_as_float(h));
    reinterpret_cast<uint32_t*>(dst)[off_hi] = h;
    reinterpret_cast<uint32_t*>(dst)[off_hi + Kp] = l;
  }
}

// Two consecutive values (off_hi even, so the pair is 4- or 8-byte aligned).
template <int KIND>
__device__ __forceinline__ void split_store2_f32(void* dst, int64_t off_hi, int64_t Kp, float a, float b) {
  if (KIND == TC_BF16) {
    const __nv_bfloat16 ha = __float2bfloat16_rn(a), hb = __float2bfloat16_rn(b);
    const __nv_bfloat16 la = __float2bfloat16_rn(a - __bfloat162float(ha));
    const __nv_bfloat16 lb = __float2bfloat16_rn(b - __bfloat162float(hb));
    __nv_bfloat162 h2, l2;
    h2.x = ha; h2.y = hb;
    l2.x = la; l2.y = lb;
    *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(dst) + off_hi) = h2;
    *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(dst) + off_hi + Kp) = l2;
  } else {
    const uint32_t ha = to_tf32(a), hb = to_tf32(b);
    const uint32_t la = to_tf32(a - __uint_as_float(ha)), lb = to_tf32(b - __uint_as_float(hb));
    *reinterpret_cast<uint2*>(reinterpret_cast<uint32_t*>(dst) + off_hi) = make_uint2(ha, hb);
    *reinterpret_cast<uint2*>(reinterpret_cast<uint32_t*>(dst) + off_hi + Kp) = make_uint2(la, lb);
  }
}

// K contiguous in the source: a thread per eight columns of a row, read in
// 16-byte loads where every row starts on such a boundary (vec).
template <int KIND, typename S>
__global__ void __launch_bounds__(256) k_split_direct(SplitView v, void* __restrict__ dst, int64_t Kp,
                                                      FastDiv by_k8, FastDiv by_n1, int vec, int wide) {
  const int64_t k8 = Kp / 8, total = v.rows * k8;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = wide ? e / k8 : (int64_t)by_k8((uint32_t)e), k = (e - r * k8) * 8;
    const int64_t r0 = wide ? r / v.n1 : (int64_t)by_n1((uint32_t)r), r1 = r - r0 * v.n1;
    const S* p = reinterpret_cast<const S*>(v.src) + r0 * v.s0 + r1 * v.s1 + k * v.sk;
    S x[8];
    if (vec && k + 8 <= v.K) {
      load_eight(p, x);
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = k + i < v.K ? p[i * v.sk] : (S)0;
    }
    typename SplitWord<KIND>::T w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = split_word<KIND, S>(x[i]);
    store_words(dst, r * 2 * Kp + k, Kp, w);
  }
}

// K strided in the source, rows close together: tiles of 64 rows x 64 columns,
// read along the rows (512 bytes a time, sixteen loads in flight per thread),
// split, and written along the columns through shared memory.
template <int KIND, typename S>
__global__ void __launch_bounds__(256) k_split_transpose(SplitView v, void* __restrict__ dst, int64_t Kp) {
  using W = typename SplitWord<KIND>::T;
  __shared__ W tile[64][65];
  const int64_t r_base = (int64_t)blockIdx.x * 64, k_base = (int64_t)blockIdx.y * 64;
  {
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int64_t r = r_base + tx, rr = r < v.rows ? r : 0;
    const int64_t r0 = rr / v.n1, r1 = rr - r0 * v.n1;
    const S* p = reinterpret_cast<const S*>(v.src) + r0 * v.s0 + r1 * v.s1 + (k_base + ty) * v.sk;
    S x[16];
#pragma unroll
    for (int j = 0; j < 16; ++j)
      x[j] = (r < v.rows && k_base + ty + 4 * j < v.K) ? p[4 * j * v.sk] : (S)0;
#pragma unroll
    for (int j = 0; j < 16; ++j) tile[ty + 4 * j][tx] = split_word<KIND, S>(x[j]);
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 512; u += 256) {
    const int row = u >> 3, g = 8 * (u & 7);
    if (r_base + row >= v.rows) continue;
    W w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = tile[g + i][row];
    store_words(dst, (r_base + row) * 2 * Kp + k_base + g, Kp, w);
  }
}

int grid_for(int64_t n, int threads) {
  int64_t b = cdiv(n, threads);
  if (b < 1) b = 1;
  if (b > 65536) b = 65536;
  return (int)b;
}

// One nonzero entry of a W-step matrix: value, input index, and whether the
// value is 1 (a comparison of float64 values runs on the float64 pipe).
template <typename T>
struct WTerm {
  T v;
  short i, one;
};

// The nonzero entries of a P x Q W-step matrix by output: output o's terms
// are terms[ptr[o] .. ptr[o + 1]), inputs ascending. MPO tensors are an
// identity in two corners and a few local operators (12 of 100 entries for
// XXZ, 4% for AKLT), so the table holds WT_CAP entries; a matrix with more of
// them is read entry by entry instead (dense).
constexpr int WT_CAP = 640;
constexpr int WT_QMAX = 64;
// how outputs are summed: from the terms; over the matrix, nonzero entries; over
// the matrix, all entries (note_top)
constexpr int W_TERMS = 0, W_NONZERO = 1, W_ALL = 2;
template <typename T>
struct WTable {
  WTerm<T> terms[WT_CAP];
  int ptr[WT_QMAX + 1];
  const double* Mat;
  int P, Q;
  int dense;
};

// V fibers of one thread.
template <typename T, int V>
struct alignas(sizeof(T) * V) Pack {
  T a[V];
};

// The largest magnitude met so far, as (upper) float bits. Where a fiber's
// inputs are below 2^63 in float32 or 2^511 in float64 and the MPO entries
// below 2^50, all that a W-step and the one fused behind it sum is finite (at
// most 2^11 terms each) and zero entries can be left out. Else (one comparison
// for all values that a thread loads) it marks the block's tables W_ALL before
// the barrier that precedes the sums, and zero entries are summed like the
// others, because 0 x Inf = NaN has to reach every output. Finite sums have the
// same bits either way, so sums of earlier fibers may still be running. (A vote
// at that barrier instead of the mark: left update at chi = 1024 239.7 us, with
// the mark 238.2.)
template <typename T, int V>
__device__ __forceinline__ void note_top(int& top, const Pack<T, V>& x) {
#pragma unroll
  for (int v = 0; v < V; ++v) {
    if constexpr (sizeof(T) == 8) top = max(top, __double2hiint(x.a[v]) & 0x7FFFFFFF);
    else top = max(top, __float_as_int(x.a[v]) & 0x7FFFFFFF);
  }
}
template <typename T>
__device__ __forceinline__ bool wild(int top) {
  return top >= (sizeof(T) == 8 ? 0x5FE00000 : 0x5F000000);
}
__device__ __forceinline__ bool wild_entry(double m) { return (__double2hiint(m) & 0x7FFFFFFF) >= 0x43100000; }

// Fill NT tables. Every thread of the block calls it (whole warps): a warp
// per output, lanes over the inputs, the nonzero ones compacted by ballots.
// Ends with a barrier. Threads that met wild values, in their inputs (top) or in
// the tables, mark them.
template <int NT, typename T>
__device__ __forceinline__ void gather_terms(int top, const double* const (&Mat)[NT], const int (&P)[NT],
                                             const int (&Q)[NT], WTable<T>* const (&tab)[NT]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  bool all = wild<T>(top);
#pragma unroll
  for (int k = 0; k < NT; ++k)
    for (int o = warp; o < Q[k]; o += warps) {
      int n = 0;
      for (int i0 = 0; i0 < P[k]; i0 += 32) {
        const double m = i0 + lane < P[k] ? Mat[k][(i0 + lane) * Q[k] + o] : 0.0;
        n += __popc(__ballot_sync(0xffffffffu, m != 0.0));
        all |= wild_entry(m);
      }
      if (lane == 0) tab[k]->ptr[o + 1] = n;
    }
  __syncthreads();
  if (lane == 0 && warp < NT) {
    WTable<T>& w = *tab[warp];
    const int q1 = Q[warp < NT ? warp : 0];
    w.ptr[0] = 0;
    for (int q = 0; q < q1; ++q) w.ptr[q + 1] += w.ptr[q];
    w.Mat = Mat[warp < NT ? warp : 0];
    w.P = P[warp < NT ? warp : 0];
    w.Q = q1;
    w.dense = w.ptr[q1] > WT_CAP || w.P > 32767 ? W_NONZERO : W_TERMS;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < NT; ++k)
    if (tab[k]->ptr[Q[k]] <= WT_CAP && P[k] <= 32767)
      for (int o = warp; o < Q[k]; o += warps) {
        int n = tab[k]->ptr[o];
        for (int i0 = 0; i0 < P[k]; i0 += 32) {
          const double m = i0 + lane < P[k] ? Mat[k][(i0 + lane) * Q[k] + o] : 0.0;
          const unsigned nz = __ballot_sync(0xffffffffu, m != 0.0);
          if (m != 0.0)
            tab[k]->terms[n + __popc(nz & ((1u << lane) - 1u))] = WTerm<T>{(T)m, (short)(i0 + lane), (short)(m == 1.0)};
          n += __popc(nz);
        }
      }
  if (all)
    for (int k = 0; k < NT; ++k) tab[k]->dense = W_ALL;
  __syncthreads();
}

// Output o of a W-step: sum over its nonzero entries of v x_i, inputs in
// ascending order; x_i is at xs[i stride]. A first entry of 1 is taken over
// as it is in float64, whose pipe is the narrow one.
template <typename T, int V>
__device__ __forceinline__ Pack<T, V> sum_terms(const WTable<T>& w, int o,
                                                const Pack<T, V>* __restrict__ xs, int64_t stride) {
  Pack<T, V> acc;
#pragma unroll
  for (int v = 0; v < V; ++v) acc.a[v] = (T)0;
  const auto add = [&](T m, const Pack<T, V>& x) {
#pragma unroll
    for (int v = 0; v < V; ++v) acc.a[v] = fma(m, x.a[v], acc.a[v]);
  };
  if (w.dense) {
    for (int i = 0; i < w.P; ++i) {
      const T m = (T)w.Mat[i * w.Q + o];
      if (w.dense == W_ALL || m != (T)0) add(m, xs[i * stride]);
    }
    return acc;
  }
  int t = w.ptr[o];
  const int t1 = w.ptr[o + 1];
  if (sizeof(T) == 8 && t < t1 && w.terms[t].one) acc = xs[w.terms[t++].i * stride];
#pragma unroll 2
  for (; t < t1; ++t) {
    const WTerm<T> e = w.terms[t];
    add(e.v, xs[e.i * stride]);
  }
  return acc;
}

// V consecutive values of a split-operand row (off_hi a multiple of V).
template <int KIND, int V>
__device__ __forceinline__ void split_store_pack(void* dst, int64_t off_hi, int64_t Kp,
                                                 const float (&x)[V]) {
  if (KIND == TC_BF16) {
    Pack<__nv_bfloat16, V> h, l;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      h.a[v] = __float2bfloat16_rn(x[v]);
      l.a[v] = __float2bfloat16_rn(x[v] - __bfloat162float(h.a[v]));
    }
    __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(dst) + off_hi;
    *reinterpret_cast<Pack<__nv_bfloat16, V>*>(d) = h;
    *reinterpret_cast<Pack<__nv_bfloat16, V>*>(d + Kp) = l;
  } else {
    Pack<uint32_t, V> h, l;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      h.a[v] = to_tf32(x[v]);
      l.a[v] = to_tf32(x[v] - __uint_as_float(h.a[v]));
    }
    uint32_t* d = reinterpret_cast<uint32_t*>(dst) + off_hi;
    *reinterpret_cast<Pack<uint32_t, V>*>(d) = h;
    *reinterpret_cast<Pack<uint32_t, V>*>(d + Kp) = l;
  }
}

// The V fibers of a thread in memory. PACKED: neighbours, one 16-byte access
// (every stride and address allows it). Otherwise fibers 32 apart, so that a
// warp's V scalar accesses are each coalesced. at[]: element offsets of the
// fibers, ok[]: false past the last fiber (such lanes read a valid fiber and
// store nothing).
template <typename T, int V, bool PACKED>
struct Fibers {
  static constexpr int N = PACKED ? 1 : V;
  int64_t at[N];
  bool ok[N];
  __device__ __forceinline__ Pack<T, V> load(const T* in, int64_t off) const {
    if (PACKED) return *reinterpret_cast<const Pack<T, V>*>(in + at[0] + off);
    Pack<T, V> p;
#pragma unroll
    for (int v = 0; v < V; ++v) p.a[v] = in[at[PACKED ? 0 : v] + off];
    return p;
  }
  // MODE 0: to out[base + off]; 1 / 2: to the bf16 / tf32 split operand
  template <int MODE>
  __device__ __forceinline__ void store(T* out, void* sdst, const int64_t (&base)[N], int64_t off,
                                        int64_t Kp, const Pack<T, V>& x) const {
    constexpr int KIND = MODE == 1 ? TC_BF16 : TC_TF32;
    if (PACKED) {
      if (!ok[0]) return;
      if (MODE == 0) {
        *reinterpret_cast<Pack<T, V>*>(out + base[0] + off) = x;
      } else {
        float f[V];
#pragma unroll
        for (int v = 0; v < V; ++v) f[v] = (float)x.a[v];
        split_store_pack<KIND, V>(sdst, base[0] + off, Kp, f);
      }
    } else {
#pragma unroll
      for (int v = 0; v < V; ++v)
        if (ok[PACKED ? 0 : v]) {
          if (MODE == 0) out[base[PACKED ? 0 : v] + off] = x.a[v];
          else split_store_f32<KIND>(sdst, base[PACKED ? 0 : v] + off, Kp, (float)x.a[v]);
        }
    }
  }
};

// n / d with d's reciprocal in f while n < 2^31 (wide: beyond that).
__device__ __forceinline__ int64_t div_by(const FastDiv& f, int64_t n, int64_t d, int wide) {
  return wide ? n / d : (int64_t)f((uint32_t)n);
}

// One W-step. A block takes 32 V fibers (o1, o2, c), V to a lane, and its
// eight warps share the work of each: first the P input rows to load into
// shared memory, then the Q outputs to sum from there. Loops over all P x Q
// entries with a thread per fiber had made this pass bound by its
// multiply-adds (P = Q = 10, 381x500 fibers, float64: 60 us, now 16).
// MODE 0: plain output, 1 / 2: split bf16 / tf32.
constexpr int FIB_WARPS = 8;
template <typename T, int MODE, int V, bool PACKED>
__global__ void __launch_bounds__(32 * FIB_WARPS)
    k_fiber(Fiber f, const double* __restrict__ Mat, const T* __restrict__ in, T* __restrict__ out,
            void* __restrict__ sdst, int64_t Kcols, int64_t Kp, int staged, FastDiv by_nc,
            FastDiv by_o2, int wide) {
  extern __shared__ __align__(16) uint8_t fsm[];
  __shared__ WTable<T> tab;
  using F = Fibers<T, V, PACKED>;
  const int P = (int)f.P, Q = (int)f.Q;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Pack<T, V>* xs = reinterpret_cast<Pack<T, V>*>(fsm) + lane;
  bool first = true;  // the table is built while the first fibers' inputs arrive
  const int64_t nc = PACKED ? f.nc / V : f.nc, total = f.n_o1 * f.n_o2 * nc;
  for (int64_t e0 = (int64_t)blockIdx.x * (32 * F::N); e0 < total; e0 += (int64_t)gridDim.x * (32 * F::N)) {
    F fib;
    int64_t ob[F::N];
#pragma unroll
    for (int v = 0; v < F::N; ++v) {
      const int64_t ev = e0 + 32 * v + lane, e = ev < total ? ev : e0;
      const int64_t o12 = div_by(by_nc, e, nc, wide), o1 = div_by(by_o2, o12, f.n_o2, wide);
      const int64_t c = (e - o12 * nc) * (PACKED ? V : 1), o2 = o12 - o1 * f.n_o2;
      fib.ok[v] = ev < total;
      fib.at[v] = o1 * f.is1 + o2 * f.is2 + c;
      ob[v] = o1 * f.os1 + o2 * f.os2 + c;
    }
    int top = 0;
#pragma unroll 4
    for (int i = warp; i < P; i += FIB_WARPS) {
      const Pack<T, V> x = fib.load(in, (int64_t)i * f.istride);
      if (staged) xs[i * 32] = x;
      note_top<T, V>(top, x);
    }
    if (first) {
      gather_terms<1, T>(top, {Mat}, {P}, {Q}, {&tab});
    } else {
      if (wild<T>(top)) tab.dense = W_ALL;  // from here on
      __syncthreads();
    }
    first = false;
    for (int o = warp; o < Q; o += FIB_WARPS) {
      Pack<T, V> acc;
      if (staged) {
        acc = sum_terms<T, V>(tab, o, xs, 32);
      } else {  // read where they are used
#pragma unroll
        for (int v = 0; v < V; ++v) acc.a[v] = (T)0;
        for (int i = 0; i < P; ++i) {
          const T m = (T)Mat[i * Q + o];
          if (tab.dense != W_ALL && m == (T)0) continue;
          const Pack<T, V> x = fib.load(in, (int64_t)i * f.istride);
#pragma unroll
          for (int v = 0; v < V; ++v) acc.a[v] = fma(m, x.a[v], acc.a[v]);
        }
      }
      const int64_t off = (int64_t)o * f.ostride;
      if (MODE == 0) {
        fib.template store<MODE>(out, sdst, ob, off, Kp, acc);
      } else {
        int64_t sb[F::N];
#pragma unroll
        for (int v = 0; v < F::N; ++v) {
          const int64_t row = (ob[v] + off) / Kcols;
          sb[v] = row * 2 * Kp + (ob[v] + off - row * Kcols);
        }
        fib.template store<MODE>(out, sdst, sb, 0, Kp, acc);
      }
    }
    if (staged) __syncthreads();  // the next fibers' inputs overwrite these
  }
}

// 16-byte packs of neighbouring fibers: every stride and address allows them.
template <typename T>
bool packs(std::initializer_list<int64_t> strides, std::initializer_list<const void*> ptrs) {
  constexpr int V = 16 / sizeof(T);
  for (int64_t x : strides)
    if (x % V != 0) return false;
  for (const void* p : ptrs)
    if ((reinterpret_cast<uintptr_t>(p) & 15) != 0) return false;
  return true;
}

// Blocks of a W-step kernel: as many as share the SMs (sm bytes of shared
// memory each), so that each builds its term table once.
int wstep_blocks(int64_t groups, size_t sm) {
  const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(2048 / (32 * FIB_WARPS), 225 * 1024 / (int64_t)sm));
  return (int)std::max<int64_t>(1, std::min<int64_t>(groups, 152 * per_sm));
}

template <typename T, int MODE>
osmps_status fiber_dispatch(const Fiber& f, const double* Mat, const T* in, T* out, void* sdst,
                            int64_t Kcols, int64_t Kp, cudaStream_t s) {
  if (f.P <= 0 || f.Q <= 0 || f.nc <= 0 || f.n_o1 <= 0 || f.n_o2 <= 0) return OSMPS_OK;
  if ((size_t)f.P * f.Q * sizeof(T) > 96 * 1024)
    return set_error(OSMPS_EUNSUPPORTED, "W-step: MPO block %lld x %lld too large",
                     (long long)f.P, (long long)f.Q);
  if (f.Q > WT_QMAX)
    return set_error(OSMPS_EUNSUPPORTED, "W-step: output block %lld > 64", (long long)f.Q);
  const auto launch = [&](auto k, int V, bool packed) -> osmps_status {
    const int64_t nc = packed ? f.nc / V : f.nc, total = f.n_o1 * f.n_o2 * nc;
    // the inputs of a block's fibers are staged while they leave room for two
    // blocks per SM; past that they are read where they are used
    const size_t stage = (size_t)f.P * 32 * V * sizeof(T);
    const bool staged = stage <= 96 * 1024;
    const size_t sm = staged ? stage : 0;
    if (sm > 32 * 1024)
      OSMPS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024));
    const bool wide = total > 2147483647ll;
    const FastDiv by_nc(wide ? 1 : (uint32_t)nc), by_o2(wide ? 1 : (uint32_t)f.n_o2);
    const int blocks = wstep_blocks(cdiv(total, 32 * (packed ? 1 : V)), sm + sizeof(WTable<T>) + 1024);
    k<<<blocks, 32 * FIB_WARPS, sm, s>>>(f, Mat, in, out, sdst, Kcols, Kp, staged ? 1 : 0, by_nc, by_o2,
                                         wide ? 1 : 0);
    note_launch();
    OSMPS_LAUNCH_CHECK();
    return OSMPS_OK;
  };
  constexpr int V = 16 / sizeof(T);
  if (packs<T>({f.nc, f.is1, f.is2, f.istride, f.os1, f.os2, f.ostride, Kcols * (MODE != 0)}, {in, out, sdst}))
    return launch(k_fiber<T, MODE, V, true>, V, true);
  return launch(k_fiber<T, MODE, 2, false>, 2, false);
}

// Both W-steps of H_eff.theta in one pass for any MPO bond dimensions
// (d1 = d2 = D), the work of 32 V fibers (a2, c) shared by a block's warps as
// in k_fiber: they load the wl D D values T1[a2, w, s1, s2, c] into shared
// memory, form T2[t1, w1, s2] beside them, then the outputs T3[t1, t2, w2], so
// the intermediate never crosses memory. The sums are those of the two
// separate passes, term by term. Traffic: one read of T1, one write of T3; in
// float64 the ~36 FMAs per fiber come next (XXZ chi = 512: 55 us, float64 pipe
// 44% active, against 158 + 158 us for two dense passes); AKLT 301x257 in
// float32 61 us against 152 + 147. Blocks per SM: for packed float64 fibers the
// five that the tables and XXZ's columns leave room for (with four, 71 us), else
// four (left to itself the compiler takes 48 registers: AKLT 2 us slower, a
// 33 x 31 float64 product 1 us).
template <typename T, int MODE, int D, int V, bool PACKED>
__global__ void __launch_bounds__(32 * FIB_WARPS, sizeof(T) == 8 && PACKED ? 5 : 4)
    k_wsteps(const T* __restrict__ T1, const double* __restrict__ Mat1,
             const double* __restrict__ Mat2, int wl, int wm, int wr, T* __restrict__ out,
             void* __restrict__ sdst, int64_t Kp, int64_t chi_l, int64_t chi_r, FastDiv by_c,
             int wide) {
  extern __shared__ __align__(16) uint8_t fsm[];
  __shared__ WTable<T> tab1, tab2;
  __shared__ int64_t ooff[WT_QMAX];  // output (t2, w2): offset from (t1, 0, 0)
  using F = Fibers<T, V, PACKED>;
  const int P1 = wl * D, Q1 = D * wm, P2 = wm * D, Q2 = D * wr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Pack<T, V>* xs = reinterpret_cast<Pack<T, V>*>(fsm) + lane;
  Pack<T, V>* ms = xs + P1 * D * 32;
  const int64_t ldo = MODE == 0 ? wr * chi_r : 2 * Kp;
  if (threadIdx.x < Q2) {
    const int t2 = threadIdx.x / wr;
    ooff[threadIdx.x] = t2 * ldo + (int64_t)(threadIdx.x - t2 * wr) * chi_r;
  }
  bool first = true;  // the tables are built while the first fibers' inputs arrive
  const int64_t nc = PACKED ? chi_r / V : chi_r, total = chi_l * nc;
  for (int64_t e0 = (int64_t)blockIdx.x * (32 * F::N); e0 < total; e0 += (int64_t)gridDim.x * (32 * F::N)) {
    F fib;
    int64_t ob[F::N];
#pragma unroll
    for (int v = 0; v < F::N; ++v) {
      const int64_t ev = e0 + 32 * v + lane, e = ev < total ? ev : e0;
      const int64_t a2 = div_by(by_c, e, nc, wide), c = (e - a2 * nc) * (PACKED ? V : 1);
      fib.ok[v] = ev < total;
      fib.at[v] = a2 * (P1 * D) * chi_r + c;
      ob[v] = a2 * (D * D) * ldo + c;
    }
    int top = 0;
#pragma unroll 4
    for (int k = warp; k < P1 * D; k += FIB_WARPS) {
      const Pack<T, V> x = fib.load(T1, k * chi_r);
      xs[k * 32] = x;
      note_top<T, V>(top, x);
    }
    if (first) {
      gather_terms<2, T>(top, {Mat1, Mat2}, {P1, P2}, {Q1, Q2}, {&tab1, &tab2});
    } else {
      if (wild<T>(top)) tab1.dense = tab2.dense = W_ALL;  // from here on
      __syncthreads();
    }
    first = false;
    for (int o = warp; o < Q1; o += FIB_WARPS)
#pragma unroll
      for (int s2 = 0; s2 < D; ++s2) ms[(o * D + s2) * 32] = sum_terms<T, V>(tab1, o, xs + s2 * 32, D * 32);
    __syncthreads();  // T2 complete; T1's copy may be overwritten by the next fibers
    for (int o = warp; o < Q2; o += FIB_WARPS)
#pragma unroll
      for (int t1 = 0; t1 < D; ++t1)
        fib.template store<MODE>(out, sdst, ob, t1 * D * ldo + ooff[o], Kp,
                                 sum_terms<T, V>(tab2, o, ms + t1 * (P2 * 32), 32));
    // (the next fibers' T2 is written only after the barrier that follows their loads)
  }
}

// *done = false where the fused pass does not apply (physical dimensions
// other than 2 to 5, MPO blocks beyond the separate passes' own limits, or
// columns of which not 64 fit shared memory).
template <typename T, int MODE>
osmps_status wsteps_dispatch(const T* T1, const double* Mat1, const double* Mat2, int64_t chi_l,
                             int64_t d1, int64_t d2, int64_t chi_r, int64_t wl, int64_t wm,
                             int64_t wr, T* out, void* sdst, int64_t Kp, cudaStream_t s,
                             bool* done) {
  *done = false;
  if (d1 != d2 || d1 < 2 || d1 > 5 || d1 * std::max(wm, wr) > WT_QMAX || d1 * wl > 2048) return OSMPS_OK;
  const int64_t P1 = wl * d1, Q1 = d1 * wm, P2 = wm * d1, Q2 = d1 * wr;
  if ((size_t)std::max(P1 * Q1, P2 * Q2) * sizeof(T) > 96 * 1024) return OSMPS_OK;
  // 16-byte packs of neighbouring fibers while two blocks still share an SM,
  // else two fibers 32 apart
  const size_t column = (size_t)(P1 + Q1) * d1 * sizeof(T);  // one fiber's T1 and T2
  constexpr size_t MOST = 180 * 1024;
  constexpr int VMAX = 16 / sizeof(T);
  if (column * 64 > MOST) return OSMPS_OK;
  const bool packed = column * 32 * VMAX <= 90 * 1024 && packs<T>({chi_r}, {T1, out, sdst});
  const auto launch = [&](auto k, int V) -> osmps_status {
    const size_t sm = column * 32 * V;
    const int64_t nc = packed ? chi_r / V : chi_r, total = chi_l * nc;
    const bool wide = total > 2147483647ll;
    const FastDiv by_c(wide ? 1 : (uint32_t)nc);
    const int blocks = wstep_blocks(cdiv(total, 32 * (packed ? 1 : V)), sm + 2 * sizeof(WTable<T>) + 1600);
    if (sm > 24 * 1024)
      OSMPS_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MOST));
    k<<<blocks, 32 * FIB_WARPS, sm, s>>>(T1, Mat1, Mat2, (int)wl, (int)wm, (int)wr, out, sdst, Kp, chi_l,
                                         chi_r, by_c, wide ? 1 : 0);
    note_launch();
    OSMPS_LAUNCH_CHECK();
    return OSMPS_OK;
  };
#define OSMPS_WSTEPS(D_) \
  OSMPS_TRY(packed ? launch(k_wsteps<T, MODE, D_, VMAX, true>, VMAX) : launch(k_wsteps<T, MODE, D_, 2, false>, 2))
  if (d1 == 2) OSMPS_WSTEPS(2);
  else if (d1 == 3) OSMPS_WSTEPS(3);
  else if (d1 == 4) OSMPS_WSTEPS(4);
  else OSMPS_WSTEPS(5);
#undef OSMPS_WSTEPS
  *done = true;
  return OSMPS_OK;
}

template <int KIND>
__global__ void k_zero_pad(void* dst, int64_t rows, int64_t Kcols, int64_t Kp) {
  const int64_t w = Kp - Kcols;
  const int64_t total = rows * w;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / w, k = Kcols + (e - r * w);
    split_store_f32<KIND>(dst, r * 2 * Kp + k, Kp, 0.0f);
  }
}

__global__ void k_w_reorder(const double* __restrict__ W, int64_t dw, int64_t d, int64_t dw2,
                            int order, double* __restrict__ Mat) {
  const int64_t total = dw * d * d * dw2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    // e enumerates W[w, t, s, w2] in row-major order
    int64_t w2 = e % dw2, r = e / dw2;
    int64_t s = r % d;
    r /= d;
    int64_t t = r % d, w = r / d;
    int64_t i, o, Q;
    if (order == WORD_IN_W_S__OUT_T_W2) {
      i = w * d + s;
      o = t * dw2 + w2;
      Q = d * dw2;
    } else if (order == WORD_IN_T_W2__OUT_W_S) {
      i = t * dw2 + w2;
      o = w * d + s;
      Q = dw * d;
    } else {
      i = s * dw2 + w2;
      o = w * d + t;
      Q = dw * d;
    }
    Mat[i * Q + o] = W[e];
  }
}

// Both W-steps of H_eff.theta in one pass, for the spin-1/2 chains (d = 2)
// whose MPO bond dimensions are fixed at compile time: for every fiber
// (a2, c) the wl*d*d values T1[a2, w, s1, s2, c] are contracted with W1 and
// then W2 in registers and written straight into the split operand
// T3[(a2, t1, t2), (w2, c)]; the intermediate T2 never touches memory.
// Identity environment channels (skip_l, skip_r >= 0): L[:, skip_l, :] = 1,
// so T1's channel skip_l is theta itself and the stage-1 GEMM leaves it out
// (T1 holds the other WL - 1 channels in order); R[:, skip_r, :] = 1, so
// output channel skip_r needs no stage-4 GEMM: it goes as float32 to yid
// (row (a2, t1, t2), column c2), which the stage-4 epilogue adds, and the
// split operand holds the other WR - 1 channels in order.
// SL, SR: the identity channels fixed at compile time (-1: none), or
// SKIP_RUNTIME to take skip_l / skip_r from the arguments. Compile-time
// values let the channel loops fold: with runtime tests in the load loop the
// kernel measured 58 instead of 38 us at chi = 1024.
constexpr int SKIP_RUNTIME = -2;
template <int D, int WL, int WM, int WR, int KIND, int V, int SL, int SR>
__global__ void __launch_bounds__(256, 2) k_fused_wsteps(const float* __restrict__ T1,
                                                         const double* __restrict__ Mat1,
                                                         const double* __restrict__ Mat2,
                                                         void* __restrict__ dst, int64_t chi_l,
                                                         int64_t chi_r, int64_t Kp,
                                                         const double* __restrict__ theta,
                                                         int skip_l_arg, int skip_r_arg,
                                                         float* __restrict__ yid) {
  const int skip_l = SL == SKIP_RUNTIME ? skip_l_arg : SL;
  const int skip_r = SR == SKIP_RUNTIME ? skip_r_arg : SR;
  constexpr int P1 = WL * D, Q1 = D * WM, P2 = WM * D, Q2 = D * WR;
  static_assert(P1 <= 32 && P2 <= 32, "input masks are 32-bit");
  __shared__ float sm1[P1 * Q1], sm2[P2 * Q2];
  __shared__ unsigned nz1[Q1], nz2[Q2];  // per output: which inputs have a nonzero W entry
  for (int i = threadIdx.x; i < P1 * Q1; i += blockDim.x) sm1[i] = (float)Mat1[i];
  for (int i = threadIdx.x; i < P2 * Q2; i += blockDim.x) sm2[i] = (float)Mat2[i];
  if (threadIdx.x < Q1) nz1[threadIdx.x] = 0u;
  if (threadIdx.x < Q2) nz2[threadIdx.x] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < P1 * Q1; i += blockDim.x)
    if (sm1[i] != 0.0f) atomicOr(&nz1[i % Q1], 1u << (i / Q1));
  for (int i = threadIdx.x; i < P2 * Q2; i += blockDim.x)
    if (sm2[i] != 0.0f) atomicOr(&nz2[i % Q2], 1u << (i / Q2));
  __syncthreads();
  // MPO tensors are mostly zeros (an identity in two corners and a few local
  // operators): every multiply-add is guarded by the output's nonzero mask,
  // a branch that is uniform over the grid, and the W entry is read from
  // shared memory only where it is nonzero (kept in registers the ~200
  // entries would leave one block per SM, too few loads in flight for HBM)
  const volatile float* m1 = sm1;
  const volatile float* m2 = sm2;
  // V consecutive fibers c per thread (V = 2: 8-byte loads, paired stores;
  // chi_r even)
  const int64_t cv = chi_r / V;
  const int64_t total = chi_l * cv;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a2 = e / cv, c = (e - a2 * cv) * V;
    const int wlt = skip_l >= 0 ? WL - 1 : WL;  // channels held in T1
    const float* src = T1 + a2 * (wlt * D * D) * chi_r + c;
    float x[WL][D][D][V];
#pragma unroll
    for (int w = 0; w < WL; ++w)
#pragma unroll
      for (int s1 = 0; s1 < D; ++s1)
#pragma unroll
        for (int s2 = 0; s2 < D; ++s2) {
          if (w == skip_l) {  // uniform branch: the identity channel is theta
            const double* q = theta + ((a2 * D + s1) * D + s2) * chi_r + c;
            if (V == 2) {
              const double2 f = *reinterpret_cast<const double2*>(q);
              x[w][s1][s2][0] = (float)f.x;
              x[w][s1][s2][V - 1] = (float)f.y;
            } else {
              x[w][s1][s2][0] = (float)q[0];
            }
            continue;
          }
          const int wt = (skip_l >= 0 && w > skip_l) ? w - 1 : w;
          const float* p = src + ((wt * D + s1) * D + s2) * chi_r;
          if (V == 2) {
            const float2 f = *reinterpret_cast<const float2*>(p);
            x[w][s1][s2][0] = f.x;
            x[w][s1][s2][V - 1] = f.y;
          } else {
            x[w][s1][s2][0] = p[0];
          }
        }
    float mid[D][WM][D][V];  // T2[t1, w1, s2]
#pragma unroll
    for (int t1 = 0; t1 < D; ++t1)
#pragma unroll
      for (int w1 = 0; w1 < WM; ++w1) {
        const unsigned mask = nz1[t1 * WM + w1];
        float acc[D][V];
#pragma unroll
        for (int s2 = 0; s2 < D; ++s2)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[s2][v] = 0.0f;
#pragma unroll
        for (int w = 0; w < WL; ++w)
#pragma unroll
          for (int s1 = 0; s1 < D; ++s1)
            if (mask & (1u << (w * D + s1))) {
              const float m = m1[(w * D + s1) * Q1 + t1 * WM + w1];
#pragma unroll
              for (int s2 = 0; s2 < D; ++s2)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[s2][v] = fmaf(m, x[w][s1][s2][v], acc[s2][v]);
            }
#pragma unroll
        for (int s2 = 0; s2 < D; ++s2)
#pragma unroll
          for (int v = 0; v < V; ++v) mid[t1][w1][s2][v] = acc[s2][v];
      }
#pragma unroll
    for (int t2 = 0; t2 < D; ++t2)
#pragma unroll
      for (int w2 = 0; w2 < WR; ++w2) {
        const unsigned mask = nz2[t2 * WR + w2];
        float acc[D][V];
#pragma unroll
        for (int t1 = 0; t1 < D; ++t1)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[t1][v] = 0.0f;
#pragma unroll
        for (int w1 = 0; w1 < WM; ++w1)
#pragma unroll
          for (int s2 = 0; s2 < D; ++s2)
            if (mask & (1u << (w1 * D + s2))) {
              const float m = m2[(w1 * D + s2) * Q2 + t2 * WR + w2];
#pragma unroll
              for (int t1 = 0; t1 < D; ++t1)
#pragma unroll
                for (int v = 0; v < V; ++v) acc[t1][v] = fmaf(m, mid[t1][w1][s2][v], acc[t1][v]);
            }
#pragma unroll
        for (int t1 = 0; t1 < D; ++t1) {
          const int64_t row = (a2 * D + t1) * D + t2;
          if (w2 == skip_r) {
            float* q = yid + row * chi_r + c;
            if (V == 2) *reinterpret_cast<float2*>(q) = make_float2(acc[t1][0], acc[t1][V - 1]);
            else q[0] = acc[t1][0];
            continue;
          }
          const int w2t = (skip_r >= 0 && w2 > skip_r) ? w2 - 1 : w2;
          const int64_t off = row * 2 * Kp + (int64_t)w2t * chi_r + c;
          if (V == 2) split_store2_f32<KIND>(dst, off, Kp, acc[t1][0], acc[t1][V - 1]);
          else split_store_f32<KIND>(dst, off, Kp, acc[t1][0]);
        }
      }
  }
}

template <int D, int WL, int WM, int WR>
bool try_fused(int64_t d, int64_t wl, int64_t wm, int64_t wr, int kind, const float* T1,
               const double* m1, const double* m2, void* dst, int64_t chi_l, int64_t chi_r,
               int64_t Kp, const WStepIdentity& id, cudaStream_t s, bool launch) {
  if (d != D || wl != WL || wm != WM || wr != WR) return false;
  if (!launch) return true;  // shape query only
  const double* th = id.theta;
  const int sl = id.skip_l, sr = id.skip_r;
  float* yid = id.yid;
  // two resident blocks per SM, each striding over many fibers (the
  // per-block set-up of the W tables is then paid a few hundred times only)
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 152;
  // pairs of fibers: 8-byte loads of T1, 16-byte loads of theta (identity
  // channel) and paired stores, so chi_r even and theta 16-byte aligned
  const bool pair = chi_r % 2 == 0 && (sl < 0 || (reinterpret_cast<uintptr_t>(th) & 15) == 0);
  const int blocks = (int)std::min<int64_t>(grid_for(chi_l * (pair ? chi_r / 2 : chi_r), 256), 2 * (int64_t)sms);
  // compile-time identity channels for the cases a sweep meets (none; L's
  // last and/or R's first channel), the runtime form for the rest
  const int combo = (sl == -1 && sr == -1) ? 0 : (sl == WL - 1 && sr == 0) ? 1
                  : (sl == WL - 1 && sr == -1) ? 2 : (sl == -1 && sr == 0) ? 3 : 4;
#define OSMPS_FUSED(K, V, L_, R_) \
  k_fused_wsteps<D, WL, WM, WR, K, V, L_, R_><<<blocks, 256, 0, s>>>(T1, m1, m2, dst, chi_l, chi_r, Kp, th, sl, sr, yid)
#define OSMPS_FUSED_KIND(K)                                                   \
  if (!pair) OSMPS_FUSED(K, 1, SKIP_RUNTIME, SKIP_RUNTIME);                    \
  else if (combo == 0) OSMPS_FUSED(K, 2, -1, -1);                             \
  else if (combo == 1) OSMPS_FUSED(K, 2, WL - 1, 0);                          \
  else if (combo == 2) OSMPS_FUSED(K, 2, WL - 1, -1);                         \
  else if (combo == 3) OSMPS_FUSED(K, 2, -1, 0);                              \
  else OSMPS_FUSED(K, 2, SKIP_RUNTIME, SKIP_RUNTIME);
  if (kind == TC_BF16) {
    OSMPS_FUSED_KIND(TC_BF16)
  } else {
    OSMPS_FUSED_KIND(TC_TF32)
  }
#undef OSMPS_FUSED_KIND
#undef OSMPS_FUSED
  note_launch();
  return true;
}

}  // namespace

template <int KIND, typename S>
static osmps_status split_operand_as(const SplitView& v, void* dst, int64_t Kp, cudaStream_t s) {
  if (v.sk == 1 || v.K == 1) {
    const int64_t units = v.rows * (Kp / 8);
    const bool wide = units > 2147483647ll || v.n1 > 2147483647ll;
    constexpr int64_t PER = 16 / sizeof(S);
    const bool vec = v.sk == 1 && (reinterpret_cast<uintptr_t>(v.src) & 15) == 0 && v.s0 % PER == 0 &&
                     (v.n1 == 1 || v.s1 % PER == 0);
    const FastDiv by_k8(wide ? 1 : (uint32_t)(Kp / 8)), by_n1(wide ? 1 : (uint32_t)v.n1);
    k_split_direct<KIND, S><<<grid_for(units, 256), 256, 0, s>>>(v, dst, Kp, by_k8, by_n1, vec ? 1 : 0,
                                                                wide ? 1 : 0);
  } else {
    if (cdiv(Kp, 64) > 65535) return set_error(OSMPS_ESHAPE, "split_operand: K too large");
    const dim3 grid((unsigned)cdiv(v.rows, 64), (unsigned)cdiv(Kp, 64));
    k_split_transpose<KIND, S><<<grid, 256, 0, s>>>(v, dst, Kp);
  }
  note_launch();
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

// Traffic: 8 (4) bytes read and 4 (8) written per value. chi = 1024, bf16: L
// (5120 rows of 1024) 41 us and theta transposed (4096 x 1024) 35 us before
// the integer split and the wide accesses.
osmps_status split_operand(const SplitView& v, int kind, void* dst, int64_t Kp, cudaStream_t s) {
  if (v.rows <= 0) return OSMPS_OK;
  if (Kp < v.K || Kp % 64 != 0) return set_error(OSMPS_ESHAPE, "split_operand: bad Kp");
  if (kind == TC_BF16)
    return v.src_f32 ? split_operand_as<TC_BF16, float>(v, dst, Kp, s)
                     : split_operand_as<TC_BF16, double>(v, dst, Kp, s);
  return v.src_f32 ? split_operand_as<TC_TF32, float>(v, dst, Kp, s)
                   : split_operand_as<TC_TF32, double>(v, dst, Kp, s);
}

osmps_status fiber_contract_f64(const Fiber& f, const double* Mat, const double* in, double* out,
                                cudaStream_t s) {
  return fiber_dispatch<double, 0>(f, Mat, in, out, nullptr, 1, 0, s);
}

osmps_status fiber_contract_f32(const Fiber& f, const double* Mat, const float* in, float* out,
                                cudaStream_t s) {
  return fiber_dispatch<float, 0>(f, Mat, in, out, nullptr, 1, 0, s);
}

osmps_status fiber_contract_f32_split(const Fiber& f, const double* Mat, const float* in,
                                      void* dst, int kind, int64_t Kcols, int64_t Kp,
                                      cudaStream_t s) {
  if (kind == TC_BF16) return fiber_dispatch<float, 1>(f, Mat, in, nullptr, dst, Kcols, Kp, s);
  return fiber_dispatch<float, 2>(f, Mat, in, nullptr, dst, Kcols, Kp, s);
}

osmps_status wsteps_f64(const double* T1, const double* Mat1, const double* Mat2, double* T3,
                        int64_t chi_l, int64_t d1, int64_t d2, int64_t chi_r, int64_t wl,
                        int64_t wm, int64_t wr, cudaStream_t s, bool* done) {
  return wsteps_dispatch<double, 0>(T1, Mat1, Mat2, chi_l, d1, d2, chi_r, wl, wm, wr, T3, nullptr,
                                    0, s, done);
}

// max over (a, b) of |E[a, w, b] - delta_ab| for w = 0 (blockIdx.y = 0) and
// w = w_count - 1 (blockIdx.y = 1), as the bit patterns of non-negative
// doubles (ordered like the values) combined by atomicMax
__global__ void k_identity_deviation(const double* __restrict__ E, int64_t chi, int64_t w_count,
                                     unsigned long long* __restrict__ out) {
  const int64_t w = blockIdx.y == 0 ? 0 : w_count - 1;
  const int64_t total = chi * chi;
  double m = 0.0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = e / chi, b = e - a * chi;
    const double v = E[(a * w_count + w) * chi + b] - (a == b ? 1.0 : 0.0);
    const double av = fabs(v);
    m = (av > m || av != av) ? (av != av ? INFINITY : av) : m;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&out[blockIdx.y], (unsigned long long)__double_as_longlong(m));
}

static bool fused_dispatch(int64_t d1, int64_t d2, int64_t wl, int64_t wm, int64_t wr, int kind,
                           const float* T1, const double* Mat1, const double* Mat2, void* dst,
                           int64_t chi_l, int64_t chi_r, int64_t Kp, const WStepIdentity& id,
                           cudaStream_t s, bool launch) {
  if (d1 != d2) return false;
  const int64_t d = d1;
#define OSMPS_TRY_FUSED(a, b, c, e) \
  try_fused<a, b, c, e>(d, wl, wm, wr, kind, T1, Mat1, Mat2, dst, chi_l, chi_r, Kp, id, s, launch)
  return OSMPS_TRY_FUSED(2, 5, 5, 5) || OSMPS_TRY_FUSED(2, 1, 5, 5) || OSMPS_TRY_FUSED(2, 5, 5, 1) ||
         OSMPS_TRY_FUSED(2, 3, 3, 3) || OSMPS_TRY_FUSED(2, 1, 3, 3) || OSMPS_TRY_FUSED(2, 3, 3, 1);
#undef OSMPS_TRY_FUSED
}

osmps_status identity_channel_deviation(const double* E, int64_t chi, int64_t w_count,
                                        double* dev_out, cudaStream_t s) {
  OSMPS_CUDA(cudaMemsetAsync(dev_out, 0, 2 * sizeof(double), s));
  if (chi <= 0 || w_count <= 0) return OSMPS_OK;
  const int bx = (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(chi * chi, 256 * 8), 1024));
  k_identity_deviation<<<dim3(bx, 2), 256, 0, s>>>(E, chi, w_count,
                                                  reinterpret_cast<unsigned long long*>(dev_out));
  note_launch();
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

bool fused_wsteps_supported(int64_t d1, int64_t d2, int64_t wl, int64_t wm, int64_t wr) {
  return fused_dispatch(d1, d2, wl, wm, wr, TC_BF16, nullptr, nullptr, nullptr, nullptr, 0, 0, 0,
                        WStepIdentity{}, nullptr, false);
}

osmps_status fused_wsteps_f32_split(const float* T1, const double* Mat1, const double* Mat2,
                                    void* dst, int kind, int64_t chi_l, int64_t d1, int64_t d2,
                                    int64_t chi_r, int64_t wl, int64_t wm, int64_t wr, int64_t Kp,
                                    const WStepIdentity& id, cudaStream_t s, bool* done) {
  *done = false;
  if ((id.skip_l >= 0 && !id.theta) || (id.skip_r >= 0 && !id.yid))
    return set_error(OSMPS_EINVAL, "fused W-steps: identity channel without its buffer");
  if (!fused_dispatch(d1, d2, wl, wm, wr, kind, T1, Mat1, Mat2, dst, chi_l, chi_r, Kp, id, s, true)) {
    if (id.skip_l >= 0 || id.skip_r >= 0) return OSMPS_OK;
    if (kind == TC_BF16)
      return wsteps_dispatch<float, 1>(T1, Mat1, Mat2, chi_l, d1, d2, chi_r, wl, wm, wr, nullptr,
                                       dst, Kp, s, done);
    return wsteps_dispatch<float, 2>(T1, Mat1, Mat2, chi_l, d1, d2, chi_r, wl, wm, wr, nullptr, dst,
                                     Kp, s, done);
  }
  OSMPS_LAUNCH_CHECK();
  *done = true;
  return OSMPS_OK;
}

osmps_status zero_pad_columns(void* dst, int kind, int64_t rows, int64_t Kcols, int64_t Kp,
                              cudaStream_t s) {
  if (Kp <= Kcols || rows <= 0) return OSMPS_OK;
  const int blocks = grid_for(rows * (Kp - Kcols), 256);
  if (kind == TC_BF16) { k_zero_pad<TC_BF16><<<blocks, 256, 0, s>>>(dst, rows, Kcols, Kp); note_launch(); }
  else { k_zero_pad<TC_TF32><<<blocks, 256, 0, s>>>(dst, rows, Kcols, Kp); note_launch(); }
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

// H_eff's two site tensors in one launch, one block row each.
__global__ void k_w_reorder_pair(const double* __restrict__ W1, const double* __restrict__ W2,
                                 int64_t wl, int64_t d1, int64_t wm, int64_t d2, int64_t wr,
                                 double* __restrict__ M1, double* __restrict__ M2) {
  const bool second = blockIdx.y == 1;
  const double* W = second ? W2 : W1;
  double* Mat = second ? M2 : M1;
  const int64_t dw = second ? wm : wl, d = second ? d2 : d1, dw2 = second ? wr : wm;
  const int64_t total = dw * d * d * dw2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w2 = e % dw2, r = e / dw2, s = r % d, q = r / d, t = q % d, w = q / d;
    Mat[(w * d + s) * (d * dw2) + t * dw2 + w2] = W[e];
  }
}

osmps_status w_reorder_pair(const double* W1, const double* W2, int64_t wl, int64_t d1, int64_t wm,
                            int64_t d2, int64_t wr, double* M1, double* M2, cudaStream_t s) {
  const int64_t most = std::max(wl * d1 * d1 * wm, wm * d2 * d2 * wr);
  k_w_reorder_pair<<<dim3(std::min(grid_for(most, 256), 1024), 2), 256, 0, s>>>(W1, W2, wl, d1, wm, d2, wr, M1, M2);
  note_launch();
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

osmps_status w_reorder(const double* W, int64_t dw, int64_t d, int64_t dw2, int order, double* Mat,
                       cudaStream_t s) {
  const int64_t total = dw * d * d * dw2;
  { k_w_reorder<<<grid_for(total, 256), 256, 0, s>>>(W, dw, d, dw2, order, Mat); note_launch(); }
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

}  // namespace osmps
