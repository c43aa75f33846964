// Float64-accurate GEMM on the bf16 tensor cores (error-free slicing).
//
// GB300's float64 units are slow; its bf16 tensor cores are about a
// thousand times faster. A float64 GEMM is emulated on them exactly in the
// manner of Ozaki's error-free transformation of matrix products:
//   * every row of A (and of B, both K-major) is scaled by a power of two
//     2^-e so that its entries lie in (-1, 1), rounded to 56 fractional bits
//     and cut into S = 8 balanced base-128 digits q_p (|q_p| <= 128), so
//     x = 2^e sum_p q_p 2^(-7(p+1)); the slices hold the integers q_p, exact
//     in bf16 (all of this with integer arithmetic on the IEEE bits);
//   * a slice pair (i, j) gives integer products q_i q_j of at most 2^14,
//     so a run of 1024 of them sums to at most 2^24: exact in the float32
//     TMEM accumulator, integers being exact there up to 2^24 (tested with
//     every top digit at 128);
//   * the epilogue converts those exact integers and adds them per slice diagonal
//     i + j (same unit 2^(-7(i+j+2))), over the 36 pairs with i + j <= 7
//     (the dropped pairs are below 2^-56 of the row scales);
//   * pairs on one diagonal share the unit, so a TMEM partial sum runs over
//     several K blocks of 64 and all pairs of its diagonal: 16 block products
//     on diagonal 0, 32 on the others;
//   * the diagonals are taken in groups of four (two while K > 2^17), one TMEM
//     accumulator of 128 columns each. Their partial sums are combined exactly
//     in int64 at weights 2^7 apart and stay below 2^53; a group sum becomes
//     a float64 by integer operations on the IEEE bits, the row and column
//     scales 2^(e_A + e_B) folded into its exponent, and the group values
//     are added in float64. One float64 addition per output element and group
//     after the first remains: GB300's float64 pipe is what limits this kind
//     of kernel otherwise. The result is stored, or subtracted from C.
// What bounds it: the MMAs, 64 clocks per 128 x 128 x 16. A group walks K once
// and forms all its pairs from one copy of the slices in shared memory: 24
// slice tiles per K block and output tile where a pass over K for each pair
// took 72, 57 bytes per clock into an SM at one pair in 570 clocks; now 380 and a
// tile's drains (ncu, 5120 x 4096 x 1024: 411 with them on the busiest SM, tensor
// pipe 64% active, 25 bytes per clock), the rest being the single issuing warp.
// 2048 x 2048 x 2048: kernel 764 -> 479 us (1290 TFLOP/s of bf16), 2560 x 2048 x
// 512: 348 -> 208, 2048 x 512 x 2560 with K in shares: 475 -> 168, 381 x 1905 x
// 1000: 201 -> 68. (Shares are added as integers: rounded to float64 first they
// cost 177 and 75 us and seven more roundings, 1.3e-16 instead of 8e-17 against
// 113-bit arithmetic at 128 x 128 x 2048.)
// The kernel is persistent and warp-specialised: a TMA producer with a ring
// of 13 slice tiles, a warp that issues the MMAs, and 16 epilogue warps each
// holding 32 exact sums per row in registers.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "operand.cuh"
#include "tcgen05.cuh"

namespace osmps {

namespace {

using namespace tc;

constexpr int SLICES = 8;
constexpr int SLICE_BITS = 7;
constexpr int EBM = 128, EBN = 128;
constexpr int E_SLOTS = 13;                // ring of 128-row, 64-element slice tiles
constexpr int E_TILE = 128 * 128;          // bytes of one
constexpr int E_BUFS = 4;                  // TMEM accumulators: one per diagonal of a group
constexpr int E_EPI_WARPS = 16;
constexpr int E_EPI_COLS = EBN / 4;
constexpr int E_THREADS = 64 + 32 * E_EPI_WARPS;
constexpr uint32_t E_TMEM_COLS = E_BUFS * EBN;
constexpr size_t E_SMEM = (size_t)E_SLOTS * E_TILE + 1024 + 512;
static_assert(EBM == 128 && EBN == 128 && E_SMEM <= 227 * 1024, "slice tile ring");

// 64-element K blocks per exact partial sum of diagonal d, whose d + 1 pairs
// share one accumulator: digit products are at most 2^14 in size on diagonal 0
// (|d_0| <= 128) and 2^13 on the others, so 16 and 32 of their 64-term sums
// stay within 2^24.
__host__ __device__ constexpr int chunk_blocks(int d) { return d == 0 ? 16 : 32 / (d + 1); }
// the same as bytes of a word (a division costs the drains more than a shift)
constexpr uint64_t chunk_bytes() {
  uint64_t w = 0;
  for (int d = 0; d < SLICES; ++d) w |= (uint64_t)chunk_blocks(d) << (8 * d);
  return w;
}

// The slices' order of arrival within a K block of diagonals d0..d1: first
// A_d1 .. A_d0 and B_0, then before each further b the slice A_(d0-b), if
// there is one, and B_b. Position in that order:
__host__ __device__ constexpr int a_pos(int a, int d0, int d1) {
  return a >= d0 ? d1 - a : d1 - d0 + 2 * (d0 - a);
}
__host__ __device__ constexpr int b_pos(int b, int d0, int d1) {
  return d1 - d0 + 1 + (b <= d0 ? 2 * b : d0 + b);
}

// x 2^k as a float64 for an integer |x| < 2^53, built from the IEEE-754 bit
// layout (sign, biased exponent, 52 fraction bits) with integer operations
// only; exact whenever the result is a normal number, else left to scalbn.
__device__ __forceinline__ double i64_ldexp(long long x, int k) {
  if (x == 0) return 0.0;
  const unsigned long long a = x < 0 ? (unsigned long long)(-x) : (unsigned long long)x;
  const int e = 63 - __clzll((long long)a);  // a in [2^e, 2^(e+1)), e <= 52
  const int E = e + k + 1023;
  if (E <= 0 || E >= 2047) return scalbn((double)x, k);
  const unsigned long long frac = (a << (52 - e)) & 0xFFFFFFFFFFFFFull;
  return __longlong_as_double((long long)(((unsigned long long)(x < 0) << 63) |
                                          ((unsigned long long)E << 52) | frac));
}

// Tile t -> (m0, n0) in groups of E_GROUP_M tile rows, columns walked within
// a group: the tiles that run at the same time then share E_GROUP_M A row
// slabs and fewer B column slabs than a row-major walk, so more of the slice
// operands stay in L2.
constexpr int E_GROUP_M = 8;
__device__ __forceinline__ void emu_tile(int tile, int tiles_m, int tiles_n, int& m0, int& n0) {
  const int per_group = E_GROUP_M * tiles_n;
  const int g = tile / per_group, first = g * E_GROUP_M;
  const int rows = min(tiles_m - first, E_GROUP_M);
  const int local = tile - g * per_group;
  m0 = (first + local % rows) * EBM;
  n0 = (local / rows) * EBN;
}

// Four float64 values of a row, at columns c .. c+3 of N; two per access where
// `vec` says that rows and base are 16-byte aligned.
__device__ __forceinline__ void load_row4(const double* p, int64_t c, int64_t N, int vec, double (&v)[4]) {
  if (vec && c + 4 <= N) {
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
      const double2 t = *reinterpret_cast<const double2*>(p + c + i);
      v[i] = t.x;
      v[i + 1] = t.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = c + i < N ? p[c + i] : 0.0;
  }
}
__device__ __forceinline__ void store_row4(double* p, int64_t c, int64_t N, int vec, const double (&v)[4]) {
  if (vec && c + 4 <= N) {
#pragma unroll
    for (int i = 0; i < 4; i += 2) *reinterpret_cast<double2*>(p + c + i) = make_double2(v[i], v[i + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (c + i < N) p[c + i] = v[i];
  }
}

// What the kernel writes: C[r][c] (subtract: C -= the product), rows of ldc
// values, two per access where `vec`. G holds the sums of the diagonal groups
// before the last, in an order of the threads' own (128 KB for each CTA,
// [column pair][thread], so that a warp's accesses are whole lines: in C itself
// they took a line for each lane).
// With K in shares (H set) nothing is rounded here: group g of share s goes to
// H[s][g][r][c] as the exact integer, planes of `slab` and rows of ldc integers
// (ldc a multiple of four), and k_emu_combine adds the shares.
struct EmuOut {
  double* C;
  double2* G;
  long long* H;
  int64_t ldc, slab;
  int subtract, vec;
};

// The MMA issuer's place in the ring: slot and phase of the next K block's
// first slice; blocks in each buffer's partial sum, and the buffers' phases.
struct EmuIssue {
  uint32_t slot = 0, phase = 0, used = 0;
  int count[E_BUFS] = {};
};

// Issue the pairs of diagonals D0 .. D0 + GD - 1 over one K block, B slice by
// B slice; false when a wait ran out. One thread issues everything, at one
// instruction per several clocks, and has 256 clocks per pair: positions in the
// ring and partial-sum lengths are constants of the unrolled loops (computed,
// they cost 1040 clocks a pair).
template <int D0, int GD>
__device__ __forceinline__ bool emu_issue_block(EmuIssue& st, uint32_t ring, uint32_t tmem,
                                                uint64_t* full, uint64_t* empty, uint64_t* tfull,
                                                uint64_t* tempty, bool last_block) {
  constexpr int D1 = D0 + GD - 1;
  const uint32_t id = idesc<TC_BF16, EBM, EBN>();
  const uint64_t desc0 = sdesc(ring);
  const auto slot_of = [&](int pos) {
    const uint32_t t = st.slot + (uint32_t)pos;  // at most 12 + 16
    return t >= 2 * E_SLOTS ? t - 2 * E_SLOTS : t >= E_SLOTS ? t - E_SLOTS : t;
  };
  const auto phase_of = [&](int pos) {
    const uint32_t t = st.slot + (uint32_t)pos;
    return st.phase ^ (t >= 2 * E_SLOTS ? 0u : t >= E_SLOTS ? 1u : 0u);
  };
#pragma unroll
  for (int b = 0; b <= D1; ++b) {
    // the slices that this b is the first to use: in order of arrival they end with B_b
    const int from = b == 0 ? 0 : b_pos(b - 1, D0, D1) + 1;
    const int to = b_pos(b, D0, D1);
#pragma unroll
    for (int p = 0; p <= GD; ++p)
      if (from + p <= to && !mbar_wait_warp(&full[slot_of(from + p)], phase_of(from + p))) return false;
    tc_fence_after();
    const uint32_t sb = slot_of(to);
    const uint64_t bd = desc0 + (uint64_t)(sb * (E_TILE >> 4));
#pragma unroll
    for (int d = (D0 > b ? D0 : b); d <= D1; ++d) {
      const int buf = d - D0;
      const bool first = b == 0 && st.count[buf] == 0;
      if (first) {
        if (!mbar_wait_warp(&tempty[buf], ((st.used >> buf) & 1u) ^ 1u)) return false;
        st.used ^= 1u << buf;
        tc_fence_after();
      }
      const uint64_t ad = desc0 + (uint64_t)(slot_of(a_pos(d - b, D0, D1)) * (E_TILE >> 4));
      const uint32_t dt = tmem + (uint32_t)(buf * EBN);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        umma<TC_BF16>(dt, ad + 2u * k, bd + 2u * k, id, (!first || k > 0) ? 1u : 0u);
      if (d == b) {  // a = 0: the diagonal's last pair
        if (++st.count[buf] == chunk_blocks(d) || last_block) {
          umma_commit(&tfull[buf]);
          st.count[buf] = 0;
        }
      }
    }
    // A_(D1-b) and B_b were used for the last time
    umma_commit(&empty[slot_of(a_pos(D1 - b, D0, D1))]);
    umma_commit(&empty[sb]);
  }
  constexpr uint32_t LOADS = 2 * (D1 + 1);
  const uint32_t phase = phase_of(LOADS);
  st.slot = slot_of(LOADS);
  st.phase = phase;
  return true;
}

template <int GD>
__global__ void __launch_bounds__(E_THREADS, 1)
    k_gemm_emu(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ EmuOut out, int64_t M, int64_t N, int nkb, int Kp, int tiles_n,
               int n_tiles, int splits, const int* __restrict__ eA, const int* __restrict__ eB,
               int* __restrict__ err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + E_SLOTS * E_TILE);
  uint64_t* empty = full + E_SLOTS;
  uint64_t* tfull = empty + E_SLOTS;
  uint64_t* tempty = tfull + E_BUFS;
  uint64_t* done = tempty + E_BUFS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < E_SLOTS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < E_BUFS; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], E_EPI_WARPS);
    }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(E_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // work item -> output tile and its share [kb0, kb1) of the K blocks
  const auto item_of = [&](int item, int& m0, int& n0, int& kb0, int& kb1) {
    const int tile = item / splits, s = item - tile * splits;
    emu_tile(tile, n_tiles / tiles_n, tiles_n, m0, n0);
    kb0 = (int)((int64_t)nkb * s / splits);
    kb1 = (int)((int64_t)nkb * (s + 1) / splits);
    return s;
  };
  const int n_items = n_tiles * splits;

  if (warp == 0 && lane == 0) {
    uint32_t g = 0, s = 0, phase = 1;
    bool ok = true;
    const auto load = [&](const CUtensorMap* map, int x, int y) {
      if (!ok || !mbar_wait(&empty[s], phase)) {
        ok = false;
        return;
      }
      mbar_expect_tx(&full[s], E_TILE);
      tma_load_2d(smem + s * E_TILE, map, x, y, &full[s]);
      ++g;
      if (++s == E_SLOTS) {
        s = 0;
        phase ^= 1u;
      }
    };
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
      int m0, n0, kb0, kb1;
      item_of(item, m0, n0, kb0, kb1);
      for (int d0 = 0; d0 < SLICES && ok; d0 += GD) {
        const int d1 = d0 + GD - 1;
        for (int kb = kb0; kb < kb1 && ok; ++kb) {
          for (int a = d1; a > d0; --a) load(&tmA, a * Kp + kb * 64, m0);
          for (int b = 0; b <= d1; ++b) {
            if (b <= d0) load(&tmA, (d0 - b) * Kp + kb * 64, m0);
            load(&tmB, b * Kp + kb * 64, n0);
          }
        }
      }
    }
    if (!ok) atomicOr(err, 1);
    for (uint32_t q = (g > E_SLOTS ? g - E_SLOTS : 0); q < g; ++q)
      if (!mbar_wait(&full[q % E_SLOTS], (q / E_SLOTS) & 1u)) atomicOr(err, 1);
  } else if (warp == 1) {
    EmuIssue st;
    const uint32_t ring = smem_u32(smem);
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
      int m0, n0, kb0, kb1;
      item_of(item, m0, n0, kb0, kb1);
      const auto group = [&](auto d0) {
        for (int kb = kb0; kb < kb1 && ok; ++kb)
          ok = emu_issue_block<decltype(d0)::value, GD>(st, ring, tmem, full, empty, tfull, tempty,
                                                        kb == kb1 - 1);
      };
      group(std::integral_constant<int, 0>());
      if constexpr (GD == 2) group(std::integral_constant<int, 2>());
      group(std::integral_constant<int, 4>());
      if constexpr (GD == 2) group(std::integral_constant<int, 6>());
    }
    umma_commit(done);
    ok = mbar_wait_warp(done, 0) && ok;
    if (!ok && lane == 0) atomicOr(err, 1);
  } else if (warp >= 2) {
    const int qd = warp & 3;
    const int part = (warp - 2) >> 2;
    const uint32_t lane_t = tmem + ((uint32_t)(qd * 32) << 16) + part * E_EPI_COLS;
    uint32_t used = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
      int m0, n0, kb0, kb1;
      const int share = item_of(item, m0, n0, kb0, kb1);
      const int64_t row = (int64_t)m0 + qd * 32 + lane;
      const int64_t col0 = (int64_t)n0 + part * E_EPI_COLS;
      for (int d0 = 0; d0 < SLICES && ok; d0 += GD) {
        const int d1 = d0 + GD - 1;
        long long H[E_EPI_COLS];  // exact group sum, diagonal d1 at weight 1
#pragma unroll
        for (int j = 0; j < E_EPI_COLS; ++j) H[j] = 0;
        uint32_t count = 0;  // blocks in each buffer's partial sum, a byte each
        for (int kb = kb0; kb < kb1 && ok; ++kb) {
          for (int d = d0; d <= d1; ++d) {
            const int buf = d - d0;
            count += 1u << (8 * buf);
            if (((count >> (8 * buf)) & 255u) != ((uint32_t)(chunk_bytes() >> (8 * d)) & 255u) &&
                kb != kb1 - 1)
              continue;
            count &= ~(255u << (8 * buf));
            if (!mbar_wait(&tfull[buf], (used >> buf) & 1u)) {
              ok = false;
              break;
            }
            used ^= 1u << buf;
            tc_fence_after();
            const int weight = 1 << (SLICE_BITS * (d1 - d));
#pragma unroll
            for (int j = 0; j < E_EPI_COLS / 16; ++j) {
              uint32_t r[16];
              tmem_ld16(lane_t + buf * EBN + 16 * j, r);
              if (j == E_EPI_COLS / 16 - 1) {
                // the words are in registers: the buffer may be written again
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[buf]);
              }
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                // an exact integer of magnitude <= 2^24: converted exactly
                H[16 * j + i] += (long long)__float2int_rn(__uint_as_float(r[i])) * weight;
              }
            }
          }
        }
        if (!ok) break;
        // close the group: its sums become float64 with the scales folded in,
        // added to those of the groups before
        if (out.H) {
          long long* h = out.H + ((int64_t)share * (SLICES / GD) + d0 / GD) * out.slab + row * out.ldc;
#pragma unroll
          for (int j = 0; j < E_EPI_COLS; j += 4)
            if (row < M && col0 + j < N) {
              *reinterpret_cast<longlong2*>(h + col0 + j) = make_longlong2(H[j], H[j + 1]);
              *reinterpret_cast<longlong2*>(h + col0 + j + 2) = make_longlong2(H[j + 2], H[j + 3]);
            }
        } else if (row < M) {
          const bool final = d1 == SLICES - 1;
          const int k0 = -SLICE_BITS * (d1 + 2) + eA[row];
          double* c = out.C + row * out.ldc;
          double2* g = out.G + (size_t)blockIdx.x * (EBM * EBN / 2) + (threadIdx.x - 64);
#pragma unroll
          for (int h = 0; h < E_EPI_COLS / 4; ++h) {
            const int64_t col = col0 + 4 * h;
            const int4 eb = *reinterpret_cast<const int4*>(eB + col);
            double v[4], t[4];
            double2* gh = g + 2 * h * (32 * E_EPI_WARPS);
            v[0] = i64_ldexp(H[4 * h], k0 + eb.x);
            v[1] = i64_ldexp(H[4 * h + 1], k0 + eb.y);
            v[2] = i64_ldexp(H[4 * h + 2], k0 + eb.z);
            v[3] = i64_ldexp(H[4 * h + 3], k0 + eb.w);
            if (d0 > 0) {
              const double2 x = gh[0], y = gh[32 * E_EPI_WARPS];
              v[0] += x.x;
              v[1] += x.y;
              v[2] += y.x;
              v[3] += y.y;
            }
            if (!final) {
              gh[0] = make_double2(v[0], v[1]);
              gh[32 * E_EPI_WARPS] = make_double2(v[2], v[3]);
            } else {
              if (out.subtract) {
                load_row4(c, col, N, out.vec, t);
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = t[i] - v[i];
              }
              store_row4(c, col, N, out.vec, v);
            }
          }
        }
      }
    }
    if (!ok) atomicOr(err, 1);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(E_TMEM_COLS));
  }
}

// C = (or -=) the product whose group sums lie in `splits` shares: the shares
// are added as integers, exactly, so the bits do not depend on their number.
template <int GD>
__global__ void k_emu_combine(const long long* __restrict__ H, int splits, int64_t slab, int64_t ldh,
                              int64_t N, const int* __restrict__ eA, const int* __restrict__ eB,
                              double* __restrict__ C, int64_t ldc, int subtract) {
  constexpr int GROUPS = SLICES / GD;
  const int64_t r = blockIdx.y;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < N; c += (int64_t)gridDim.x * blockDim.x) {
    long long h[GROUPS] = {};
#pragma unroll 4
    for (int s = 0; s < splits; ++s)
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) h[g] += H[((int64_t)s * GROUPS + g) * slab + r * ldh + c];
    double t = 0.0;
#pragma unroll
    for (int g = 0; g < GROUPS; ++g) {
      const double v = i64_ldexp(h[g], -SLICE_BITS * (GD * (g + 1) + 1) + eA[r] + eB[c]);
      t = g == 0 ? v : v + t;
    }
    double* dst = C + r * ldc + c;
    *dst = subtract ? *dst - t : t;
  }
}

// ---------------------------------------------------------------------------
// Slicing
// ---------------------------------------------------------------------------
// Biased exponent field of |x| (0 for zero and subnormals): comparing the
// magnitude bits as integers orders doubles by size.
__device__ __forceinline__ unsigned long long mag_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

__device__ __forceinline__ int exponent_of_max(unsigned long long mbits) {
  const int E = (int)(mbits >> 52);
  return E == 0 ? 0 : E - 1022;  // |x| < 2^(E - 1022) for every x of the row
}

// x * 2^(56 - e) rounded to the nearest integer, from the IEEE bits (integer
// arithmetic only). |x| < 2^e, so |X| <= 2^56. Subnormal inputs count as 0.
__device__ __forceinline__ long long fixed56(double x, int e) {
  const long long bits = __double_as_longlong(x);
  const int E = (int)((bits >> 52) & 0x7FF);
  if (E == 0) return 0;
  const long long mant = (bits & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int sh = E - 1075 + 56 - e;  // value = mant * 2^(E - 1075)
  long long X;
  if (sh >= 0) X = mant << sh;  // sh <= 3 since |x| < 2^e
  else if (sh < -62) X = 0;
  else X = (mant + (1ll << (-sh - 1))) >> (-sh);
  return bits < 0 ? -X : X;
}

// Balanced base-128 digits of X: X = sum_p d_p 128^(7 - p); d_1..d_7 in
// [-64, 63], d_0 in [-128, 128]; slice p of the operand is the integer d_p
// (exact in bf16) and stands for d_p 2^(-7 (p + 1)) 2^e. Eight consecutive
// columns of a row are cut together and stored 16 bytes per slice. An integer
// |d| < 2^22 added to the bits of 1.5 2^23 is that float plus d, so the
// difference is (float)d without a conversion; its upper half is the bf16.
__device__ __forceinline__ void store_slices8(__nv_bfloat16* dst, int64_t base, int64_t Kp,
                                              const long long (&Xs)[8]) {
  uint32_t w[SLICES][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    long long X0 = Xs[2 * i], X1 = Xs[2 * i + 1];
#pragma unroll
    for (int p = SLICES - 1; p >= 0; --p) {
      int d0 = (int)X0, d1 = (int)X1;
      if (p > 0) {
        d0 = (int)(((uint32_t)d0 + 64u) & 127u) - 64;
        d1 = (int)(((uint32_t)d1 + 64u) & 127u) - 64;
        X0 = (X0 - d0) >> SLICE_BITS;
        X1 = (X1 - d1) >> SLICE_BITS;
      }
      const float f0 = __int_as_float(0x4B400000 + d0) - 12582912.0f;
      const float f1 = __int_as_float(0x4B400000 + d1) - 12582912.0f;
      w[p][i] = __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
    }
  }
#pragma unroll
  for (int p = 0; p < SLICES; ++p)
    *reinterpret_cast<uint4*>(dst + base + (int64_t)p * Kp) = make_uint4(w[p][0], w[p][1], w[p][2], w[p][3]);
}

// Rows whose K index is contiguous: one block per row finds the row's largest
// exponent, writes it to e[r] and cuts the row (read a second time from L1
// where it is longer than eight columns per thread).
template <typename S>
__global__ void __launch_bounds__(256) k_slice_rows(SplitView v, int* __restrict__ e,
                                                    __nv_bfloat16* __restrict__ dst, int64_t Kp,
                                                    int vec) {
  __shared__ unsigned long long sh[8];
  const int64_t r = blockIdx.x, r0 = r / v.n1, r1 = r - r0 * v.n1;
  const S* src = reinterpret_cast<const S*>(v.src) + r0 * v.s0 + r1 * v.s1;
  const auto load = [&](int64_t k, double (&x)[8]) {
    if (vec && k + 8 <= v.K) {
      S q[8];
      load_eight(src + k, q);
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = (double)q[i];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = k + i < v.K ? (double)src[k + i] : 0.0;
    }
  };
  const int64_t step = 8 * (int64_t)blockDim.x, first = 8 * (int64_t)threadIdx.x;
  double x[8];
  unsigned long long m = 0;
  if (first < Kp) load(first, x);
#pragma unroll
  for (int i = 0; i < 8; ++i) m = first < Kp ? max(m, mag_bits(x[i])) : m;
  for (int64_t k = first + step; k < Kp; k += step) {
    double y[8];
    load(k, y);
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, mag_bits(y[i]));
  }
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) m = max(m, sh[i]);
  const int ex = exponent_of_max(m);
  if (threadIdx.x == 0) e[r] = ex;
  for (int64_t k = first; k < Kp; k += step) {
    if (k != first) load(k, x);
    long long X[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) X[i] = fixed56(x[i], ex);
    store_slices8(dst, r * SLICES * Kp + k, Kp, X);
  }
}

// Rows that are adjacent in memory (K strided), first pass: row maxima of the
// magnitude bits, 64 rows x a chunk of K per block, neighbouring threads on
// neighbouring rows, partial maxima combined with atomicMax into m[r].
constexpr int ROWMAX_KCHUNK = 256;
template <typename S>
__global__ void __launch_bounds__(256) k_rowmax_strided(SplitView v, unsigned long long* __restrict__ m) {
  __shared__ unsigned long long sh[4][64];
  const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
  const int64_t r = (int64_t)blockIdx.x * 64 + tx, rr = r < v.rows ? r : 0;
  const int64_t r0 = rr / v.n1, r1 = rr - r0 * v.n1;
  const S* src = reinterpret_cast<const S*>(v.src) + r0 * v.s0 + r1 * v.s1;
  const int64_t k0 = (int64_t)blockIdx.y * ROWMAX_KCHUNK, k1 = min(k0 + (int64_t)ROWMAX_KCHUNK, v.K);
  unsigned long long a = 0;
#pragma unroll 8
  for (int64_t k = k0 + ty; k < k1; k += 4) a = max(a, mag_bits((double)src[k * v.sk]));
  sh[ty][tx] = a;
  __syncthreads();
  if (ty == 0 && r < v.rows) {
    for (int i = 1; i < 4; ++i) a = max(a, sh[i][tx]);
    atomicMax(&m[r], a);
  }
}

// Second pass: tiles of 64 rows x 64 columns read along the rows, brought to
// fixed point, and cut along the columns through shared memory. The blocks of
// the first column tile also write the exponents.
template <typename S>
__global__ void __launch_bounds__(256) k_slice_transpose(SplitView v,
                                                         const unsigned long long* __restrict__ m,
                                                         int* __restrict__ e,
                                                         __nv_bfloat16* __restrict__ dst, int64_t Kp) {
  __shared__ long long tile[64][65];
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
    const int ex = exponent_of_max(m[rr]);
    if (blockIdx.y == 0 && ty == 0 && r < v.rows) e[r] = ex;
#pragma unroll
    for (int j = 0; j < 16; ++j) tile[ty + 4 * j][tx] = fixed56((double)x[j], ex);
  }
  __syncthreads();
  for (int u = threadIdx.x; u < 512; u += 256) {
    const int row = u >> 3, g = 8 * (u & 7);
    if (r_base + row >= v.rows) continue;
    long long X[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) X[i] = tile[g + i][row];
    store_slices8(dst, (r_base + row) * SLICES * Kp + k_base + g, Kp, X);
  }
}

// Traffic: 8 bytes read (twice for strided rows) and 16 written per value.
template <typename S>
osmps_status slice_operand(osmps_ctx* ctx, const SplitView& v, int64_t Kp, int* e,
                           __nv_bfloat16* dst, cudaStream_t s) {
  if (v.rows <= 0) return OSMPS_OK;
  if (v.sk == 1) {
    if (v.rows > 2147483647ll) return set_error(OSMPS_ESHAPE, "emulated GEMM: too many rows");
    constexpr int64_t PER = 16 / sizeof(S);
    const bool vec = (reinterpret_cast<uintptr_t>(v.src) & 15) == 0 && v.s0 % PER == 0 &&
                     (v.n1 == 1 || v.s1 % PER == 0);
    const int threads = (int)std::min<int64_t>(256, round_up(cdiv(Kp, 8), 32));
    k_slice_rows<S><<<(unsigned)v.rows, threads, 0, s>>>(v, e, dst, Kp, vec ? 1 : 0);
    note_launch();
  } else {
    if (cdiv(Kp, 64) > 65535 || cdiv(v.K, ROWMAX_KCHUNK) > 65535)
      return set_error(OSMPS_ESHAPE, "emulated GEMM: K too large");
    osmps_status st = OSMPS_OK;
    auto* mx = (unsigned long long*)ws_get(ctx, SLOT_EMU_MAX, (size_t)v.rows * 8, s, &st);
    if (!mx) return st;
    OSMPS_CUDA(cudaMemsetAsync(mx, 0, (size_t)v.rows * 8, s));
    const dim3 g1((unsigned)cdiv(v.rows, 64), (unsigned)std::max<int64_t>(1, cdiv(v.K, ROWMAX_KCHUNK)));
    k_rowmax_strided<S><<<g1, 256, 0, s>>>(v, mx);
    note_launch();
    const dim3 grid((unsigned)cdiv(v.rows, 64), (unsigned)cdiv(Kp, 64));
    k_slice_transpose<S><<<grid, 256, 0, s>>>(v, mx, e, dst, Kp);
    note_launch();
  }
  OSMPS_LAUNCH_CHECK();
  return OSMPS_OK;
}

// Tiles of shares at most, per SM: the scratch of the kernel then has one size
// for all products up to K = 2^17 (two planes of two tiles for each SM, 80 MB)
// and never grows after the first (a growing one would be refused inside a
// graph capture).
constexpr int E_SLAB_WAVES = 2;

// Shares of K per output tile. A tile takes its K blocks one after the other
// on one SM, so a product of few tiles leaves SMs idle; its K blocks are then
// shared out, the shares' integer sums added by a second kernel.
// Taken by estimated clocks: 36 slice pairs of 380 per K block, 8000 per tile for
// its drains and sums, and for the shares one more launch and 16 bytes per group
// and element at 2600 bytes a clock. Kernels with one share and with the shares
// taken: 128 x 128 x 2048 234 and 49 us, 512 x 512 x 2048 231 and 56, 1024 x 1024
// x 2048 240 and 140, 381 x 1905 x 1000 130 and 68.
int emu_splits(int64_t M, int64_t N, int64_t n_tiles, int64_t nkb, int groups, int sms) {
  if (M > 65535) return 1;
  int best = 1;
  double t_best = 0;
  for (int s = 1; s <= 8 && (s == 1 || (nkb / s >= 2 && n_tiles * s <= E_SLAB_WAVES * sms)); ++s) {
    double t = (double)cdiv(n_tiles * s, sms) * ((double)cdiv(nkb, s) * 36 * 380 + 8000);
    if (s > 1) t += (double)s * M * N * 16 * groups / 2600 + 6000;
    if (s == 1 || t < t_best) {
      best = s;
      t_best = t;
    }
  }
  return best;
}

}  // namespace

osmps_status gemm_emu(osmps_ctx* ctx, const SplitView& a, const SplitView& b, int64_t M,
                      int64_t N, int64_t K, double* C, int64_t ldc, cudaStream_t s,
                      bool subtract, bool small_on_dmma) {
  if (M <= 0 || N <= 0) return OSMPS_OK;
  if (K <= 0 || a.rows != M || b.rows != N || a.K != K || b.K != K)
    return set_error(OSMPS_ESHAPE, "gemm_emu: inconsistent operand views");
  // Small products go to the float64 DMMA kernel, which is float64-accurate
  // too: the emulation costs 52 to 62 us even for a few tiles (three launches,
  // 36 slice pairs; 128x128x64: 53, 300x300x340: 62), so whatever the DMMA
  // kernel finishes sooner runs there.
  if (small_on_dmma && a.n1 == 1 && b.n1 == 1 && !a.src_f32 && !b.src_f32 && gemm_f64_us(M, N, K) < 56.0) {
    GemmF64 g;
    g.M = M; g.N = N; g.K = K;
    g.A = static_cast<const double*>(a.src); g.sam = a.s0; g.sak = a.sk;
    g.B = static_cast<const double*>(b.src); g.sbk = b.sk; g.sbn = b.s0;
    g.C = C; g.scm = ldc; g.scn = 1;
    if (subtract) {
      g.alpha = -1.0;
      g.beta = 1.0;
    }
    return gemm_f64(g, s);
  }
  const int64_t Kp = round_up(K, 64);
  if (SLICES * Kp > ((int64_t)1 << 31) || cdiv(M, EBM) * cdiv(N, EBN) > ((int64_t)1 << 31))
    return set_error(OSMPS_ESHAPE, "gemm_emu: dimensions exceed the supported range");
  osmps_status st = OSMPS_OK;
  auto* sa = (__nv_bfloat16*)ws_get(ctx, SLOT_EMU_A, (size_t)M * SLICES * Kp * 2, s, &st);
  if (!sa) return st;
  auto* sb = (__nv_bfloat16*)ws_get(ctx, SLOT_EMU_B, (size_t)N * SLICES * Kp * 2, s, &st);
  if (!sb) return st;
  int* ex = (int*)ws_get(ctx, SLOT_EMU_EXP, (size_t)(M + N + 64 + EBN) * sizeof(int), s, &st);
  if (!ex) return st;
  int* eA = ex;
  int* eB = ex + ((M + 63) / 64) * 64;
  OSMPS_TRY(a.src_f32 ? slice_operand<float>(ctx, a, Kp, eA, sa, s) : slice_operand<double>(ctx, a, Kp, eA, sa, s));
  OSMPS_TRY(b.src_f32 ? slice_operand<float>(ctx, b, Kp, eB, sb, s) : slice_operand<double>(ctx, b, Kp, eB, sb, s));
  CUtensorMap ma, mb;
  OSMPS_TRY(tc_make_map(&ma, sa, TC_BF16, M, SLICES * Kp, EBM));
  OSMPS_TRY(tc_make_map(&mb, sb, TC_BF16, N, SLICES * Kp, EBN));
  const int tiles_n = (int)cdiv(N, EBN);
  const int n_tiles = tiles_n * (int)cdiv(M, EBM);
  const int nkb = (int)(Kp / 64);
  // diagonals per exact int64 group: four while a group sum stays below 2^53
  // (|I_d| < (d + 1) K 2^14 with slice digits of at most 2^7 and 2^6), else two
  const int groups = Kp <= ((int64_t)1 << 17) ? 2 : 4;
  const int splits = emu_splits(M, N, n_tiles, nkb, groups, ctx->sm_count);
  const int grid = std::min(n_tiles * splits, ctx->sm_count);
  EmuOut out{C, nullptr, nullptr, ldc, 0, subtract ? 1 : 0, 0};
  const size_t tile_sums = (size_t)ctx->sm_count * EBM * EBN;
  void* scratch = ws_get(ctx, SLOT_EMU_PART, groups * E_SLAB_WAVES * tile_sums * 8, s, &st);
  if (!scratch) return st;
  if (splits > 1) {
    out.H = static_cast<long long*>(scratch);
    out.ldc = round_up(N, 4);
    out.slab = M * out.ldc;
  } else {
    out.G = static_cast<double2*>(scratch);
    out.vec = (reinterpret_cast<uintptr_t>(C) & 15) == 0 && ldc % 2 == 0;
  }
  const auto run = [&](auto kernel, cudaError_t configured) -> osmps_status {
    OSMPS_CUDA(configured);
    kernel<<<grid, E_THREADS, E_SMEM, s>>>(ma, mb, out, M, N, nkb, (int)Kp, tiles_n, n_tiles, splits, eA, eB,
                                           ctx->dev_flags);
    note_launch();
    return OSMPS_OK;
  };
  const int ph = prof_begin(s);
  // thread-safe one-time setups (function-local static initialisation)
  if (groups == 2) {
    static const cudaError_t configured =
        cudaFuncSetAttribute(k_gemm_emu<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)E_SMEM);
    OSMPS_TRY(run(k_gemm_emu<4>, configured));
  } else {
    static const cudaError_t configured =
        cudaFuncSetAttribute(k_gemm_emu<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)E_SMEM);
    OSMPS_TRY(run(k_gemm_emu<2>, configured));
  }
  if (splits > 1) {
    const dim3 cg((unsigned)std::min<int64_t>(cdiv(N, 256), 64), (unsigned)M);
    const auto combine = groups == 2 ? k_emu_combine<4> : k_emu_combine<2>;
    combine<<<cg, 256, 0, s>>>(out.H, splits, out.slab, out.ldc, N, eA, eB, C, ldc, subtract ? 1 : 0);
    note_launch();
  }
  OSMPS_LAUNCH_CHECK();
  const double logical = 2.0 * (double)M * (double)N * (double)K;
  prof_end(ph, s, OSMPS_KERNEL_GEMM_EMU, logical, (double)(SLICES * (SLICES + 1) / 2) * logical);
  return OSMPS_OK;
}

}  // namespace osmps

using namespace osmps;

extern "C" osmps_status osmps_dgemm_emu(osmps_ctx* ctx, const double* A, const double* B, double* C,
                                        int64_t M, int64_t N, int64_t K, void* stream) {
  clear_error();
  if (!ctx || !A || !B || !C) return set_error(OSMPS_EINVAL, "osmps_dgemm_emu: null argument");
  if (C == A || C == B) return set_error(OSMPS_EINVAL, "osmps_dgemm_emu: C aliases an input");
  if (M <= 0 || N <= 0 || K <= 0) return set_error(OSMPS_ESHAPE, "osmps_dgemm_emu: dimensions");
  OSMPS_CUDA(cudaSetDevice(ctx->device));
  CtxScope scope_(ctx);
  SplitView a;
  a.src = A; a.rows = M; a.K = K; a.s0 = K; a.sk = 1;
  SplitView b;  // row n of the B operand = column n of B
  b.src = B; b.rows = N; b.K = K; b.s0 = 1; b.sk = N;
  return gemm_emu(ctx, a, b, M, N, K, C, N, (cudaStream_t)stream, false, false);
}
