// Householder reduction of a symmetric matrix to tridiagonal form,
// T = Q^T A Q (the first step of the float64 eigendecomposition used by the
// split, Sec. 2 Eq. AAD_ULLUD), with the reflectors stored as LAPACK's dsytrd
// (lower) stores them: Q = H(0) ... H(n-2), H(j) = I - tau_j v_j v_j^T,
// v_j = (0, .., 0, 1 at j+1, A[j+2.., j]).
//
// Blocked as in LAPACK's dlatrd: panels of NB columns. Inside a panel, column
// j is brought up to date with the panel's earlier reflectors
// (x = A e_j - V W^T e_j - W V^T e_j), its reflector is formed, and
//   w = tau (A22 v - W y - V z) + alpha2 v,   y = V^T v,  z = W^T v,
//   alpha2 = -(tau^2/2) (v^T A22 v - 2 y^T z)
// with A22 the trailing matrix as it stood at the start of the panel. After
// the panel the trailing block is updated, A22 -= V W^T + W V^T, by the
// float64-accurate emulated tensor-core GEMM, subtracting in its epilogue.
// The matrix is kept full (both triangles), so row r of the trailing block is
// contiguous; the reflectors overwrite column j below the subdiagonal (row j
// of the row-major view), which later columns never read.
//
// A panel is one cooperative launch, its rows dealt to the blocks round robin;
// each block keeps its rows of V and W in shared memory. What bounds a column
// below m of about 1000 is not its float64 work (A22 v: under 2 us below m = 700,
// 13 at 2048, where the float64 pipe issues for two thirds of the column, 16.7 us
// at m = 1750 with the rows in L2 or in shared memory alike) but the way of its
// numbers between the blocks and the dependent float64 chains around it, so the
// column is arranged for few exchanges off the critical
// path and none through a barrier:
//   * v = e_(j+1) + inv u with u the column below j + 1 and inv known only
//     after sigma = u^T u, a square root and two divisions (2000 clocks, formed
//     by one warp of every block from its own copy of u beside the rest):
//     everything linear in v is formed from u. A22 v = A e_(j+1) + inv A22 u,
//     y = V^T e_(j+1) + inv V^T u, v^T A22 v = A_(j+1)(j+1) + 2 inv s1 + inv^2 s2
//     with s1 = e_(j+1)^T A u and s2 = u^T A22 u. Only s2 needs the product
//     A22 u; the other 2 jj + 1 sums are on their way while it runs, and what
//     is left to do when s2 arrives is four operations per row.
//   * every number crosses the GPU as a 16-byte word of value and column
//     number, written and read in one access; a reader polls for the number,
//     so an exchange is one store and one load, not a fence, an atomic, a wait
//     and a load. Words alternate between two buffers: a block can publish
//     column j + 2 only after it has read every block's column j + 1, which a
//     block publishes after its last read of column j.
//   * the 2 jj + 1 sums: up to 32 blocks, every block adds up all partial
//     sums itself; beyond, one warp per sum adds it up and publishes it.
//   * row j + 1 of W (needed by every block for the next column) is published
//     by its owner a column ahead; row j + 1 of V every block has.
// Polls are bounded: after ~2 s a block records the failure in the error
// flag and leaves, and later panels leave at once.
// Measured per column, averaged over a reduction, against two grid barriers
// per column with every block adding up all partial sums: n = 128 12.4 -> 5.7
// us, 512 13.8 -> 7.8, 1024 15.0 -> 8.0, 2048 18.9 -> 11.2.
#include <cooperative_groups.h>

#include <cfloat>
#include <cmath>

#include "common.cuh"
#include "tagged.cuh"

namespace osmps {
namespace {

constexpr int NB = 32;            // panel width (one lane per earlier reflector)
constexpr int ROW_WARPS = 8;      // warps that share the block's rows
constexpr int ROW_THREADS = 32 * ROW_WARPS;
constexpr int ST_THREADS = ROW_THREADS + 64;  // and one warp each for sums and scalars
constexpr int MAXLOC = 64;        // rows per block at most
constexpr int MAXSUM = 64;        // 2 jj + 1 < 64 sums
constexpr int LINE = 8;             // words per 128-byte line
constexpr int DIRECT_G = 32;      // blocks up to which every block adds up all partial sums

struct SytrdArgs {
  double* A;         // n x n, full symmetric (row r contiguous)
  int n, k0, nbp;    // panel [k0, k0 + nbp)
  double* d;         // diagonal of T
  double* e;         // off-diagonal of T
  double* tau;       // reflector scalars
  double* Vp;        // panel reflectors, column-major NB x n: Vp[q * n + r]
  double* Wp;        // panel w vectors, same layout
  // tagged words, two buffers each (column parity), laid out so that no
  // 128-byte line holds words of two blocks (a line that several blocks write
  // while all poll it moves between the two dies' caches: gathering a column
  // of 1024 entries from 152 blocks took 4 us in row order)
  ulonglong2* X;     // [2][G][lw] column entries, block by block
  ulonglong2* Wn;    // [2][NB] row j + 1 of W
  ulonglong2* part;  // [2][G][MAXSUM] partial sums
  ulonglong2* R;     // [2][MAXSUM][LINE] sums (G > DIRECT_G)
  ulonglong2* T2;    // [2][G][LINE] partial u^T A22 u
  int lw;            // words per block in X: its rows, rounded up to whole lines
  const int* emax;   // largest biased exponent of the whole matrix
  int sa;            // row stride of the block's rows in shared memory (0: they stay in L2)
  int* err;          // bit 0: a poll gave up
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// SA: the block's rows of A22 are kept in shared memory for the whole panel
// (loaded once; a column then waits for no L2 round trip). VEC: rows in global
// memory start on 16-byte boundaries.
template <bool VEC, bool SA>
__global__ void __launch_bounds__(ST_THREADS, 1) k_sytrd_panel(SytrdArgs a) {
  extern __shared__ __align__(16) double su[];  // u over rows [0, n + 64): zero up to j + 1 and past n
  double* sA = su + ((a.n + 64 + 1) & ~1);      // (SA) rows of A, columns k0 ..
  __shared__ double sV[MAXLOC][NB];         // this block's rows of V and W
  __shared__ double sW[MAXLOC][NB];
  __shared__ double sVp[NB][NB + 1];        // V_q[k0 + 1 + i]
  __shared__ double spart[ROW_WARPS][MAXLOC];
  __shared__ double st[MAXLOC];             // this block's rows of A22 u
  __shared__ double sAc[MAXLOC];            // A[r][j + 1]
  __shared__ double sR[MAXSUM];             // V^T u | W^T u | s1
  __shared__ double sVn[NB], sWn[NB];       // V_q[j + 1], W_q[j + 1]
  __shared__ double sa0, sAd, ss2;          // x[j + 1], A[j + 1][j + 1], s2
  __shared__ double sti[2];                 // tau, inv
  __shared__ int sE[2];                     // largest biased exponent of the column, by parity
  __shared__ double sc[3];                  // alpha2 = sc[0] + sc[1] s2, w[j + 1] = sc[2] + alpha2
  const int n = a.n, k0 = a.k0, G = gridDim.x, b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool direct = G <= DIRECT_G;
  const int amax = *a.emax - 1023;
  const int cnt = k0 + b < n ? (n - k0 - b + G - 1) / G : 0;  // rows k0 + b, k0 + b + G, ...
  if (__syncthreads_or(tid == 0 ? *(volatile int*)a.err & 1 : 0)) return;  // an earlier panel failed
  // per-row work: eight or four neighbouring threads per row, so that up to 32
  // rows lie in warps 0-3, one per sub-partition (a float64 instruction takes
  // 64 clocks of its sub-partition whatever number of its lanes is active)
  const int lg = cnt <= 16 ? 3 : 2, tpr = 1 << lg;
  const int rloc = tid >> lg, sub = tid & (tpr - 1);
  const bool row_warp = tid < ROW_THREADS && ((warp * 32) >> lg) < cnt;
  const bool has_row = tid < ROW_THREADS && rloc < cnt;
  const int row = k0 + b + G * rloc;
  for (int k = tid; k < n + 64; k += ST_THREADS) su[k] = 0.0;
  if (tid < 2) sE[tid] = 0;
  __syncthreads();
  if (SA) {
    for (int loc = warp; loc < cnt; loc += ST_THREADS / 32) {
      const double* src = a.A + (size_t)(k0 + b + G * loc) * n + k0;
      for (int k = lane; k < a.sa; k += 32) sA[loc * a.sa + k] = k0 + k < n ? src[k] : 0.0;
    }
    __syncthreads();
  }
  double xv = 0.0, ac = 0.0;  // x[row] and A[row][j + 1]
  if (has_row) {
    xv = a.A[(size_t)k0 * n + row];
    if (k0 + 1 < n) ac = a.A[(size_t)row * n + k0 + 1];
  }
  for (int jj = 0; jj < a.nbp; ++jj) {
    const int j = k0 + jj, NV = 2 * jj + 1;
    const uint64_t tag = (uint64_t)j + 1;
    ulonglong2* X = a.X + (size_t)(j & 1) * G * a.lw;
    ulonglong2* Wn = a.Wn + (j & 1) * NB;
    ulonglong2* part = a.part + (size_t)(j & 1) * MAXSUM * G;
    ulonglong2* R = a.R + (j & 1) * MAXSUM * LINE;
    ulonglong2* T2 = a.T2 + (size_t)(j & 1) * G * LINE;
    // ---- publish this block's rows of the column, and row j + 1 of W
    if (has_row && row >= j) {
      if (sub == 0) {
        if (jj == 0) put_word(X + b * a.lw + rloc, xv, tag);  // (else published as soon as it was known)
        if (row == j) a.d[j] = xv;
        sAc[rloc] = ac;
      }
      if (row == j + 1)
        for (int q = sub; q < jj; q += tpr) put_word(Wn + q, sW[rloc][q], tag);
    }
    if (j == n - 1) break;  // the last column has nothing below its diagonal
    // ---- gather the whole column
    bool bad = false;
    int em = 0;
    for (int w0 = tid; w0 < G * a.lw; w0 += 4 * ST_THREADS) {
      const ulonglong2* p[4];
      double v[4];
      int r[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int w = w0 + i * ST_THREADS, bb = w / a.lw;
        r[i] = k0 + bb + G * (w - bb * a.lw);
        p[i] = bb < G && r[i] > j && r[i] < n ? X + w : nullptr;
      }
      bad |= !get_words<4>(p, tag, v);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (p[i]) {
          em = max(em, (__double2hiint(v[i]) >> 20) & 0x7FF);
          if (r[i] == j + 1) sa0 = v[i];
          else su[r[i]] = v[i];
        }
    }
    if (tid == 0) su[j + 1] = 0.0;
    em = __reduce_max_sync(0xffffffffu, em);
    if (lane == 0) atomicMax(&sE[j & 1], em);
    double vpan = 0.0;  // (warp 9) V row of lane's panel row, before scaling
    if (warp == 9) {
      const ulonglong2* p[1] = {lane < jj ? Wn + lane : nullptr};
      double v[1];
      bad |= !get_words<1>(p, tag, v);
      sWn[lane] = lane < jj ? v[0] : 0.0;
      sVn[lane] = lane < jj ? sVp[lane][jj] : 0.0;
      if (lane == 0) sAd = a.A[(size_t)(j + 1) * n + j + 1];
    }
    if (__syncthreads_or(bad)) {
      if (bad) atomicOr(a.err, 1);
      return;
    }
    // u is not scaled, so A22 u and s2 hold |A| |u| and |A| |u|^2, which can leave
    // the float64 range where |A| does not. A column is brought under 2^-7 (|u| < 1
    // up to 8192 rows) by a power of two where its largest entry 2^ec and the
    // matrix's 2^amax (|A22| <= n 2^(amax + 1) throughout, the reduction being
    // orthogonal) say 2 ec + amax > 960, i.e. n^2 |u|^2 |A| could pass 2^1023, and
    // where ec < -200. v, tau and everything below stay as they are, inv absorbs
    // the factor, beta gets it back. (Always scaling costs 6% to 11% a column on
    // random matrices: 2048 13.0 -> 14.5 us.)
    const int em_all = sE[j & 1], ec = em_all - 1023, ex = ec + 8;
    const bool scaled = (2 * ec + amax > 960 || ec < -200) && em_all > 0 && em_all < 0x7FF;  // the same in every block
    if (scaled) {
      for (int r = j + 2 + tid; r < n; r += ST_THREADS) su[r] = scalbn(su[r], -ex);
      if (tid == 0) sa0 = scalbn(sa0, -ex);
      __syncthreads();
    }
    if (tid == 0) sE[(j + 1) & 1] = 0;
    const double ur = has_row && row > j + 1 ? su[row] : 0.0;
    if (warp == 9 && k0 + 1 + lane < n) vpan = su[k0 + 1 + lane];
    const int loc0 = j + 1 > k0 + b ? (j + 1 - k0 - b + G - 1) / G : 0;  // first row >= j + 1
    double Cr = 0.0, acn = 0.0;
    if (tid < ROW_THREADS) {
      // ---- partial sums over this block's rows, four threads to a sum
      {
        const int c = tid >> 2, s4 = tid & 3;
        double p = 0.0;
        if (c < NV) {
          const double* f = c < jj ? &sV[0][c] : c < 2 * jj ? &sW[0][c - jj] : sAc;
          const int fs = c < 2 * jj ? NB : 1;
#pragma unroll 4
          for (int loc = loc0 + s4; loc < cnt; loc += 4) p = fma(f[loc * fs], su[k0 + b + G * loc], p);
        }
        p += __shfl_xor_sync(0xffffffffu, p, 1);
        p += __shfl_xor_sync(0xffffffffu, p, 2);
        if (c < NV && s4 == 0) put_word(part + (size_t)b * MAXSUM + c, p, tag);
      }
      if (has_row && j + 2 < n)  // the next column's
        acn = SA ? sA[rloc * a.sa + j + 2 - k0] : a.A[(size_t)row * n + j + 2];
      // ---- A22 u: each warp takes every eighth chunk of 64 columns for all
      // rows (so the warps, and the four float64 pipes behind them, have
      // equal shares), eight rows at a time
      const int kbeg = (j + 2) & ~1, nch = (n - kbeg + 63) >> 6;
      for (int g0 = loc0; g0 < cnt; g0 += 8) {
        double acc[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[i] = 0.0;
        const double* rp = SA ? sA + g0 * a.sa - k0 : a.A + (size_t)(k0 + b + G * g0) * n;
        const size_t rs = SA ? (size_t)a.sa : (size_t)G * n;
        const int rows = cnt - g0;  // (the same for the whole block)
#pragma unroll 2
        for (int ch = warp; ch < nch; ch += ROW_WARPS) {
          const int k = kbeg + 64 * ch + 2 * lane;
          const double u0 = su[k], u1 = su[k + 1];
          double2 x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            x[i] = make_double2(0.0, 0.0);
            if (i < rows) {
              if (VEC || SA) {
                if (k < n) x[i] = *reinterpret_cast<const double2*>(rp + i * rs + k);
              } else {
                if (k < n) x[i].x = rp[i * rs + k];
                if (k + 1 < n) x[i].y = rp[i * rs + k + 1];
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i < rows) acc[i] = fma(x[i].x, u0, fma(x[i].y, u1, acc[i]));
        }
        if (warp >= nch) {  // no columns left for this warp
          if (lane < 8 && lane < rows) spart[warp][g0 + lane] = 0.0;
          continue;
        }
        // eight sums by a butterfly that halves the live values
        const bool b16 = lane & 16, b8 = lane & 8, b4 = lane & 4;
        double h4[4], h2[2], h1;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          h4[i] = (b16 ? acc[i + 4] : acc[i]) + __shfl_xor_sync(0xffffffffu, b16 ? acc[i] : acc[i + 4], 16);
#pragma unroll
        for (int i = 0; i < 2; ++i)
          h2[i] = (b8 ? h4[i + 2] : h4[i]) + __shfl_xor_sync(0xffffffffu, b8 ? h4[i] : h4[i + 2], 8);
        h1 = (b4 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, b4 ? h2[0] : h2[1], 4);
        h1 += __shfl_xor_sync(0xffffffffu, h1, 2);
        h1 += __shfl_xor_sync(0xffffffffu, h1, 1);
        const int loc = g0 + (b16 ? 4 : 0) + (b8 ? 2 : 0) + (b4 ? 1 : 0);
        if ((lane & 3) == 0 && loc < cnt) spart[warp][loc] = h1;
      }
      asm volatile("bar.sync 1, %0;" ::"n"(ROW_THREADS) : "memory");
      if (warp == 0) {
        double s2 = 0.0;
        for (int loc = loc0 + lane; loc < cnt; loc += 32) {
          double t0 = spart[0][loc] + spart[1][loc], t1 = spart[2][loc] + spart[3][loc];
          t0 += spart[4][loc] + spart[5][loc];
          t1 += spart[6][loc] + spart[7][loc];
          st[loc] = t0 + t1;
          s2 = fma(t0 + t1, su[k0 + b + G * loc], s2);
        }
        for (int o = cnt <= 16 ? 8 : 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        if (lane == 0) put_word(T2 + b * LINE, s2, tag);
      }
      // ---- C_r = sum_q V_q[r] W_q[j+1] + W_q[r] V_q[j+1]
      if (row_warp) {  // warps without rows keep off the float64 pipe
        double c2 = 0.0;
#pragma unroll 4
        for (int q = sub; q < jj; q += tpr) {
          Cr = fma(sV[rloc][q], sWn[q], Cr);
          c2 = fma(sW[rloc][q], sVn[q], c2);
        }
        Cr += c2;
        for (int o = tpr >> 1; o > 0; o >>= 1) Cr += __shfl_xor_sync(0xffffffffu, Cr, o);
      }
      if (direct && warp >= 4) {  // all sums from the partial sums, two threads to a sum
        const int c = (tid - 128) >> 1, s2 = tid & 1;
        double p = 0.0;
        for (int b0 = s2; b0 < G; b0 += 16) {
          const ulonglong2* w[8];
          double v[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = c < NV && b0 + 2 * i < G ? part + (size_t)(b0 + 2 * i) * MAXSUM + c : nullptr;
          bad |= !get_words<8>(w, tag, v);
          p += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
        p += __shfl_xor_sync(0xffffffffu, p, 1);
        if (s2 == 0) sR[c] = p;
      }
    } else if (warp == 8) {
      if (!direct)  // this block's sums, added up for everybody
        for (int c = b; c < NV; c += G) {
          const ulonglong2* w[5];
          double v[5];
#pragma unroll
          for (int i = 0; i < 5; ++i) w[i] = lane + 32 * i < G ? part + (size_t)(lane + 32 * i) * MAXSUM + c : nullptr;
          bad |= !get_words<5>(w, tag, v);
          const double s = warp_sum(((v[0] + v[1]) + (v[2] + v[3])) + v[4]);
          if (lane == 0) put_word(R + c * LINE, s, tag);
        }
    } else {
      // sigma from this block's own copy of u, and what follows from it
      double q0 = 0.0, q1 = 0.0, q2 = 0.0, q3 = 0.0;
      for (int r = j + 2 + lane; r < n; r += 128) {  // (su is zero past n; 64 entries of it exist)
        const double x0 = su[r], x1 = r + 32 < n ? su[r + 32] : 0.0, x2 = r + 64 < n ? su[r + 64] : 0.0,
                     x3 = r + 96 < n ? su[r + 96] : 0.0;
        q0 = fma(x0, x0, q0);
        q1 = fma(x1, x1, q1);
        q2 = fma(x2, x2, q2);
        q3 = fma(x3, x3, q3);
      }
      const double sigma = warp_sum((q0 + q1) + (q2 + q3)), a0 = sa0;
      double tau = 0.0, inv = 0.0, beta = a0;  // sigma = 0: nothing below the subdiagonal, H = I
      if (sigma != 0.0) {
        const double q = fma(a0, a0, sigma), rn = rsqrt(q), nrm = q * rn;
        if (nrm > 0.0 && rn < 1e308) {  // |beta| = nrm, tau = 1 + |a0| / nrm: one division on the way
          beta = a0 >= 0.0 ? -nrm : nrm;
          tau = fma(fabs(a0), rn, 1.0);
        } else {  // out of range of the reciprocal root, or not finite
          const double root = sqrt(q);
          beta = a0 >= 0.0 ? -root : root;
          tau = (beta - a0) / beta;
        }
        inv = 1.0 / (a0 - beta);
      }
      if (lane == 0) {
        sti[0] = tau;
        sti[1] = inv;
        if (b == 0) {
          a.e[j] = scaled ? scalbn(beta, ex) : beta;
          a.tau[j] = tau;
        }
      }
      // row jj of V on the panel's rows (k0 + 1 + lane)
      const int r = k0 + 1 + lane;
      sVp[jj][lane] = r == j + 1 ? 1.0 : r > j + 1 ? inv * vpan : 0.0;
    }
    if (warp == 9 && !direct) {
      const ulonglong2* w[2] = {lane < NV ? R + lane * LINE : nullptr,
                                lane + 32 < NV ? R + (lane + 32) * LINE : nullptr};
      double v[2];
      bad |= !get_words<2>(w, tag, v);
      sR[lane] = v[0];
      sR[lane + 32] = v[1];
    }
    if (__syncthreads_or(bad)) {
      if (bad) atomicOr(a.err, 1);
      return;
    }
    // ---- D_r = sum_q W_q[r] (V^T u)_q + V_q[r] (W^T u)_q on the row threads,
    // s2 on warp 8, the scalars on warp 9
    const double tau = sti[0], inv = sti[1];
    double v = 0.0, B = 0.0, E = 0.0;  // w = B + alpha2 v, the next column's entry E - v w[j+1] - w
    if (tid < ROW_THREADS) {
      if (row_warp) {
        double d1 = 0.0, d2 = 0.0;
#pragma unroll 4
        for (int q = sub; q < jj; q += tpr) {
          d1 = fma(sW[rloc][q], sR[q], d1);
          d2 = fma(sV[rloc][q], sR[jj + q], d2);
        }
        d1 += d2;
        for (int o = tpr >> 1; o > 0; o >>= 1) d1 += __shfl_xor_sync(0xffffffffu, d1, o);
        if (has_row && sub == 0) {
          E = ac - Cr;
          if (row == j + 1) {
            v = 1.0;
          } else if (row > j + 1) {
            v = inv * ur;
            B = tau * fma(inv, st[rloc] - d1, E);
          }
        }
      }
    } else if (warp == 8) {
      const ulonglong2* w[5];
      double x[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) w[i] = lane + 32 * i < G ? T2 + (lane + 32 * i) * LINE : nullptr;
      bad |= !get_words<5>(w, tag, x);
      const double s = direct ? warp_sum(x[0]) : warp_sum(((x[0] + x[1]) + (x[2] + x[3])) + x[4]);
      if (lane == 0) ss2 = s;
    } else {
      const double s1 = sR[2 * jj], vn = sVn[lane], wn = sWn[lane];
      const double y = lane < jj ? fma(inv, sR[lane], vn) : 0.0;
      const double z = lane < jj ? fma(inv, sR[jj + lane], wn) : 0.0;
      // sum of y z (lower half-warp) and of w_n y + v_n z (upper) together
      const double p = y * z, q = fma(wn, y, vn * z);
      const bool up = lane & 16;
      double h = (up ? q : p) + __shfl_xor_sync(0xffffffffu, up ? p : q, 16);
      for (int o = 8; o > 0; o >>= 1) h += __shfl_xor_sync(0xffffffffu, h, o);
      const double yz = __shfl_sync(0xffffffffu, h, 0), sj = __shfl_sync(0xffffffffu, h, 16);
      const double at = fma(inv, s1, sAd), f = -0.5 * tau * tau;
      if (lane == 0) {
        sc[0] = f * fma(-2.0, yz, fma(inv, s1, at));
        sc[1] = f * (inv * inv);
        sc[2] = tau * (at - sj);
      }
    }
    if (__syncthreads_or(bad)) {
      if (bad) atomicOr(a.err, 1);
      return;
    }
    // ---- v, w and the next column on this block's rows
    if (has_row && sub == 0) {
      const double alpha2 = fma(sc[1], ss2, sc[0]), w1 = sc[2] + alpha2;
      double w = 0.0;
      if (row == j + 1) w = w1;
      else if (row > j + 1) w = fma(alpha2, v, B);
      xv = fma(-v, w1, E - w);
      sV[rloc][jj] = v;
      sW[rloc][jj] = w;
      // (published before the slower stores below)
      if (row >= j + 1 && jj + 1 < a.nbp) put_word(a.X + ((size_t)((j + 1) & 1) * G + b) * a.lw + rloc, xv, tag + 1);
      if (row > j + 1) a.A[(size_t)j * n + row] = v;
      a.Vp[(size_t)jj * n + row] = v;
      a.Wp[(size_t)jj * n + row] = w;
    }
    ac = acn;
    __syncwarp();  // (the row's other threads read this column's w when they publish its row)
  }
}

// Largest biased exponent field of x[0..n) into *emax (cleared before).
__global__ void k_max_exponent(const double* __restrict__ x, int64_t n, int* __restrict__ emax) {
  int m = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (__double2hiint(x[i]) >> 20) & 0x7FF);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(emax, m);
}

// [V | W] and [W | V] as m x 2 NB row-major operands for the trailing update
// (rows k.. of the panel's column-major V, W).
__global__ void k_pack_vw(const double* __restrict__ Vp, const double* __restrict__ Wp,
                          int64_t n, int64_t k, int64_t m, int nbp, double* __restrict__ X,
                          double* __restrict__ Y) {
  const int64_t w = 2 * NB;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m * w;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / w, q = e - r * w;
    const int64_t qq = q % NB;
    double vx = 0.0, vy = 0.0;
    if (qq < nbp) {
      const double v = Vp[qq * n + k + r], ww = Wp[qq * n + k + r];
      vx = q < NB ? v : ww;
      vy = q < NB ? ww : v;
    }
    X[e] = vx;
    Y[e] = vy;
  }
}

int grid_1d(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>(cdiv(n, 256), 16384)); }

}  // namespace

bool sytrd_supported(int64_t n) { return n >= 2 && n <= 8192; }

// A (n x n, symmetric, full) -> reflectors in A (lower, dsytrd layout), d, e, tau.
osmps_status sytrd_tc(osmps_ctx* ctx, double* A, int64_t n, double* d, double* e, double* tau,
                      cudaStream_t s) {
  osmps_status st = OSMPS_OK;
  if (!sytrd_supported(n)) return set_error(OSMPS_EUNSUPPORTED, "sytrd: n=%lld", (long long)n);
  const size_t smem = (size_t)((n + 64 + 1) & ~(int64_t)1) * 8;
  const bool vec = n % 2 == 0 && (reinterpret_cast<uintptr_t>(A) & 15) == 0;  // 16-byte rows
  const auto in_l2 = vec ? k_sytrd_panel<true, false> : k_sytrd_panel<false, false>;
  const auto in_smem = k_sytrd_panel<false, true>;
  // dynamic shared memory beside the kernels' 48 KB
  constexpr size_t SMEM_MOST = (size_t)(227 - 48) * 1024;
  OSMPS_CUDA(cudaFuncSetAttribute(in_l2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MOST));
  OSMPS_CUDA(cudaFuncSetAttribute(in_smem, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MOST));
  int per_sm = 0;
  OSMPS_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, in_smem, ST_THREADS, SMEM_MOST));
  if (per_sm < 1) return set_error(OSMPS_EUNSUPPORTED, "sytrd: panel kernel does not fit an SM");
  // Blocks of a panel with m trailing rows: about 8 rows each, at most one
  // block per SM (all co-resident). Up to SMALL_M rows, no more than DIRECT_G:
  // the product A22 v (m^2 / 64 clocks on 32 SMs, 2.3 us at 544) costs less
  // there than the second exchange of the sums (line at 768: n = 1024 9.3
  // instead of 8.0 us a column, n = 768 9.8 instead of 8.0).
  constexpr int64_t SMALL_M = 544;
  const auto blocks_for = [&](int64_t m) {
    const int64_t most = m <= SMALL_M ? (m <= 256 ? DIRECT_G / 2 : DIRECT_G) : 160;
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(ctx->sm_count, most), cdiv(m, 8)));
  };
  const int Gmax = (int)std::max<int64_t>(std::min<int64_t>(ctx->sm_count, 160), DIRECT_G);
  if (cdiv(n, blocks_for(n)) > MAXLOC)
    return set_error(OSMPS_EUNSUPPORTED, "sytrd: n=%lld needs more than %d rows per block",
                     (long long)n, MAXLOC);
  // panel vectors, GEMM operands, then the tagged words (cleared: tags start at 1)
  const size_t xwords = (size_t)n + (size_t)LINE * Gmax;  // rows of every block rounded up to lines
  const size_t words = 2 * xwords + 2 * NB + 2 * (size_t)MAXSUM * Gmax + 2 * MAXSUM * LINE + 2 * (size_t)Gmax * LINE;
  const size_t vecs = (size_t)(2 * NB * n + 2 * n * 2 * NB);
  double* buf = (double*)ws_get(ctx, SLOT_TRD, (vecs + 2 * words + 64) * 8, s, &st);
  if (!buf) return st;
  double* Vp = buf;
  double* Wp = Vp + NB * n;
  double* X = Wp + NB * n;
  double* Y = X + 2 * NB * n;
  ulonglong2* word = reinterpret_cast<ulonglong2*>(buf + vecs);
  int* emax = reinterpret_cast<int*>(word + words);
  OSMPS_CUDA(cudaMemsetAsync(word, 0, (words + 1) * sizeof(ulonglong2), s));
  { k_max_exponent<<<(int)std::min<int64_t>(cdiv(n * n, 1024), 1216), 256, 0, s>>>(A, n * n, emax); note_launch(); }
  OSMPS_LAUNCH_CHECK();
  int* err = ctx->dev_flags + 3;
  for (int64_t k0 = 0; k0 < n; k0 += NB) {
    const int nbp = (int)std::min<int64_t>(NB, n - k0);
    const int G = blocks_for(n - k0);
    SytrdArgs a;
    a.A = A; a.n = (int)n; a.k0 = (int)k0; a.nbp = nbp;
    a.d = d; a.e = e; a.tau = tau; a.Vp = Vp; a.Wp = Wp;
    a.X = word; a.Wn = a.X + 2 * xwords; a.part = a.Wn + 2 * NB; a.R = a.part + 2 * (size_t)MAXSUM * Gmax;
    a.T2 = a.R + 2 * MAXSUM * LINE; a.err = err; a.emax = emax;
    const int64_t rows = cdiv(n - k0, G);
    a.lw = (int)round_up(rows, LINE);
    const int64_t stride = round_up(n - k0, 2);
    const size_t with_rows = smem + (size_t)(rows * stride) * 8;
    a.sa = with_rows <= SMEM_MOST ? (int)stride : 0;
    void* args[] = {&a};
    // algorithmic float64 work of the panel: per column j (i columns of the
    // panel before it, m = n - j - 1 trailing rows) the product A22 v
    // (2 m^2) and the corrections V (W^T v) + W (V^T v) (8 m i)
    double pf = 0.0;
    for (int i = 0; i < nbp; ++i) {
      const double mm = (double)(n - (k0 + i) - 1);
      pf += 2.0 * mm * mm + 8.0 * mm * i;
    }
    const int ph = prof_begin(s);
    OSMPS_CUDA(cudaLaunchCooperativeKernel((void*)(a.sa ? in_smem : in_l2), dim3(G), dim3(ST_THREADS), args,
                                           a.sa ? with_rows : smem, s));
    note_launch();
    prof_end(ph, s, OSMPS_KERNEL_SYTRD_PANEL, pf, 0.0);
    const int64_t k = k0 + nbp, m = n - k;
    if (m <= 0) break;
    { k_pack_vw<<<grid_1d(m * 2 * NB), 256, 0, s>>>(Vp, Wp, n, k, m, nbp, X, Y); note_launch(); }
    OSMPS_LAUNCH_CHECK();
    // A22 -= [V W] [W V]^T = V W^T + W V^T on the trailing block
    SplitView xv; xv.src = X; xv.rows = m; xv.K = 2 * NB; xv.s0 = 2 * NB; xv.sk = 1;
    SplitView yv; yv.src = Y; yv.rows = m; yv.K = 2 * NB; yv.s0 = 2 * NB; yv.sk = 1;
    OSMPS_TRY(gemm_emu(ctx, xv, yv, m, m, 2 * NB, A + k * n + k, n, s, true));
  }
  return OSMPS_OK;
}

}  // namespace osmps

using namespace osmps;

extern "C" osmps_status osmps_sytrd(osmps_ctx* ctx, double* A, int64_t n, double* d, double* e,
                                    double* tau, void* stream) {
  clear_error();
  if (!ctx || !A || !d || !e || !tau) return set_error(OSMPS_EINVAL, "osmps_sytrd: null argument");
  if (!sytrd_supported(n)) return set_error(OSMPS_ESHAPE, "osmps_sytrd: n=%lld outside [2, 8192]", (long long)n);
  OSMPS_CUDA(cudaSetDevice(ctx->device));
  CtxScope scope_(ctx);
  cudaStream_t s = (cudaStream_t)stream;
  OSMPS_TRY(sytrd_tc(ctx, A, n, d, e, tau, s));
  int flag = 0;
  OSMPS_CUDA(cudaMemcpyAsync(&flag, ctx->dev_flags + 3, sizeof(int), cudaMemcpyDeviceToHost, s));
  OSMPS_CUDA(cudaStreamSynchronize(s));
  if (flag) {
    cudaMemsetAsync(ctx->dev_flags + 3, 0, sizeof(int), s);
    return set_error(OSMPS_ETIMEOUT, "osmps_sytrd: a wait of the panel reduction gave up");
  }
  return OSMPS_OK;
}
