// Float64 strided batched GEMM on the FP64 tensor path (mma.sync m8n8k4 f64).
//
// Used for the plain float64 contractions (Sec. 3.4 matvec and environment
// updates at OSMPS_PREC_FP64), the Gram matrices and projections of the
// eigendecomposition split (Sec. 2, Eq. AAD_ULLUD), theta formation and the
// QR shifts. Arbitrary element strides let one kernel express every
// transpose and index grouping the contractions need without copies.
//
// An SM does about two float64 FMAs per clock, half of one from each of its
// four sub-partitions, so a product is bound by how evenly its FMAs spread
// over the sub-partitions of all SMs, never by its loads (8 to 16 bytes of
// operand per 128 clocks of DMMA at the tiles below). Hence small tiles for
// every size: a CTA is four warps, one per sub-partition, on one 16x16 or 8x8
// tile of C. With tiles enough for four CTAs per SM each warp has an 8x8 part
// of the tile and all of K, in order; with fewer, the warps share the K range
// (K group of four number g goes to warp g mod 4) and their partial tiles are
// added in warp order. Fragments are read straight from global memory (eight
// rows x 32 bytes or four rows x 64 bytes per load), a round of groups ahead
// of the DMMAs.
// Measured against 64x64 tiles staged through shared memory (M x N x K, us):
// 128x32x96 119 -> 6.3, 64x64x64 82 -> 4.2, 300x340x300 367 -> 74,
// 512x512x512 615 -> 274, 1024x1024x1024 2445 -> 2074 (1.04 TFLOP/s),
// 2048x2048x1024 8546 -> 8253.
#include <algorithm>

#include "common.cuh"

namespace osmps {

namespace {

struct Args {
  int64_t M, N, K;
  const double* A;
  int64_t sam, sak, sab;
  const double* B;
  int64_t sbk, sbn, sbb;
  double* C;
  int64_t scm, scn, scb;
  double alpha, beta;
};

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

// FM x FN: 8x8 fragments per warp. SPLIT: all four warps on the CTA's one
// 8 FM x 8 FN tile, sharing K; else 2 x 2 warps on a tile of twice that edge.
template <int FM, int FN, bool SPLIT>
__global__ void __launch_bounds__(128) k_gemm_f64(Args p, int tiles_n) {
  constexpr int KU = FM * FN > 1 ? 2 : 4;  // K groups in flight per warp
  constexpr int TM = 8 * FM, TN = 8 * FN, W = SPLIT ? 1 : 2;
  constexpr int KSTEP = SPLIT ? 16 : 4;    // between a warp's K groups
  __shared__ double red[SPLIT ? 4 : 1][SPLIT ? TM : 1][SPLIT ? TN : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, tq = lane & 3;
  const int64_t m0 = (int64_t)(blockIdx.x / tiles_n) * (W * TM) + (SPLIT ? 0 : (warp >> 1) * TM);
  const int64_t n0 = (int64_t)(blockIdx.x % tiles_n) * (W * TN) + (SPLIT ? 0 : (warp & 1) * TN);
  const double* A = p.A + (int64_t)blockIdx.y * p.sab;
  const double* B = p.B + (int64_t)blockIdx.y * p.sbb;
  // this lane's rows / columns, those past the edge read as zero
  const double* ap[FM];
  const double* bp[FN];
  bool am[FM], bm[FN];
#pragma unroll
  for (int i = 0; i < FM; ++i) {
    const int64_t m = m0 + 8 * i + g;
    am[i] = m < p.M;
    ap[i] = A + (am[i] ? m : 0) * p.sam;
  }
#pragma unroll
  for (int j = 0; j < FN; ++j) {
    const int64_t n = n0 + 8 * j + g;
    bm[j] = n < p.N;
    bp[j] = B + (bm[j] ? n : 0) * p.sbn;
  }
  double a[KU][FM], b[KU][FN];
  auto load = [&](int64_t k) {  // the warp's KU groups from K index k on, KSTEP apart
#pragma unroll
    for (int u = 0; u < KU; ++u) {
      const int64_t kk = k + KSTEP * u + tq;
      const bool in = kk < p.K;
#pragma unroll
      for (int i = 0; i < FM; ++i) a[u][i] = in && am[i] ? ap[i][kk * p.sak] : 0.0;
#pragma unroll
      for (int j = 0; j < FN; ++j) b[u][j] = in && bm[j] ? bp[j][kk * p.sbk] : 0.0;
    }
  };
  double acc[FM][FN][2];
#pragma unroll
  for (int i = 0; i < FM; ++i)
#pragma unroll
    for (int j = 0; j < FN; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
  int64_t k = SPLIT ? 4 * warp : 0;
  load(k);
  for (; k < p.K; k += KSTEP * KU) {
    double ca[KU][FM], cb[KU][FN];
#pragma unroll
    for (int u = 0; u < KU; ++u) {
#pragma unroll
      for (int i = 0; i < FM; ++i) ca[u][i] = a[u][i];
#pragma unroll
      for (int j = 0; j < FN; ++j) cb[u][j] = b[u][j];
    }
    load(k + KSTEP * KU);  // past the end: all zero, nothing is read
#pragma unroll
    for (int u = 0; u < KU; ++u)
      if (k + KSTEP * u < p.K) {  // the same for the whole warp
#pragma unroll
        for (int i = 0; i < FM; ++i)
#pragma unroll
          for (int j = 0; j < FN; ++j) dmma(acc[i][j][0], acc[i][j][1], ca[u][i], cb[u][j]);
      }
  }
  double* C = p.C + (int64_t)blockIdx.y * p.scb;
  const auto put = [&](int64_t gm, int64_t gn, double sum) {
    if (gm < p.M && gn < p.N) {
      double* dst = C + gm * p.scm + gn * p.scn;
      double v = p.alpha * sum;
      if (p.beta != 0.0) v = fma(p.beta, *dst, v);
      *dst = v;
    }
  };
  if constexpr (SPLIT) {
#pragma unroll
    for (int i = 0; i < FM; ++i)
#pragma unroll
      for (int j = 0; j < FN; ++j)
#pragma unroll
        for (int r = 0; r < 2; ++r) red[warp][8 * i + g][8 * j + 2 * tq + r] = acc[i][j][r];
    __syncthreads();
    for (int e = threadIdx.x; e < TM * TN; e += 128) {
      const int r = e / TN, c = e % TN;
      put(m0 + r, n0 + c, ((red[0][r][c] + red[1][r][c]) + red[2][r][c]) + red[3][r][c]);
    }
  } else {
#pragma unroll
    for (int i = 0; i < FM; ++i)
#pragma unroll
      for (int j = 0; j < FN; ++j)
#pragma unroll
        for (int r = 0; r < 2; ++r) put(m0 + 8 * i + g, n0 + 8 * j + 2 * tq + r, acc[i][j][r]);
  }
}

// Tile edge, 16 or 8: the one whose busiest SM has the least to do, i.e. the
// smaller ceil(tiles / SMs) edge^2. The 8x8 tile is counted 15% dearer per
// FMA: with several rounds of tiles it measured 2% (300x300x340) to 40%
// (256x256x256) slower at equal load, so it wins where it halves the rounds
// (128x128x128: 8.3 against 14.4 us) and not for a few per cent of balance.
constexpr int F64_SMS = 152;  // of the one GPU this code is for
constexpr double COST_8 = 1.15;
double busiest_sm(int64_t M, int64_t N, int64_t batch, int64_t t) {
  return (double)cdiv(cdiv(M, t) * cdiv(N, t) * batch, F64_SMS) * (double)(t * t);
}
int f64_tile(int64_t M, int64_t N, int64_t batch) {
  return COST_8 * busiest_sm(M, N, batch, 8) < busiest_sm(M, N, batch, 16) ? 8 : 16;
}

}  // namespace

double gemm_f64_us(int64_t M, int64_t N, int64_t K) {
  const double fma = std::min(busiest_sm(M, N, 1, 16), COST_8 * busiest_sm(M, N, 1, 8)) * (double)K;
  return 4.0 + fma / 3500.0;  // 3.5 GFMA/s per SM measured
}

osmps_status gemm_f64(const GemmF64& g, cudaStream_t stream) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return OSMPS_OK;
  if (g.K <= 0) {
    return set_error(OSMPS_ESHAPE, "gemm_f64: K=%lld", (long long)g.K);
  }
  // (M: a row limit that callers have always met; the grid's own is the tiles')
  if (g.M > (int64_t)64 * 65535 || g.batch > 65535)
    return set_error(OSMPS_ESHAPE, "gemm_f64: M=%lld batch=%lld exceed the supported range",
                     (long long)g.M, (long long)g.batch);
  const int t = f64_tile(g.M, g.N, g.batch);
  const int64_t tiles_n = cdiv(g.N, t), tiles = tiles_n * cdiv(g.M, t);
  if (tiles > 2147483647ll)
    return set_error(OSMPS_ESHAPE, "gemm_f64: %lld output tiles exceed the grid limit", (long long)tiles);
  Args a{g.M, g.N, g.K, g.A, g.sam, g.sak, g.sab, g.B, g.sbk, g.sbn, g.sbb,
         g.C, g.scm, g.scn, g.scb, g.alpha, g.beta};
  const dim3 grid((unsigned)tiles, (unsigned)g.batch);
  const int ph = prof_begin(stream);
  if (t == 16 && tiles * g.batch >= 4 * F64_SMS) k_gemm_f64<1, 1, false><<<grid, 128, 0, stream>>>(a, (int)tiles_n);
  else if (t == 16) k_gemm_f64<2, 2, true><<<grid, 128, 0, stream>>>(a, (int)tiles_n);
  else k_gemm_f64<1, 1, true><<<grid, 128, 0, stream>>>(a, (int)tiles_n);
  note_launch();
  OSMPS_LAUNCH_CHECK();
  const double f = 2.0 * (double)g.M * (double)g.N * (double)g.K * (double)g.batch;
  prof_end(ph, stream, OSMPS_KERNEL_GEMM_F64, f, f);
  return OSMPS_OK;
}

}  // namespace osmps
