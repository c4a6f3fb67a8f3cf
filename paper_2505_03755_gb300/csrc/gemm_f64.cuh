// FP64 GEMM on the double-precision tensor path (mma.sync.m16n8k4.f64, "DMMA").
//
//   C[z](m, n) (=|+=) alpha * sum_{k in split} A[b](m, k) * B[b](k, n),   b = z / ksplit
//
// The FP64 pipe of this part delivers about 3.5 flop per clock and SM, so one 16x8x4 DMMA occupies
// an SM for some 290 clocks: the time of a launch is the largest number of DMMAs on any SM, and
// staging operands element by element through loader objects (see las_common.cuh) is never the
// bound.  Hence the shape of the kernel: CTA tile 64 x 8 NJ with NJ = 4, 6, 8 or 10 picked per
// product (f64_nj), four warps of 16 rows, and every 16 x 8 block beyond M or N, or above the
// diagonal of a symmetric result, is left out; K steps of 16 are double-buffered so that one CTA per
// SM keeps the pipe busy.  Against a fixed 64 x 64 tile (half transform of 237 x 237 blocks and 48
// columns, 948 auxiliary rows: 6.86 ms, now 4.97) a quarter of the DMMAs were padding columns.
#pragma once
#include "las_common.cuh"

namespace lasdf {

__device__ __forceinline__ void dmma_16x8x4(double (&c)[4], double a0, double a1, double b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k4.row.col.f64.f64.f64.f64 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};\n"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a0), "d"(a1), "d"(b0));
}

// SYM: the result is symmetric (M = N): blocks that touch the lower triangle are computed and
// their elements with row >= column are stored at both places.
template <int NJ, bool SYM, class LA, class LB, class SC>
__global__ void __launch_bounds__(128)
k_gemm_f64(int M, int N, int K, int ksplit, int kchunk, LA la, LB lb, SC sc) {
  pdl_begin();
  constexpr int BN = 8 * NJ, PA = 8, PB = BN / 8;   // A and B elements per thread and K step
  __shared__ double As[2][16][64 + 2];
  __shared__ double Bs[2][16][BN + 2];
  const int z = blockIdx.z;
  const int b = z / ksplit;
  const int ks = z - b * ksplit;
  const int m0 = blockIdx.x * 64, n0 = blockIdx.y * BN;
  if (SYM && n0 > m0 + 63) return;
  const int kbeg = ks * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wrow = m0 + warp * 16;
  // live column blocks of this warp
  int nlive = wrow < M ? min(NJ, (N - n0 + 7) / 8) : 0;
  if (SYM) nlive = min(nlive, (wrow + 15 - n0) / 8 + 1);
  const int g = lane >> 2, t = lane & 3;
  double acc[NJ][4];
#pragma unroll
  for (int j = 0; j < NJ; ++j)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[j][r] = 0.0;

  double pa[PA], pb[PB];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int i = 0; i < PA; ++i) {
      const int mm = tid & 63, kk = (tid >> 6) + 2 * i;
      const int m = m0 + mm, k = k0 + kk;
      pa[i] = (m < M && k < kend) ? la(b, m, k) : 0.0;
    }
#pragma unroll
    for (int i = 0; i < PB; ++i) {
      const int e = tid + 128 * i, kk = e / BN, n = n0 + e - kk * BN, k = k0 + kk;
      pb[i] = (n < N && k < kend) ? lb(b, k, n) : 0.0;
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int i = 0; i < PA; ++i) As[buf][(tid >> 6) + 2 * i][tid & 63] = pa[i];
#pragma unroll
    for (int i = 0; i < PB; ++i) {
      const int e = tid + 128 * i, kk = e / BN;
      Bs[buf][kk][e - kk * BN] = pb[i];
    }
  };
  if (kbeg < kend) {
    fetch(kbeg);
    put(0);
  }
  __syncthreads();
  int buf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += 16, buf ^= 1) {
    const bool more = k0 + 16 < kend;
    if (more) fetch(k0 + 16);
#pragma unroll
    for (int kk = 0; kk < 16; kk += 4) {
      const double a0 = As[buf][kk + t][warp * 16 + g], a1 = As[buf][kk + t][warp * 16 + g + 8];
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (j < nlive) dmma_16x8x4(acc[j], a0, a1, Bs[buf][kk + t][j * 8 + g]);
    }
    if (more) put(buf ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    if (j >= nlive) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int row = wrow + g + ((r >> 1) << 3);
      const int col = n0 + j * 8 + 2 * t + (r & 1);
      if (row < M && col < N && (!SYM || col <= row)) {
        sc(z, row, col, acc[j][r]);
        if (SYM && col < row) sc(z, col, row, acc[j][r]);
      }
    }
  }
}

}  // namespace lasdf

// 8-column blocks per CTA tile for N columns: as few tiles as possible, of equal width.
static inline int f64_nj(int N) {
  const int n8 = (N + 7) / 8, tiles = (n8 + 9) / 10, per = (n8 + tiles - 1) / tiles;
  return per <= 4 ? 4 : per <= 6 ? 6 : per <= 8 ? 8 : 10;
}
static inline int f64_tiles(int M, int N) {
  const int bn = 8 * f64_nj(N);
  return ((M + 63) / 64) * ((N + bn - 1) / bn);
}
static inline int f64_kchunk(int K, int ksplit) {
  const int k = ((K + ksplit - 1) / ksplit + 15) / 16 * 16;
  return k < 16 ? 16 : k;
}
// K split in [1, cap] that ends first on `sms` SMs: CTAs on the fullest SM times the K steps of
// each, with one more step per CTA for its start and the sum of its partial.
static inline int f64_balanced_ksplit(int tiles, int K, int cap, int sms) {
  int best = 1;
  long best_t = -1;
  for (int ks = 1; ks <= cap; ++ks) {
    const long t = (((long)tiles * ks + sms - 1) / sms) * (f64_kchunk(K, ks) / 16 + 1);
    if (best_t < 0 || t < best_t) {
      best_t = t;
      best = ks;
    }
  }
  return best;
}

template <bool SYM = false, class LA, class LB, class SC>
void gemm_f64(int M, int N, int K, int batch, int ksplit, LA a, LB b, SC c, cudaStream_t s) {
  if (M <= 0 || N <= 0 || batch <= 0) return;
  if (ksplit < 1) ksplit = 1;
  const int kchunk = f64_kchunk(K, ksplit);
  const int nj = f64_nj(N);
  dim3 grid((M + 63) / 64, (N + 8 * nj - 1) / (8 * nj), batch * ksplit);
  // an ordinary launch: blocks placed while the launch before drains would gather on the SMs that
  // are free first, and the fullest SM is the time (a chained C^T G at 400 orbitals lost 45 us)
  auto go = [&](auto kern) { kern<<<grid, 128, 0, s>>>(M, N, K, ksplit, kchunk, a, b, c); };
  switch (nj) {
    case 4: go(lasdf::k_gemm_f64<4, SYM, LA, LB, SC>); break;
    case 6: go(lasdf::k_gemm_f64<6, SYM, LA, LB, SC>); break;
    case 8: go(lasdf::k_gemm_f64<8, SYM, LA, LB, SC>); break;
    default: go(lasdf::k_gemm_f64<10, SYM, LA, LB, SC>); break;
  }
  las_count_launch();
}
