// gemm_simt.cu - CUDA-core GEMM for the FP64 reference mode and the FP32 mode.
//
// C[m][n] = alpha * sum_k A[m*lda + k] B[n*ldb + k] + beta * C[m*ldc + n]: both operands
// K-major (the layout the block-spin contraction builds, the same one the tensor-core
// path consumes). 128x64 output tile per CTA (64x32 where that leaves SMs idle), 256 threads
// with an 8x4 (4x2) register tile, 16-wide k slices staged in shared memory. FP64 mode uses DFMA; FP32 mode FFMA with FP32
// accumulation. Ragged M, N and K edges are guarded.
#include <type_traits>

#include "common.cuh"

namespace hotrg {

constexpr int kBK = 16;

// Tile kBM x kBN, 256 threads of kTM x kTN outputs each.
template <typename R, int kTM, int kTN>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const R* __restrict__ A, int64_t lda, const R* __restrict__ B,
                                                        int64_t ldb, R* __restrict__ C, int64_t ldc, int64_t M,
                                                        int64_t N, int64_t K, R alpha, R beta,
                                                        const __grid_constant__ OneProduct one) {
  constexpr int kBM = 16 * kTM, kBN = 16 * kTN;
  __shared__ R As[kBK][kBM + 4];
  __shared__ R Bs[kBK][kBN + 4];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;   // 16 x 16 threads; rows ty*kTM.., cols tx*kTN..
  int64_t m0 = (int64_t)blockIdx.y * kBM, n0 = (int64_t)blockIdx.x * kBN;
  if (one.sec.tab.base) {
    // a product by sectors: tile rows of charge 0, then of charge 1 (each against the columns and over
    // the summed indices of its own charge class, packed to the front of a row)
    const SectorPlan& p = *one.sec.tab.at(one.elem).plan;
    const GemmSectors& s = one.sec;
    const int r0 = p.row[0][s.xa + s.na] - p.row[0][s.xa], r1 = p.row[1][s.xa + s.na] - p.row[1][s.xa];
    const int c0 = p.row[0][s.xb + s.nb] - p.row[0][s.xb], c1 = p.row[1][s.xb + s.nb] - p.row[1][s.xb];
    const int64_t lim = s.row_limit > 0 ? s.row_limit : 0x7fffffff;
    const int64_t t0 = (min((int64_t)r0, lim) + kBM - 1) / kBM;
    const int q = (int64_t)blockIdx.y >= t0, qc = q ^ (one.parity & p.odd);
    if (q) m0 -= t0 * kBM;
    M = min((int64_t)(q ? r1 : r0), lim);
    N = qc ? c1 : c0;
    K = p.K[q ^ (one.pa & p.odd)];
    if (m0 >= M || n0 >= N) return;
    A += (q ? (int64_t)r0 : 0) * lda;
    C += (q ? (int64_t)r0 : 0) * ldc;
    B += (qc ? (int64_t)c0 : 0) * ldb;
  }
  R acc[kTM][kTN];
#pragma unroll
  for (int i = 0; i < kTM; ++i)
#pragma unroll
    for (int j = 0; j < kTN; ++j) acc[i][j] = 0;

  for (int64_t k0 = 0; k0 < K; k0 += kBK) {
    // A tile: kBM x 16 elements, kTM per thread; k fastest for coalescing
#pragma unroll
    for (int r = 0; r < kTM; ++r) {
      const int e = tid + r * 256;
      const int row = e / kBK, kk = e % kBK;
      const int64_t gm = m0 + row, gk = k0 + kk;
      As[kk][row] = (gm < M && gk < K) ? A[gm * lda + gk] : (R)0;
    }
#pragma unroll
    for (int r = 0; r < kTN; ++r) {
      const int e = tid + r * 256;
      const int col = e / kBK, kk = e % kBK;
      const int64_t gn = n0 + col, gk = k0 + kk;
      Bs[kk][col] = (gn < N && gk < K) ? B[gn * ldb + gk] : (R)0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kBK; ++kk) {
      R a[kTM], b[kTN];
#pragma unroll
      for (int i = 0; i < kTM; ++i) a[i] = As[kk][ty * kTM + i];
#pragma unroll
      for (int j = 0; j < kTN; ++j) b[j] = Bs[kk][tx * kTN + j];
#pragma unroll
      for (int i = 0; i < kTM; ++i)
#pragma unroll
        for (int j = 0; j < kTN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kTM; ++i) {
    const int64_t gm = m0 + ty * kTM + i;
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < kTN; ++j) {
      const int64_t gn = n0 + tx * kTN + j;
      if (gn >= N) continue;
      R* c = C + gm * ldc + gn;
      *c = beta == (R)0 ? alpha * acc[i][j] : alpha * acc[i][j] + beta * *c;
    }
  }
}

template <typename R>
cudaError_t launch_gemm_simt(const R* A, int64_t lda, const R* B, int64_t ldb, R* C, int64_t ldc, int64_t M,
                             int64_t N, int64_t K, double alpha, double beta, cudaStream_t st, const OneProduct& one) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  // Tiles of 128 x 64 do 32 products per 12 operand reads, 64 x 32 ones 8 per 6, but four times as many of them share
  // the SMs more evenly. FP64: the FP64 pipe bounds either, so small tiles win below two large ones per SM (M = N, K =
  // 1024: 1.35 at M = 896, 1.6 at 1100, 1.0 at 1024 and 1536; D = 4 by sectors: 1088 -> 779 us). FP32: operand reads bound
  // the small ones, which win while at most three of them per SM hold the whole product (operands from HBM, M = N, K =
  // 1024: 1.7 at M = 512, 1.38 at 768, 1.10 at 960 - from L2 0.97 there - then 0.84 at 1024, 0.66 at 1536).
  auto go = [&](auto tm, auto tn) -> cudaError_t {
    constexpr int TM = decltype(tm)::value, TN = decltype(tn)::value;
    const int64_t more = one.sec.tab.base ? 1 : 0;   // two sectors: at most one more tile row
    const int64_t gy = (M + 16 * TM - 1) / (16 * TM) + more, gx = (N + 16 * TN - 1) / (16 * TN);
    if (gy > 65535 || gx > 0x7fffffffLL) return cudaErrorInvalidValue;
    gemm_simt_kernel<R, TM, TN><<<dim3((unsigned)gx, (unsigned)gy), 256, 0, st>>>(A, lda, B, ldb, C, ldc, M, N, K, (R)alpha,
                                                                                  (R)beta, one);
    return cudaGetLastError();
  };
  using I2 = std::integral_constant<int, 2>;
  using I4 = std::integral_constant<int, 4>;
  using I8 = std::integral_constant<int, 8>;
  const int64_t blocks = one.sec.tab.base ? 2 : 1;   // by sectors: half of the tiles of the dense product
  const int64_t large = ((M + 127) / 128) * ((N + 63) / 64) / blocks, small = ((M + 63) / 64) * ((N + 31) / 32) / blocks;
  return (sizeof(R) == 8 ? large < 2 * 152 : small <= 3 * 152) ? go(I4{}, I2{}) : go(I8{}, I4{});
}
template cudaError_t launch_gemm_simt<double>(const double*, int64_t, const double*, int64_t, double*, int64_t,
                                              int64_t, int64_t, int64_t, double, double, cudaStream_t,
                                              const OneProduct&);
template cudaError_t launch_gemm_simt<float>(const float*, int64_t, const float*, int64_t, float*, int64_t, int64_t,
                                             int64_t, int64_t, double, double, cudaStream_t, const OneProduct&);

}  // namespace hotrg
