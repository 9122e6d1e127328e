// FP64 GEMM on the CUDA cores: the DMPT products and the back-transformation of small FP64
// systems (up to 256 and 66 basis functions), and all FP64 products where tensor maps are
// not available (tc_gemm64.cu does the others).  Row-major
// C = alpha op(A) op(B) + beta C.  What bounds it is the FP64 pipe (2 FMAs a clock and
// SM), so a tile is as small as its loads allow, one output per thread of a
// 16 x 16 block: no padded work beyond 16 and n^2 / 256 blocks to spread over the SMs;
// the next 16 columns are loaded while the current ones are multiplied.  n = 26, 131,
// 240: 39, 168, 280 us with 64 x 64 tiles of 4 x 4 outputs a thread, 6, 13, 37 so.
// With sym != 0 the result is known to be symmetric (M == N): only
// tiles on or above the diagonal run, and each value is stored at (i, j) and
// (j, i), so the output is bitwise symmetric (D0 = Q f Q^T, Q^T F1 Q and
// Q Y Q^T of eqs. 19 and 36 are symmetric by definition).
#include "common.cuh"
#include "kernels.h"

namespace kx {

constexpr int kGT = 16;     // tile edge and K slice

__global__ void __launch_bounds__(kGT * kGT) dgemm_kernel(int ta, int tb, int M, int N, int K, double alpha,
                                                        const double* __restrict__ A, int lda,
                                                        const double* __restrict__ B, int ldb, double beta,
                                                        double* __restrict__ C, int ldc, int sym, const int* gate) {
  if (gate && *gate == 0) return;
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (sym && bi > bj) return;
  __shared__ double As[2][kGT][kGT + 1];     // [k][i]
  __shared__ double Bs[2][kGT][kGT + 1];     // [k][j]
  const int lo = threadIdx.x % kGT, hi = threadIdx.x / kGT;
  const int m0 = bi * kGT, n0 = bj * kGT;
  // this thread's element of a slice, the fast index along memory
  const int ia = ta ? lo : hi, ka = ta ? hi : lo, jb = tb ? hi : lo, kb = tb ? lo : hi;
  const double* pa = A + (ta ? (size_t)ka * lda + m0 + ia : (size_t)(m0 + ia) * lda + ka);
  const double* pb = B + (tb ? (size_t)(n0 + jb) * ldb + kb : (size_t)kb * ldb + n0 + jb);
  const size_t sa = ta ? (size_t)lda : 1, sb = tb ? 1 : (size_t)ldb;
  const bool ina = m0 + ia < M, inb = n0 + jb < N;
  double va = (ina && ka < K) ? pa[0] : 0.0, vb = (inb && kb < K) ? pb[0] : 0.0;
  double acc = 0.0;
  for (int k0 = 0, s = 0; k0 < K; k0 += kGT, s ^= 1) {
    As[s][ka][ia] = va;
    Bs[s][kb][jb] = vb;
    __syncthreads();                          // (the other buffer was read before the barrier)
    const int kn = k0 + kGT;
    va = (ina && kn + ka < K) ? pa[(size_t)kn * sa] : 0.0;
    vb = (inb && kn + kb < K) ? pb[(size_t)kn * sb] : 0.0;
    const int kk1 = min(kGT, K - k0);
    if (kk1 == kGT) {
#pragma unroll
      for (int kk = 0; kk < kGT; ++kk) acc = fma(As[s][kk][hi], Bs[s][kk][lo], acc);
    } else {
      for (int kk = 0; kk < kk1; ++kk) acc = fma(As[s][kk][hi], Bs[s][kk][lo], acc);
    }
  }
  const int gi = m0 + hi, gj = n0 + lo;
  if (gi >= M || gj >= N || (sym && gi > gj)) return;
  double v = alpha * acc;
  if (beta != 0.0) v += beta * C[(size_t)gi * ldc + gj];
  C[(size_t)gi * ldc + gj] = v;
  if (sym && gi != gj) C[(size_t)gj * ldc + gi] = v;
}

void dgemm(cudaStream_t s, int ta, int tb, int M, int N, int K, double alpha, const double* A, int lda,
           const double* B, int ldb, double beta, double* C, int ldc, int sym, const int* gate) {
  if (M <= 0 || N <= 0) return;
  dim3 grid((N + kGT - 1) / kGT, (M + kGT - 1) / kGT);
  dgemm_kernel<<<grid, kGT * kGT, 0, s>>>(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, sym, gate);
  count_launch();
}

}  // namespace kx
