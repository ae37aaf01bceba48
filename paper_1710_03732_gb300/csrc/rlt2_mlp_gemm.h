// The tcgen05 GEMM of the learned start's training (umma_gemm.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace rlt2 {

// C[M x N] = A[M x K] B[K x N], BF16 operands, FP32 accumulation on tcgen05.
struct UmmaGemmArgs {
  int M, N, K;               // N <= 256 and a multiple of 8; K a multiple of 64
  const __nv_bfloat16* A;    // a_kmajor: A(m, k) at A[m * lda + k]; else at A[k * lda + m]
  int lda;
  bool a_kmajor;
  const __nv_bfloat16* B;    // b_kmajor: B(k, n) at B[n * ldb + k]; else at B[k * ldb + n]
  int ldb;
  bool b_kmajor;
  int epi;                   // 0: FP32 C (atomic add when K is split), 1: bias + ReLU -> BF16 Cb,
                             // 2: masked by mask > 0 -> BF16 Cb (C, Cb, mask: leading dimension ldc)
  float* C;
  int ldc;
  __nv_bfloat16* Cb;
  const float* bias;
  const __nv_bfloat16* mask;
  int* err;                  // set on a timed-out wait
  int kps;                   // K per split (set by umma_gemm)
  unsigned tmem_cols;        // TMEM columns allocated (set by umma_gemm)
  int withhold;              // diagnostics (tall products): issue no MMA and no commit, so that
                             // the bounded waits run out (failure detection without a fault)
};

// How many ways the K = batch rows of a weight gradient are split over CTAs (grid.z)
// where each part is `blocks` CTAs, on a device of `sms` SMs.  Accuracy sets the least
// number: a part is one FP32 accumulator in the tensor cores, which cut each sum
// rather than round it, so its error grows with the rows that it sums: at most 1,024
// (512 up to 32,768 rows; below 2,048 rows no split).  From there up to whole rounds of one
// CTA per SM, or up to one round of parts of 256 rows.  256 x 256 over 65,536 rows,
// error against FP64 and time: 64 parts 4.0e-7, 55 us; 74, two rounds, 3.6e-7, 49;
// one round (38) 6.9e-7, 45.  262,144 rows: 256 parts 4.7e-7, 187 us; one round 3.7e-6,
// 162.  8,192 rows: 16 parts 1.9e-7, 18.4 us; 32 1.4e-7, 12.3.
inline int wgrad_parts(int K, int blocks, int sms) {
  if (K < 2048) return 1;
  const int by_1024 = K < 256 * 1024 ? (K + 1023) / 1024 : 256, by_512 = K < 64 * 512 ? (K + 511) / 512 : 64;
  const int least = by_1024 > by_512 ? by_1024 : by_512;
  const int round = blocks < sms ? sms / blocks : 1;  // parts of one round
  if (least > round) return (least + round - 1) / round * round;
  const int by_256 = K / 256 < round ? K / 256 : round;
  return least > by_256 ? least : by_256;
}

// Shapes the kernel takes (the caller falls back to the mma.sync GEMM otherwise).
bool umma_gemm_supported(int M, int N, int K);
// Launches the GEMM with K split `splits` ways (grid.z); EPI 0 adds atomically when split.
cudaError_t umma_gemm(UmmaGemmArgs a, int splits, cudaStream_t s);

}  // namespace rlt2
