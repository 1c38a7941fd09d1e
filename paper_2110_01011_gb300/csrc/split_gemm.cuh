// out = op(A) X on the tensor cores with A read in FP32 and split into BF16
// parts on its way to tensor memory (see split_gemm.cu).
#pragma once

#include "common.cuh"

namespace rqlp {

// Scratch of split_gemm for products with K <= k_cap and N <= n_cap, laid out
// once in the caller's workspace. The words and the tile counters must be zero
// before the first product of a call (split_gemm_reset); the block (X's image
// and the partial tiles) carries nothing from one product to the next.
struct SplitGemmWs {
  uint16_t* img = nullptr;   // X's parts as shared-memory stage images
  float* part = nullptr;     // partial tiles of split K ranges
  int* words = nullptr;      // [0..1] X low part nonzero, [2..3] sums that are not finite, by turn
  int* cnt = nullptr;        // tile arrival counters
  size_t words_bytes = 0;    // words and counters, one block
  int slots = 0;             // 128-row partial slots that fit in part
  int turn = 0;
  int stall = 0;             // fault-injection tests: see Args::stall
};
// Block that serves every product at full width (16-byte aligned); parts: 2 or
// 3 (the largest used).
size_t split_gemm_block_bytes(int64_t k_cap, int n_cap, int parts);
// m_cap: largest number of output rows. The words come from `ar`, the block is
// given (bytes may be fewer than the above: fewer CTAs then take a product).
// False when the block is too small for half of the SMs.
bool split_gemm_layout(Arena& ar, SplitGemmWs* ws, void* block, size_t bytes, int64_t m_cap, int64_t k_cap, int n_cap,
                       int parts);
cudaError_t split_gemm_reset(SplitGemmWs* ws, cudaStream_t st);

// kSplitTwo: two parts, three products (BF16x3 form); kSplitThree: three parts,
// six products, chains as in the BF16x3 form; kSplitFp32: three parts, short
// chains, FP32 accuracy.
enum SplitMode { kSplitTwo = 2, kSplitThree = 3, kSplitFp32 = 4 };

// transA: out (M x N) = A^T X with A K x M; else out = A X with A M x K; X is
// K x N (N <= 256), all row-major FP32. sumsq (optional) += sum of squares of
// A. *range_word (optional) receives the device word that a kSplitFp32 product
// raises when a sum is not finite, because of values of A or X that are not or
// are too large for the form (split_device.cuh), or because a wait ran out: the
// result then has to be recomputed in FP32, gated on that word, before the next
// product, which clears it. Null in the other modes, where results that a wait lost
// are NaN.
cudaError_t split_gemm(SplitGemmWs* ws, bool transA, int64_t M, int N, int64_t K, const float* A, int64_t lda,
                       const float* X, int64_t ldx, float* out, int64_t ldo, SplitMode mode, double* sumsq,
                       const int** range_word, int* info, bool profiled, cudaStream_t st);

// ---------------------------------------------------------------- grouped products (batched form)
struct SplitJob {           // out (M x N) = op(A) X
  const void* maps;         // tensor maps over A and X's parts, on the device (split_job_maps)
  float* out;
  long long ldo;
  const int* xlo;           // raised when X has a low part
  int* bad;                 // raised on sums that are not finite (FP32; else null)
  double* sumsq;            // += sum of squares of A (or null)
  int M, N, npad, kb, vec_out;
  uint32_t idesc;
  int shift[4], past[4];
};
struct SplitXJob {          // X (K x N) -> stage images
  const float* X;
  long long ldx, K;
  uint16_t* img;
  int* xlo;
  int N, npad;
};
constexpr size_t kSplitMapBytes = 5 * 128;   // five tensor maps
// Encodes the maps of A (rows x cols, row stride lda; A K x M when trans) and of
// X's parts (`img`, written by split_x_grouped) into host memory (128-byte
// entries) and sets the job's shifts. The job's kb and npad are set before.
bool split_job_maps(void* maps, SplitJob* j, const float* A, int64_t rows, int64_t cols, int64_t lda, bool trans,
                    const uint16_t* img, int parts);
int split_npad(int n);
size_t split_image_bytes(int64_t K, int n, int parts);
uint32_t split_idesc(int npad);
int split_x_blocks(int64_t K, int npad);
// start: count + 1 block prefix sums (split_x_blocks).
cudaError_t split_x_grouped(const SplitXJob* jobs, const int* start, int count, int total, SplitMode mode,
                            cudaStream_t st);
// units: (job, 256-row tile) pairs, N <= 128; CTA pair p takes units
// cta_start[p] .. cta_start[p + 1] - 1. pairs = 0 only configures the kernel
// (call before capturing). stall != 0 (fault-injection tests): CTA 0 withholds
// its first stage of X, its bounded waits run out and `info` receives
// RQLP_ERR_TIMEOUT.
cudaError_t split_grouped(bool transA, const SplitJob* jobs, const int2* units, const int* cta_start, int pairs,
                          int npad_max, SplitMode mode, int* info, int stall, cudaStream_t st);

}  // namespace rqlp
