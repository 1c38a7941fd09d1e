// Tensor-core (tcgen05 / TMEM / TMA) products of CholeskyQR in BF16 split precision.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace rqlp {

// cuTensorMapEncodeTiled, or null.
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn();

// True when the tensor-core products can run on the current device (sm_103 with the
// tensor-map encoder available).
bool tc_supported(const float* A, int64_t lda, const float* Omega, int64_t ldo);

// Workspace and launch state of the tensor-core products over one split operand:
// the BF16 parts of a tall X (written by split()) and of the second operand
// (transposed, K-major), and the partial sums of the Gram. Capacities are fixed
// by layout(); split() must be called again whenever X's contents change.
class TcEngine {
 public:
  // rows_cap x cols_cap: largest split X (products and Grams are cols_cap wide at most).
  void layout(Arena& ar, int64_t rows_cap, int cols_cap);
  void reset() { split_of_ = nullptr; }
  // X (rows x cols FP32) -> its parts.
  cudaError_t split(const float* X, int64_t rows, int64_t cols, int64_t lda, cudaStream_t st);
  // out (rows x d) = X_cur B (B cols x d), six products.
  cudaError_t product(const float* B, int64_t ldb, int d, float* out, int64_t ldout, int* info, cudaStream_t st);
  // G (cols x cols, ldg) = X^T X of the current split (cols <= 256).
  cudaError_t gram(float* G, int64_t ldg, int* info, cudaStream_t st);

 private:
  int64_t rows_cap_ = 0, cols_cap_ = 0;
  int G_ = 0;
  int64_t m_ = 0, n_ = 0;   // dims of the current split
  uint16_t *Ahi_ = nullptr, *Alo_ = nullptr, *Alo2_ = nullptr, *Xhi_ = nullptr, *Xlo_ = nullptr, *Xlo2_ = nullptr;
  float* gpart_ = nullptr;
  const float* split_of_ = nullptr;
};

}  // namespace rqlp
