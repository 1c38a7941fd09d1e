// Gram matrix of a long X in FP32 (see gram.cu).
#pragma once

#include "common.cuh"

namespace rqlp {

struct GramJob {             // G (lower triangle, ldg) = X^T X, X rows x d, d <= 256
  const float* X; int64_t ldx;
  int64_t rows;
  float* G; int64_t ldg;
  const int* gate;           // optional: *gate == 0 -> nothing is written
  int d;
};
// Whether gram_f32 beats the general product, with this much scratch.
bool gram_pays(int64_t rows, int d, size_t part_floats);
// part (16-byte aligned): partial sums of row ranges; more let more SMs take part.
cudaError_t gram_f32(const GramJob& j, float* part, size_t part_floats, cudaStream_t st);

}  // namespace rqlp
