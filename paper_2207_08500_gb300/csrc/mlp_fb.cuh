// What the training step (mlp_train.cu) and the FP32 loss gradient (mlp_bwd.cu)
// share: the parameter layout of the 6-64-32-16-8-4 ReLU network of Sec. 3.1
// (weights-file order: per layer W[out][in] then b[out]), the rows in which every
// layer's input and every delta are staged feature-major in shared memory, and the
// loss term of Eq. (Crossentropy).
#pragma once

#include <cmath>

#include "internal.h"

namespace neno6 {
namespace mlpfb {

// parameter offsets and layer widths
__host__ __device__ constexpr int wofs(int l) { return l == 0 ? 0 : l == 1 ? 448 : l == 2 ? 2528 : l == 3 ? 3056 : 3192; }
__host__ __device__ constexpr int wid(int l) { return l == 0 ? 6 : l == 1 ? 64 : l == 2 ? 32 : l == 3 ? 16 : l == 4 ? 8 : 4; }
// staged rows: inputs x0 (6) x1 (64) x2 (32) x3 (16) x4 (8); deltas d1..d5
constexpr int kX0 = 0, kX1 = 6, kX2 = 70, kX3 = 102, kX4 = 118;
constexpr int kD1 = 126, kD2 = 190, kD3 = 222, kD4 = 238, kD5 = 246, kRows = 250;

__device__ __forceinline__ float softplus(float z) {  // log(1 + e^z), stable
  return fmaxf(z, 0.0f) + log1pf(__expf(-fabsf(z)));
}

}  // namespace mlpfb
}  // namespace neno6
