// The tcgen05 training kernels (nn_tc.cu) and their operand layout, used by
// the network's training step (nn.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nn.cuh"

namespace vfisv {
namespace nn {

// Byte offset of element (r, c) of an R x C BF16 matrix in the tiled
// canonical layout TL(R, C): 64-column chunks one after the other (R * 128
// bytes each), 8-row groups of 1024 bytes, 128-byte core matrices of 8 rows
// x 8 columns along K.
__host__ __device__ constexpr size_t tl_off(int64_t r, int c, int64_t R) {
  return (size_t)(c >> 6) * (size_t)R * 128 + (size_t)(r >> 3) * 1024 +
         (size_t)((c & 63) >> 3) * 128 + (size_t)(r & 7) * 16 + (size_t)(c & 7) * 2;
}

// Padded widths of the training operands: the transposed features (24) have
// 32 rows, the outputs (11) and their gradient 16; the packed weights' K is a
// multiple of 64.
constexpr int XK = 64, XT = 32, YN = 16, DYK = 64;

// Forward and backward pass of the rows 0 .. 128 tiles - 1 of a batch, of
// which the first `rows` are samples and the rest padding.
struct TrainPassArgs {
  const float *blob, *obs, *params;
  Perm perm;
  int64_t rows;
  PackedNet P;
  uint8_t *XT, *HT[3];    // transposed features TL(32, M), activations TL(256, M)
  uint8_t *dYT, *dZT[3];  // transposed gradients TL(16, M), TL(256, M)
  float* loss;            // a row's loss (0 on padding), [M]
  int* err;
};
cudaError_t train_pass(const TrainPassArgs& a, int64_t tiles, cudaStream_t s);

// Weight and bias gradients, split over the batch: split s takes K-chunks
// (64 rows) s per .. s per + per - 1 of `chunks`; and the loss of each 256 rows.
struct TrainDwArgs {
  const uint8_t *XT, *HT[3], *dYT, *dZT[3];
  float* wpart[4];  // [splits][256][32: W0^T | 256 | 256 | 16]
  float* bpart[4];  // [splits][256 | 256 | 256 | 16]
  const float* loss;
  float* lossp;
  int nloss, chunks, per;
  int* err;
};
// cudaErrorInvalidValue unless every split owns at least one chunk.
cudaError_t train_dw(const TrainDwArgs& a, int splits, cudaStream_t s);

}  // namespace nn
}  // namespace vfisv
