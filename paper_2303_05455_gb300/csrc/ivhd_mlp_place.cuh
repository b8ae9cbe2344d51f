// ivhd_mlp_place.cuh -- the warm-start network applied to rows in one kernel
// (see ivhd_mlp_place.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ivhd {

// The network's operands: BF16 weights of the hidden layers (row-major), FP32
// biases and output layer; err receives a flag if a bounded wait expired.
struct MlpPlace {
  int n_in, hidden;
  const __nv_bfloat16 *w1, *w2;
  const float *b1, *b2, *W3, *b3;
  int32_t* err;
};

// Whether a hidden width is taken (both chunks of 256 columns fit tensor memory).
bool mlp_place_supported(int hidden);

// The rows to give mlp_place at once, at most max_rows: whole rounds of tiles over the SMs.
int mlp_place_rows(int max_rows);

// y (rows x 2; 8-byte aligned) of `rows` BF16 rows x; y_copy (may be null) gets the same values.
cudaError_t mlp_place(const MlpPlace& P, int rows, const __nv_bfloat16* x, float* y, float* y_copy,
                      cudaStream_t s);

}  // namespace ivhd
