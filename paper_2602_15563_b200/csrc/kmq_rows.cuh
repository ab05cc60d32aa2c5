// The layer on row-major packed weights: the canonical layout (a codebook per row) and the paper's block format in its
// byte layout (a shared codebook, a bf16 scale per block of 64).  Launchers of kmq_rows.cu.
#pragma once
#include "kmq_common.cuh"

namespace kmq {

// canonical layout, any legal shape
cudaError_t launch_linear_rows(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N,
                               int64_t K, int bits, int64_t M, cudaStream_t s);
// its batch rows per launch
int linear_rows_per_launch();

// block format, bits = 1, 2, 4, 8, K a multiple of 64
cudaError_t launch_block_rows(const uint8_t* wq, const uint16_t* scales, const uint16_t* codebook, const uint16_t* x,
                              uint16_t* y, int64_t N, int64_t K, int bits, int64_t M, cudaStream_t s);

}  // namespace kmq
