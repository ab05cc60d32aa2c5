// The paper's own k-means block format: one codebook of 2^b centroids per weight tensor, one bf16 scale per block
// of 64 consecutive inputs of a row, indices packed along the input dimension into bytes (8 / b per byte, LSB
// first), b = 1, 2, 4, 8:   W^[n, k] = scale[n, k / 64] * c[idx[n, k]],   P_w = b + 0.25 bits per weight.
// kmq_block_linear itself is kmq_rows.cu.
#include "kmq_common.cuh"
#include "kmq_rows.cuh"

namespace kmq {
namespace {

constexpr int kBlock = 64;          // inputs per scale
// W[n, k] = bf16(scale * centroid): the product of two bf16 numbers is exact in fp32, one rounding to nearest even.
template <int BITS>
__global__ void __launch_bounds__(256) block_dequant_kernel(const uint8_t* __restrict__ wq,
                                                            const uint16_t* __restrict__ scales,
                                                            const uint16_t* __restrict__ codebook,
                                                            uint16_t* __restrict__ W, int64_t N, int64_t K) {
  constexpr int E = 1 << BITS;
  __shared__ float table[E];
  for (int i = threadIdx.x; i < E; i += blockDim.x) table[i] = bf16_bits_to_float(__ldg(codebook + i));
  __syncthreads();
  const int64_t groups = N * (K / 8);   // 8 weights = BITS bytes in, 16 bytes out
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < groups; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t n = i / (K / 8), k0 = (i % (K / 8)) * 8;
    const uint8_t* src = wq + n * (K * BITS / 8) + k0 * BITS / 8;
    uint64_t bits8 = 0;
#pragma unroll
    for (int b = 0; b < BITS; ++b) bits8 |= (uint64_t)__ldg(src + b) << (8 * b);
    const float s = bf16_bits_to_float(__ldg(scales + n * (K / kBlock) + k0 / kBlock));
    uint32_t o[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t i0 = (uint32_t)(bits8 >> (2 * p * BITS)) & (E - 1), i1 = (uint32_t)(bits8 >> ((2 * p + 1) * BITS)) & (E - 1);
      o[p] = float_to_bf16_bits(s * table[i0]) | (float_to_bf16_bits(s * table[i1]) << 16);
    }
    stg_stream_u4(reinterpret_cast<uint4*>(W + n * K + k0), make_uint4(o[0], o[1], o[2], o[3]));
  }
}

// idx uint8 [N, K] -> bytes [N, K * BITS / 8], fields LSB first; one thread per output byte.
template <int BITS>
__global__ void __launch_bounds__(256) block_pack_kernel(const uint8_t* __restrict__ idx, uint8_t* __restrict__ wq,
                                                         int64_t total_bytes) {
  constexpr int PER = 8 / BITS;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total_bytes; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t out = 0;
#pragma unroll
    for (int f = 0; f < PER; ++f) out |= (uint32_t)(idx[i * PER + f] & ((1u << BITS) - 1u)) << (f * BITS);
    wq[i] = (uint8_t)out;
  }
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

kmq_status check_block_shape(int64_t N, int64_t K, int bits, int64_t M) {
  if (bits != 1 && bits != 2 && bits != 4 && bits != 8) return KMQ_ERR_BITS;
  if (N < 1 || M < 1 || K < kBlock || (K % kBlock) != 0) return KMQ_ERR_SHAPE;
  if (N > (int64_t(1) << 31) || K > (int64_t(1) << 31) || M > (int64_t(1) << 24)) return KMQ_ERR_SHAPE;
  return KMQ_OK;
}

}  // namespace
}  // namespace kmq

using namespace kmq;

extern "C" {

size_t kmq_block_packed_bytes(int64_t N, int64_t K, int bits) {
  return check_block_shape(N, K, bits, 1) == KMQ_OK ? (size_t)N * (size_t)K * bits / 8 : 0;
}

kmq_status kmq_block_pack(const uint8_t* idx, int64_t N, int64_t K, int bits, uint8_t* wq, void* stream) {
  if (!idx || !wq) return KMQ_ERR_NULL;
  if (kmq_status s = check_block_shape(N, K, bits, 1)) return s;
  if (!aligned16(idx) || !aligned16(wq)) return KMQ_ERR_ALIGN;
  const DeviceInfo* di = device_info();
  if (!di) return KMQ_ERR_CUDA;
  const int64_t total = N * K * bits / 8;
  int64_t grid = (total + 255) / 256;
  if (grid > (int64_t)di->sm_count * 16) grid = (int64_t)di->sm_count * 16;
  cudaStream_t s = (cudaStream_t)stream;
  if (bits == 1) block_pack_kernel<1><<<(int)grid, 256, 0, s>>>(idx, wq, total);
  else if (bits == 2) block_pack_kernel<2><<<(int)grid, 256, 0, s>>>(idx, wq, total);
  else if (bits == 4) block_pack_kernel<4><<<(int)grid, 256, 0, s>>>(idx, wq, total);
  else block_pack_kernel<8><<<(int)grid, 256, 0, s>>>(idx, wq, total);
  return cudaGetLastError() == cudaSuccess ? KMQ_OK : KMQ_ERR_CUDA;
}

kmq_status kmq_block_linear(const uint8_t* wq, const uint16_t* scales, const uint16_t* codebook, const uint16_t* x,
                            uint16_t* y, int64_t N, int64_t K, int bits, int64_t M, int scale_order, void* stream) {
  if (!wq || !scales || !codebook || !x || !y) return KMQ_ERR_NULL;
  if (kmq_status s = check_block_shape(N, K, bits, M)) return s;
  if (scale_order != KMQ_SCALE_DIRECT && scale_order != KMQ_SCALE_DEFERRED) return KMQ_ERR_LAYOUT;
  if (!aligned16(wq) || !aligned16(scales) || !aligned16(codebook) || !aligned16(x) || !aligned16(y)) return KMQ_ERR_ALIGN;
  return launch_block_rows(wq, scales, codebook, x, y, N, K, bits, M, (cudaStream_t)stream) == cudaSuccess
             ? KMQ_OK
             : KMQ_ERR_CUDA;
}

kmq_status kmq_block_dequant_to_bf16(const uint8_t* wq, const uint16_t* scales, const uint16_t* codebook, uint16_t* W,
                                     int64_t N, int64_t K, int bits, void* stream) {
  if (!wq || !scales || !codebook || !W) return KMQ_ERR_NULL;
  if (kmq_status s = check_block_shape(N, K, bits, 1)) return s;
  if (!aligned16(wq) || !aligned16(scales) || !aligned16(codebook) || !aligned16(W)) return KMQ_ERR_ALIGN;
  const DeviceInfo* di = device_info();
  if (!di) return KMQ_ERR_CUDA;
  int64_t grid = (N * (K / 8) + 255) / 256;
  if (grid > (int64_t)di->sm_count * 16) grid = (int64_t)di->sm_count * 16;
  cudaStream_t s = (cudaStream_t)stream;
  if (bits == 1) block_dequant_kernel<1><<<(int)grid, 256, 0, s>>>(wq, scales, codebook, W, N, K);
  else if (bits == 2) block_dequant_kernel<2><<<(int)grid, 256, 0, s>>>(wq, scales, codebook, W, N, K);
  else if (bits == 4) block_dequant_kernel<4><<<(int)grid, 256, 0, s>>>(wq, scales, codebook, W, N, K);
  else block_dequant_kernel<8><<<(int)grid, 256, 0, s>>>(wq, scales, codebook, W, N, K);
  return cudaGetLastError() == cudaSuccess ? KMQ_OK : KMQ_ERR_CUDA;
}

}  // extern "C"
