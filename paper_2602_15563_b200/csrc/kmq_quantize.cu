// Quantiser side of libkmq next to the fit (kmq_fit.cu): nearest-centroid assignment fused with the bit packing, block
// scales of the paper's block format.  Paper: Section 2.1 "Rounding to nearest centroids" (Eq. "centroid quantizer"),
// "Block formats"; Section 2.2 (the two scale functions, "Nonlinear k-means quantization").  Everything that decides
// an index or a stored value is done in float64 with explicit round-to-nearest operations, or in float32 where that is
// exactly the same decision, so that a result does not depend on how the compiler contracts expressions.
#include "kmq_assign.cuh"
#include "kmq_common.cuh"
#include "kmq_fit.cuh"
#include "kmq_table_layout.cuh"

namespace kmq {
namespace {

// CTA (x, y) takes share y of the output words of tile x (16 rows); the tile's thresholds and its lowest-equal-index
// maps sit in shared memory; a thread builds one 32-bit word of the packed output from the float32 weights that word
// covers.
template <int BITS, int LAYOUT>
__global__ void __launch_bounds__(256) assign_pack_kernel(const float* __restrict__ W,
                                                          const uint16_t* __restrict__ codebooks,
                                                          uint32_t* __restrict__ packed, int64_t N, int64_t K) {
  constexpr int Q = 1 << BITS, PER = 32 / BITS;
  __shared__ float thr[16][Q];
  __shared__ uint8_t first[16][Q];
  const int64_t tile = blockIdx.x, wpr = K / PER;
  for (int i = threadIdx.x; i < 16 * (Q - 1); i += blockDim.x) {
    const int r = i / (Q - 1), m = i % (Q - 1);
    const int64_t n = tile * 16 + r;
    if (n < N) thr[r][m] = mid_threshold(exact_mid(codebooks[n * Q + m], codebooks[n * Q + m + 1]));
  }
  if (threadIdx.x < 16 && tile * 16 + threadIdx.x < N) {
    const uint16_t* cb = codebooks + (tile * 16 + threadIdx.x) * Q;
    int f = 0;
    first[threadIdx.x][0] = 0;
    for (int i = 1; i < Q; ++i) {
      if (bf16_bits_to_float(cb[i]) != bf16_bits_to_float(cb[i - 1])) f = i;
      first[threadIdx.x][i] = (uint8_t)f;
    }
  }
  __syncthreads();

  // indices of the 8 weights W[n, k0 .. k0 + 8), one per byte
  auto assign8 = [&](int r, int64_t n, int64_t k0, uint32_t& lo, uint32_t& hi) {
    const float4 a = *reinterpret_cast<const float4*>(W + n * K + k0);
    const float4 b = *reinterpret_cast<const float4*>(W + n * K + k0 + 4);
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    lo = hi = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const uint32_t q = first[r][count_below<BITS>(v[t], thr[r])];
      if (t < 4) lo |= q << (8 * t);
      else hi |= q << (8 * (t - 4));
    }
  };

  if constexpr (LAYOUT == kLayoutPlanes) {
    const int64_t chunks = table_chunks(K);
    const int64_t words = chunks * BITS * 128;
    uint32_t* out = packed + tile * words;
    for (int64_t l = words * blockIdx.y / gridDim.y + threadIdx.x; l < words * (blockIdx.y + 1) / gridDim.y;
         l += blockDim.x) {
      const int64_t unit = l >> 7;
      const int lane = (int)(l & 127) >> 2, q = (int)(l & 3);
      const int plane = (int)(unit % BITS);
      const int64_t chunk = unit / BITS;
      uint32_t word = 0;
#pragma unroll
      for (int bi = 0; bi < 4; ++bi) {
        int r, gl;
        table_unit_coords(lane, 4 * q + bi, r, gl);
        const int64_t n = tile * 16 + r, k0 = (chunk * 32 + gl) * 8;
        if (n < N && k0 < K) {
          uint32_t e[2];
          assign8(r, n, k0, e[0], e[1]);
          uint32_t byte = 0;
#pragma unroll
          for (int t = 0; t < 8; ++t) byte |= ((e[t >> 2] >> ((t & 3) * 8 + plane)) & 1u) << t;
          word |= byte << (8 * bi);
        }
      }
      out[l] = word;
    }
  } else {
    constexpr bool TUNED = LAYOUT == kLayoutTuned;
    const int64_t steps = tuned_steps(wpr);
    const int64_t words = TUNED ? steps * 256 : 16 * wpr;
    for (int64_t l = words * blockIdx.y / gridDim.y + threadIdx.x; l < words * (blockIdx.y + 1) / gridDim.y;
         l += blockDim.x) {
      int r;
      int64_t j;
      if constexpr (TUNED) {
        r = (int)(l >> 4) & 15;
        j = (l >> 8) * 16 + (l & 15);
      } else {
        r = (int)(l / wpr);
        j = l % wpr;
      }
      const int64_t n = tile * 16 + r;
      uint32_t word = 0;
      const bool real = n < N && j < wpr;
      if (real) {
#pragma unroll
        for (int g = 0; g < PER / 8; ++g) {
          uint32_t e[2];
          assign8(r, n, j * PER + g * 8, e[0], e[1]);
#pragma unroll
          for (int t = 0; t < 8; ++t)
            word |= ((e[t >> 2] >> ((t & 3) * 8)) & (uint32_t)(Q - 1)) << field_pos<BITS>(g * 8 + t, TUNED);
        }
      }
      if constexpr (TUNED) packed[tile * words + l] = word;
      else if (real) packed[n * wpr + j] = word;
    }
  }
}

// ---------------------------------------------------------------------------------------------------------------
// Block format: scales, normalised sample, assignment against the shared codebook.
// ---------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t stored_scale(float lambda) {
  const uint32_t bits = float_to_bf16_bits(lambda);
  return bf16_bits_to_float(bits) > 0.0f ? bits : 0x3F80u;      // a zero scale is stored as 1
}
__device__ __forceinline__ float abs_max(float4 v) {
  return fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
}
// absmean adds the 64 magnitudes in float64 in index order
__device__ __forceinline__ double abs_add(double acc, float4 v) {
  acc = __dadd_rn(acc, (double)fabsf(v.x));
  acc = __dadd_rn(acc, (double)fabsf(v.y));
  acc = __dadd_rn(acc, (double)fabsf(v.z));
  return __dadd_rn(acc, (double)fabsf(v.w));
}
__device__ __forceinline__ float mean64(double sum) { return __double2float_rn(__dmul_rn(sum, 1.0 / 64.0)); }

// absmax: half a warp per block of 64 weights, one coalesced 16-byte load per lane; a warp has the loads of eight blocks
// in flight (4096 x 4096: 18.8 us with a thread per block, whose loads were 256 bytes apart).
// `release`: the assignment is next, which waits for this kernel.
__global__ void __launch_bounds__(256) block_absmax_kernel(const float* __restrict__ W, uint16_t* __restrict__ scales,
                                                           int64_t blocks, int release) {
  if (release) asm volatile("griddepcontrol.launch_dependents;");
  const int lane = threadIdx.x & 31, half = lane >> 4, at = lane & 15;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t b0 = warp * 8; b0 < blocks; b0 += warps * 8) {
    float m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t b = b0 + 2 * i + half;
      m[i] = b < blocks ? abs_max(__ldg(reinterpret_cast<const float4*>(W + b * 64) + at)) : 0.0f;
    }
#pragma unroll
    for (int d = 8; d > 0; d >>= 1)
#pragma unroll
      for (int i = 0; i < 4; ++i) m[i] = fmaxf(m[i], __shfl_xor_sync(0xFFFFFFFFu, m[i], d));
    const float mine = at == 0 ? m[0] : at == 1 ? m[1] : at == 2 ? m[2] : m[3];
    const int64_t b = b0 + 2 * at + half;
    if (at < 4 && b < blocks) scales[b] = (uint16_t)stored_scale(mine);
  }
  // Where this runs beside the previous kernel, it must not be complete before that one is: what follows on the stream
  // needs both.  One CTA waits for all (none does when there was no such launch).
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// absmean: 128 blocks at a time are brought to shared memory with coalesced loads (16-byte piece i of block b at
// 129 i + b: conflict-free both ways), then a thread adds up a block.
constexpr int kMeanBlocks = 128;
__global__ void __launch_bounds__(kMeanBlocks) block_absmean_kernel(const float* __restrict__ W,
                                                                    uint16_t* __restrict__ scales, int64_t blocks,
                                                                    int release) {
  if (release) asm volatile("griddepcontrol.launch_dependents;");
  __shared__ float4 piece[16 * (kMeanBlocks + 1)];
  for (int64_t b0 = (int64_t)blockIdx.x * kMeanBlocks; b0 < blocks; b0 += (int64_t)gridDim.x * kMeanBlocks) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int j = i * kMeanBlocks + threadIdx.x, b = j >> 4;
      if (b0 + b < blocks)
        piece[(j & 15) * (kMeanBlocks + 1) + b] = __ldg(reinterpret_cast<const float4*>(W + b0 * 64) + j);
    }
    __syncthreads();
    double acc = 0.0;
#pragma unroll
    for (int i = 0; i < 16; ++i) acc = abs_add(acc, piece[i * (kMeanBlocks + 1) + threadIdx.x]);
    if (b0 + threadIdx.x < blocks) scales[b0 + threadIdx.x] = (uint16_t)stored_scale(mean64(acc));
  }
  if (blockIdx.x == 0) asm volatile("griddepcontrol.wait;" ::: "memory");   // as above
}

__device__ __forceinline__ double normalised(float w, uint32_t scale_bits) {
  return __ddiv_rn((double)w, (double)bf16_bits_to_float(scale_bits));
}

// MODE: how a sampled weight's scale is found: a stored one, or (when the sample is drawn ahead of the scales) worked
// out from its block here.
constexpr int kStoredScales = -1;
template <int MODE>
__global__ void __launch_bounds__(128) block_sample_kernel(const float* __restrict__ W,
                                                           const uint16_t* __restrict__ scales, int64_t K,
                                                           int64_t stride, int64_t count, float* __restrict__ out) {
  // ahead of the scales the fit is next, which waits for the sample
  if constexpr (MODE != kStoredScales) asm volatile("griddepcontrol.launch_dependents;");
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t f = i * stride;                 // a row is a whole number of blocks: block f / 64 of the tensor
  uint32_t scale;
  if constexpr (MODE == kStoredScales) {
    scale = scales[f >> 6];
  } else {
    const float4* const p = reinterpret_cast<const float4*>(W + (f & ~int64_t(63)));
    float4 v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = __ldg(p + q);
    double acc = 0.0;
    float mx = 0.0f;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      if constexpr (MODE == KMQ_LAMBDA_ABSMAX) mx = fmaxf(mx, abs_max(v[q]));
      else acc = abs_add(acc, v[q]);
    }
    scale = stored_scale(MODE == KMQ_LAMBDA_ABSMAX ? mx : mean64(acc));
  }
  out[i] = __double2float_rn(normalised(W[f], scale));
}

// One thread per 8 consecutive weights (they share a block): BITS output bytes.  The index is the number of midpoints
// below the float64 quotient w / scale.  Where a midpoint is itself a float32 (always, short of centroids 2^16 apart)
// the quotient lies above it iff w > mid * scale: the quotient's rounding cannot bridge the gap, because w has 24
// significant bits and mid * scale at most 32; and w, a float32, lies above that product iff it lies above the product
// rounded down.  That is one multiply and one compare per step in place of a float64 division and float64 compares
// (4096 x 4096, b = 4: 60 us with those).
// At b = 4 the 15 steps of the search are one look into a grid of cells over the quotient's approximation w * (1 / scale):
// the grid is only used where an error of 2^-20 in that moves no midpoint across a cell's edge, and the comparison with the
// cell's midpoint is the exact one above.
template <int BITS>
__global__ void __launch_bounds__(256) block_assign_kernel(const float* __restrict__ W,
                                                           const uint16_t* scales, const uint16_t* codebook,
                                                           uint8_t* __restrict__ wq, int64_t groups) {
  constexpr int Q = 1 << BITS;
  __shared__ Mid mids[Q];
  __shared__ float fmid[Q];
  __shared__ uint8_t first[Q];
  __shared__ uint8_t cells[BITS == 4 ? kCells : 4];
  __shared__ uint16_t cb[Q];
  int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const bool wide = (reinterpret_cast<uintptr_t>(W) & 31) == 0;
  // The weights are nobody's output: a thread's first ones are on their way while the scales and the codebook, which the
  // kernels before may still write, are waited for.
  float v[8];
  if (g < groups) ldg_stream_f8(v, W + g * 8, wide);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = threadIdx.x; i < Q; i += blockDim.x) cb[i] = ld_input_u16(codebook + i);
  __syncthreads();
  bool inexact = false, same = false;
  for (int i = threadIdx.x; i < Q - 1; i += blockDim.x) {
    mids[i] = exact_mid(cb[i], cb[i + 1]);
    const double half = __dmul_rn(0.5, mids[i].s);
    fmid[i] = __double2float_rn(half);
    inexact |= mids[i].e != 0.0 || (double)fmid[i] != half;
  }
  for (int i = threadIdx.x; i < Q; i += blockDim.x) {
    int f = i;                                    // equal centroids: the lowest index
    while (f > 0 && bf16_bits_to_float(cb[f]) == bf16_bits_to_float(cb[f - 1])) --f;
    first[i] = (uint8_t)f;
    same |= f != i;
  }
  const bool slow = __syncthreads_or(inexact), duplicates = __syncthreads_or(same);
  const CellGrid grid(fmid, Q - 1);
  bool by_cells = false;
  if constexpr (BITS == 4) {
    if (threadIdx.x == 0) fmid[Q - 1] = __int_as_float(0x7F800000);
    const bool good = grid.fill(cells, threadIdx.x, blockDim.x, fmid, Q - 1, 1.0f / (1 << 20));
    by_cells = !__syncthreads_or(slow || duplicates || !good);
  }
  while (g < groups) {
    const uint32_t sb = ld_input_u16(scales + (g >> 3));
    const float scale = bf16_bits_to_float(sb);
    int n[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (BITS == 4 && by_cells && scale > 1e-30f && scale < 1e30f) {   // 1 / scale is exact to 2^-24
      const float r = __frcp_rn(scale);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        n[k] = cells[grid.of(v[k] * r)];
        n[k] += v[k] > __fmul_rd(fmid[n[k]], scale) ? 1 : 0;
      }
    } else if (!slow) {
      if constexpr (BITS <= 2) {
#pragma unroll
        for (int i = 0; i < Q - 1; ++i) {
          const float t = __fmul_rd(fmid[i], scale);
#pragma unroll
          for (int k = 0; k < 8; ++k) n[k] += v[k] > t ? 1 : 0;
        }
      } else {
#pragma unroll
        for (int step = 1 << (BITS - 1); step > 0; step >>= 1) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (v[k] > __fmul_rd(fmid[n[k] + step - 1], scale)) n[k] += step;
        }
      }
    } else {
      for (int step = 1 << (BITS - 1); step > 0; step >>= 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k)
          if (above(__dmul_rn(2.0, normalised(v[k], sb)), mids[n[k] + step - 1])) n[k] += step;
      }
    }
    if (duplicates) {
#pragma unroll
      for (int k = 0; k < 8; ++k) n[k] = first[n[k]];
    }
    uint64_t bits = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) bits |= (uint64_t)n[k] << (k * BITS);
    uint8_t* dst = wq + g * BITS;
    if constexpr (BITS == 8) *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)bits, (uint32_t)(bits >> 32));
    else if constexpr (BITS == 4) *reinterpret_cast<uint32_t*>(dst) = (uint32_t)bits;
    else if constexpr (BITS == 2) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)bits;
    else *dst = (uint8_t)bits;
    g += stride;
    if (g < groups) ldg_stream_f8(v, W + g * 8, wide);
  }
}

inline int capped_grid(int64_t items, int threads, int sm_count, int per_sm) {
  int64_t blocks = (items + threads - 1) / threads;
  const int64_t cap = (int64_t)sm_count * per_sm;
  if (blocks > cap) blocks = cap;
  return (int)(blocks < 1 ? 1 : blocks);
}

template <int BITS>
cudaError_t launch_assign_bits(const float* W, const uint16_t* cb, int64_t N, int64_t K, int layout, uint32_t* packed,
                               cudaStream_t s) {
  const DeviceInfo* di = device_info();
  if (!di) return cudaErrorInvalidDevice;
  const int64_t tiles = (N + 15) / 16;
  // enough CTAs to fill the machine several times over, each with at least a few words per thread
  int64_t shares = ((int64_t)di->sm_count * 16 + tiles - 1) / tiles;
  const int64_t max_shares = 16 * (K / (32 / BITS)) / 1024;
  if (shares > max_shares) shares = max_shares;
  if (shares < 1) shares = 1;
  if (shares > 65535) shares = 65535;
  const dim3 grid((unsigned)tiles, (unsigned)shares);
  if (layout == KMQ_LAYOUT_CANONICAL) assign_pack_kernel<BITS, kLayoutCanonical><<<grid, 256, 0, s>>>(W, cb, packed, N, K);
  else if (layout == KMQ_LAYOUT_TABLE && BITS != 4)
    assign_pack_kernel<BITS == 4 ? 1 : BITS, kLayoutPlanes><<<grid, 256, 0, s>>>(W, cb, packed, N, K);
  else assign_pack_kernel<BITS, kLayoutTuned><<<grid, 256, 0, s>>>(W, cb, packed, N, K);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_assign_pack(const float* W, const uint16_t* cb, int64_t N, int64_t K, int bits, int layout,
                               uint32_t* packed, cudaStream_t s) {
  if (bits == 1) return launch_assign_bits<1>(W, cb, N, K, layout, packed, s);
  if (bits == 2) return launch_assign_bits<2>(W, cb, N, K, layout, packed, s);
  return launch_assign_bits<4>(W, cb, N, K, layout, packed, s);
}

// `beside_previous`: may run beside the kernel launched before it, of which it needs nothing (programmatic dependent
// launch without a wait; that kernel has to release its dependents).
cudaError_t launch_block_scales(const float* W, int64_t N, int64_t K, int mode, uint16_t* scales, bool beside_previous,
                                cudaStream_t s) {
  const DeviceInfo* di = device_info();
  if (!di) return cudaErrorInvalidDevice;
  const int64_t blocks = N * (K >> 6);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = beside_previous ? 1 : 0;
  if (mode == KMQ_LAMBDA_ABSMAX) {
    cfg.blockDim = dim3(256);
    cfg.gridDim = dim3((unsigned)capped_grid(blocks, 64, di->sm_count, 16));
    return cudaLaunchKernelEx(&cfg, block_absmax_kernel, W, scales, blocks, beside_previous ? 1 : 0);
  }
  cfg.blockDim = dim3(kMeanBlocks);
  cfg.gridDim = dim3((unsigned)capped_grid(blocks, kMeanBlocks, di->sm_count, 6));
  return cudaLaunchKernelEx(&cfg, block_absmean_kernel, W, scales, blocks, beside_previous ? 1 : 0);
}

// mode: kStoredScales, or the scale function (`scales` is then not read)
cudaError_t launch_block_sample(const float* W, const uint16_t* scales, int64_t N, int64_t K, int64_t samples, int mode,
                                float* out, cudaStream_t s) {
  const int64_t total = N * K, stride = total / samples > 1 ? total / samples : 1;
  int64_t count = (total + stride - 1) / stride;
  if (count > samples) count = samples;
  const unsigned grid = (unsigned)((count + 127) / 128);
  if (mode == KMQ_LAMBDA_ABSMAX)
    block_sample_kernel<KMQ_LAMBDA_ABSMAX><<<grid, 128, 0, s>>>(W, scales, K, stride, count, out);
  else if (mode == KMQ_LAMBDA_ABSMEAN)
    block_sample_kernel<KMQ_LAMBDA_ABSMEAN><<<grid, 128, 0, s>>>(W, scales, K, stride, count, out);
  else
    block_sample_kernel<kStoredScales><<<grid, 128, 0, s>>>(W, scales, K, stride, count, out);
  return cudaGetLastError();
}

// `chained`: launched behind launch_block_scales(..., true) on the same stream, may start beside it.
cudaError_t launch_block_assign(const float* W, const uint16_t* scales, const uint16_t* codebook, int64_t N, int64_t K,
                                int bits, bool chained, uint8_t* wq, cudaStream_t s) {
  const DeviceInfo* di = device_info();
  if (!di) return cudaErrorInvalidDevice;
  const int64_t groups = N * (K >> 3);
  const int grid = capped_grid(groups, 256, di->sm_count, 4);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  const auto kernel = bits == 1   ? block_assign_kernel<1>
                      : bits == 2 ? block_assign_kernel<2>
                      : bits == 4 ? block_assign_kernel<4>
                                  : block_assign_kernel<8>;
  return cudaLaunchKernelEx(&cfg, kernel, W, scales, codebook, wq, groups);
}

}  // namespace kmq

using namespace kmq;

namespace {

inline bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline kmq_status st(cudaError_t e) { return e == cudaSuccess ? KMQ_OK : KMQ_ERR_CUDA; }

kmq_status check_fit(int64_t N, int64_t K, int bits, int iters) {
  if (bits != 1 && bits != 2 && bits != 4 && bits != 8) return KMQ_ERR_BITS;
  if (N < 1 || N > (int64_t(1) << 31) || iters < 0 || !fit_supports(K, bits)) return KMQ_ERR_SHAPE;
  return KMQ_OK;
}

kmq_status check_rows(int64_t N, int64_t K, int bits, int layout) {
  if (bits != 1 && bits != 2 && bits != 4) return KMQ_ERR_BITS;
  const int64_t per = 32 / bits;
  if (N < 1 || K < per || (K % per) != 0 || N > (int64_t(1) << 31) || K > (int64_t(1) << 31)) return KMQ_ERR_SHAPE;
  if (layout != KMQ_LAYOUT_CANONICAL && layout != KMQ_LAYOUT_TUNED && layout != KMQ_LAYOUT_TABLE) return KMQ_ERR_LAYOUT;
  return KMQ_OK;
}

kmq_status check_block(int64_t N, int64_t K, int bits) {
  if (bits != 1 && bits != 2 && bits != 4 && bits != 8) return KMQ_ERR_BITS;
  if (N < 1 || K < 64 || (K % 64) != 0 || N > (int64_t(1) << 31) || K > (int64_t(1) << 31)) return KMQ_ERR_SHAPE;
  return KMQ_OK;
}

}  // namespace

extern "C" {

kmq_status kmq_kmeans_rows(const float* W, int64_t N, int64_t K, int bits, int iters, uint16_t* codebooks,
                           double* centroids, void* stream) {
  if (!W || !codebooks) return KMQ_ERR_NULL;
  if (kmq_status s = check_fit(N, K, bits, iters)) return s;
  if (!al16(W) || !al16(codebooks) || !al16(centroids)) return KMQ_ERR_ALIGN;
  return st(launch_kmeans_rows(W, N, K, bits, iters, codebooks, centroids, (cudaStream_t)stream));
}

kmq_status kmq_assign_pack(const float* W, const uint16_t* codebooks, int64_t N, int64_t K, int bits, int layout,
                           uint32_t* packed, void* stream) {
  if (!W || !codebooks || !packed) return KMQ_ERR_NULL;
  if (kmq_status s = check_rows(N, K, bits, layout)) return s;
  if (!al16(W) || !al16(codebooks) || !al16(packed)) return KMQ_ERR_ALIGN;
  return st(launch_assign_pack(W, codebooks, N, K, bits, layout, packed, (cudaStream_t)stream));
}

kmq_status kmq_quantize_rows(const float* W, int64_t N, int64_t K, int bits, int iters, int layout,
                             uint16_t* codebooks, uint32_t* packed, void* stream) {
  if (!W || !codebooks || !packed) return KMQ_ERR_NULL;
  if (kmq_status s = check_rows(N, K, bits, layout)) return s;
  if (kmq_status s = check_fit(N, K, bits, iters)) return s;
  if (!al16(W) || !al16(codebooks) || !al16(packed)) return KMQ_ERR_ALIGN;
  return st(launch_quantize_rows(W, N, K, bits, iters, layout, codebooks, packed, (cudaStream_t)stream));
}

kmq_status kmq_block_scales(const float* W, int64_t N, int64_t K, int lambda, uint16_t* scales, void* stream) {
  if (!W || !scales) return KMQ_ERR_NULL;
  if (kmq_status s = check_block(N, K, 1)) return s;
  if (lambda != KMQ_LAMBDA_ABSMAX && lambda != KMQ_LAMBDA_ABSMEAN) return KMQ_ERR_LAYOUT;
  if (!al16(W) || !al16(scales)) return KMQ_ERR_ALIGN;
  return st(launch_block_scales(W, N, K, lambda, scales, false, (cudaStream_t)stream));
}

int64_t kmq_block_sample_count(int64_t N, int64_t K, int64_t samples) {
  if (check_block(N, K, 1) != KMQ_OK || samples < 1) return 0;
  const int64_t total = N * K, stride = total / samples > 1 ? total / samples : 1;
  const int64_t count = (total + stride - 1) / stride;
  return count < samples ? count : samples;
}

kmq_status kmq_block_sample(const float* W, const uint16_t* scales, int64_t N, int64_t K, int64_t samples, float* out,
                            void* stream) {
  if (!W || !scales || !out) return KMQ_ERR_NULL;
  if (kmq_status s = check_block(N, K, 1)) return s;
  if (samples < 1) return KMQ_ERR_SHAPE;
  if (!al16(W) || !al16(scales) || !al16(out)) return KMQ_ERR_ALIGN;
  return st(launch_block_sample(W, scales, N, K, samples, kStoredScales, out, (cudaStream_t)stream));
}

kmq_status kmq_block_assign_pack(const float* W, const uint16_t* scales, const uint16_t* codebook, int64_t N,
                                 int64_t K, int bits, uint8_t* wq, void* stream) {
  if (!W || !scales || !codebook || !wq) return KMQ_ERR_NULL;
  if (kmq_status s = check_block(N, K, bits)) return s;
  if (!al16(W) || !al16(scales) || !al16(codebook) || !al16(wq)) return KMQ_ERR_ALIGN;
  return st(launch_block_assign(W, scales, codebook, N, K, bits, false, wq, (cudaStream_t)stream));
}

kmq_status kmq_block_quantize(const float* W, int64_t N, int64_t K, int bits, int lambda, int iters, int64_t samples,
                              uint16_t* scales, uint16_t* codebook, uint8_t* wq, float* sample_workspace,
                              void* stream) {
  if (!W || !scales || !codebook || !wq || !sample_workspace) return KMQ_ERR_NULL;
  if (kmq_status s = check_block(N, K, bits)) return s;
  if (lambda != KMQ_LAMBDA_ABSMAX && lambda != KMQ_LAMBDA_ABSMEAN) return KMQ_ERR_LAYOUT;
  const int64_t count = kmq_block_sample_count(N, K, samples);
  if (kmq_status s = check_fit(1, count, bits, iters)) return s;
  if (!al16(W) || !al16(scales) || !al16(codebook) || !al16(wq) || !al16(sample_workspace)) return KMQ_ERR_ALIGN;
  cudaStream_t cs = (cudaStream_t)stream;
  // The fit is one CTA and 28 us (b = 2: 33); the scales of the whole tensor (a full read of it) are worked out beside it.  The
  // sample therefore comes first and finds the scales it needs itself.  Every kernel starts beside the one before it and waits
  // for it before it touches what that wrote: the fit for the sample, one CTA of the scales for the fit, the assignment for the
  // scales, and so for all of them (4096 x 4096, b = 4: 55.4 us; 57.5 to 60 with only the scales beside the fit).  The
  // first kernel waits for all earlier work and the last one releases nothing early: outside, the call is like any other.
  if (launch_block_sample(W, nullptr, N, K, samples, lambda, sample_workspace, cs) != cudaSuccess) return KMQ_ERR_CUDA;
  if (launch_fit_sample(sample_workspace, count, bits, iters, codebook, cs) != cudaSuccess) return KMQ_ERR_CUDA;
  if (launch_block_scales(W, N, K, lambda, scales, true, cs) != cudaSuccess) return KMQ_ERR_CUDA;
  return st(launch_block_assign(W, scales, codebook, N, K, bits, true, wq, cs));
}

}  // extern "C"
