// kmq_dequant_to_bf16: W^[n,k] = C_n[idx[n,k]] as a dense bf16 matrix.
// The kernels are bound by the 2-byte-per-weight output stream.  A warp has a share of one row, up to kBatch x 32 chunks of
// 8 weights: it loads the packed bits of all of them, then decodes and stores, 16 bytes a lane, consecutive lanes writing
// consecutive pieces.  CTAs are short and many, dealt out by the hardware: SMs do not all reach memory equally fast, and a
// grid that stays resident, with equal shares for all, ends with the slowest (470 MB of plain stores: 76.6 us from 1184 CTAs
// in a loop, 64 to 68 us from 9472 and more).  8192 x 28672, b = 4 106.0 -> 92.4 us.
#include "kmq_common.cuh"
#include "kmq_mma_common.cuh"
#include "kmq_table_layout.cuh"

namespace kmq {
namespace {

// 8 weights (8*BITS index bits, fields LSB first) -> 8 bf16 = one 16-byte value.
template <int BITS>
__device__ __forceinline__ uint4 decode8(uint32_t v, uint32_t c0, uint32_t c1, const uint16_t* __restrict__ row_cb) {
  uint32_t o[4];
  if constexpr (BITS == 1) {
    // codebook = 4 bytes {c0, c1}; a selector nibble pair picks bytes (2i, 2i+1)
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t i0 = (v >> (2 * p)) & 1u, i1 = (v >> (2 * p + 1)) & 1u;
      o[p] = __byte_perm(c0, c0, 0x1010u + i0 * 0x22u + i1 * 0x2200u);
    }
  } else if constexpr (BITS == 2) {
    // codebook = 8 bytes {c0,c1 | c2,c3}: byte pair (2i, 2i+1) of the two words
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t i0 = (v >> (4 * p)) & 3u, i1 = (v >> (4 * p + 2)) & 3u;
      o[p] = __byte_perm(c0, c1, 0x1010u + i0 * 0x22u + i1 * 0x2200u);
    }
  } else {
    // c0 = this lane's share of the row's codebook: centroid (lane % 16) in the low half word.  A lookup is a
    // shuffle from the lane that holds the entry (all 32 lanes of the warp must be here); two lookups are packed
    // by one PRMT.  This keeps the 16 entries out of the load path, which the packed words and the stores need.
    (void)row_cb;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const uint32_t i0 = (v >> (8 * p)) & 15u, i1 = (v >> (8 * p + 4)) & 15u;
      const uint32_t lo = __shfl_sync(0xFFFFFFFFu, c0, (int)i0), hi = __shfl_sync(0xFFFFFFFFu, c0, (int)i1);
      o[p] = __byte_perm(lo, hi, 0x5410u);
    }
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// 8 weights of the tuned layout (b = 1, 2), whose fields lie where few instructions take several: one shift and the decoders of
// the tensor-core kernels.  Cutting the fields out one by one and putting them back in order for decode8 took more integer
// instructions than the stores left time for: 8192 x 28672, b = 1 100.5 us, so 76.2; b = 2 96.5, so 82.8.
template <int BITS>
struct TunedDecoder {};
template <>
struct TunedDecoder<1> : Dec1 {
  // fields 2c', 2c'+1 at bits 15 - c', 31 - c'; chunk q holds c' = 4q .. 4q+3
  __device__ __forceinline__ uint4 chunk(uint32_t t, int q) const {
    const uint32_t u = t << (4 * q);
    return make_uint4(select(u), select(u << 1), select(u << 2), select(u << 3));
  }
};
template <>
struct TunedDecoder<2> : Dec2 {
  // field 4p + c' at bits 2p + 8c'; chunk q holds p = 2q, 2q+1
  __device__ __forceinline__ uint4 chunk(uint32_t t, int q) const {
    const uint32_t u = t >> (4 * q);
    uint4 o;
    pair(u, 0, o.x, o.y);
    pair(u, 1, o.z, o.w);
    return o;
  }
};

template <int BITS>
__device__ __forceinline__ void load_codebook(const uint16_t* __restrict__ row_cb, uint32_t& c0, uint32_t& c1) {
  c0 = c1 = 0;
  if constexpr (BITS == 1) c0 = __ldg(reinterpret_cast<const uint32_t*>(row_cb));
  if constexpr (BITS == 2) {
    const uint2 cw = __ldg(reinterpret_cast<const uint2*>(row_cb));
    c0 = cw.x;
    c1 = cw.y;
  }
  if constexpr (BITS == 4) c0 = __ldg(row_cb + (threadIdx.x & 15));
}

constexpr int kWarps = 8, kBatch = 4;

// Shares of a row (in chunks of 8 weights) and the grid for N rows; CTAs beyond the largest grid are made up for by a loop.
inline int row_shares(int64_t K) { return (int)((K / 8 + 32 * kBatch - 1) / (32 * kBatch)); }
inline unsigned share_grid(int64_t N, int64_t K) {
  const int64_t ctas = (N * row_shares(K) + kWarps - 1) / kWarps;
  return (unsigned)(ctas < (int64_t(1) << 30) ? ctas : int64_t(1) << 30);
}

// f(row, first chunk) for every share of this warp.
template <class F>
__device__ __forceinline__ void for_each_share(int64_t N, int shares, F f) {
  const int64_t all = N * shares;
  for (int64_t t = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); t < all; t += (int64_t)gridDim.x * kWarps) {
    const int64_t n = all <= 0xFFFFFFFFll ? (int64_t)((uint32_t)t / (uint32_t)shares) : t / shares;
    f(n, (int)(t - n * shares) * (32 * kBatch));
  }
}

// In the tuned layout the row's words come in 64-byte runs, one per 1 KB step of its tile.
template <int BITS, bool TUNED>
__global__ void __launch_bounds__(kWarps * 32) dequant_rows_kernel(const uint32_t* __restrict__ packed,
                                                                   const uint16_t* __restrict__ cb,
                                                                   uint16_t* __restrict__ W, int64_t N, int64_t K,
                                                                   int shares) {
  constexpr int Q = 1 << BITS;
  constexpr int CPW = 4 / BITS;                  // 8-weight chunks per word
  const int cpr = (int)(K >> 3);                 // 8-weight chunks per row
  const int64_t wpr = K / (32 / BITS);           // words per row
  const int64_t steps = tuned_steps(wpr);
  for_each_share(N, shares, [&](int64_t n, int first) {
    const uint32_t* row_words =
        TUNED ? packed + ((n >> 4) * steps * kTileRows + (n & 15)) * 16 : packed + n * wpr;
    const uint16_t* row_cb = cb + n * Q;
    constexpr bool kFields = TUNED && BITS != 4;
    TunedDecoder<kFields ? BITS : 1> dec;
    uint32_t c0, c1;
    if constexpr (kFields) dec.init(row_cb);
    else load_codebook<BITS>(row_cb, c0, c1);
    uint4* const out = reinterpret_cast<uint4*>(W + n * K);
    const int c_lane = first + (threadIdx.x & 31);
    uint32_t t[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int c = c_lane + 32 * i, j = c / CPW;
      t[i] = 0;
      if (c >= cpr) continue;
      if constexpr (TUNED) t[i] = __ldg(row_words + (int64_t)(j >> 4) * 256 + (j & 15));
      else if constexpr (BITS == 4) t[i] = __ldg(row_words + c);
      else if constexpr (BITS == 2) t[i] = __ldg(reinterpret_cast<const uint16_t*>(row_words) + c);
      else t[i] = __ldg(reinterpret_cast<const uint8_t*>(row_words) + c);
    }
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int c = c_lane + 32 * i;
      if (first + 32 * i >= cpr) break;          // whole warps: at b = 4 the lanes look centroids up for each other
      uint4 w8;
      if constexpr (kFields) w8 = dec.chunk(t[i], c % CPW);
      else w8 = decode8<BITS>(t[i], c0, c1, row_cb);
      if (c < cpr) stg_stream_u4(out + c, w8);
    }
  });
}

// Four bits -> the lowest bits of four bytes.
__device__ __forceinline__ uint32_t spread(uint32_t nibble) { return (nibble & 15u) * 0x00204081u; }

// Table (bit-plane) layout: a thread gathers the plane bytes of one group of 8 weights and stores the 8 decoded weights as one
// 16-byte piece.  b = 2: the planes' bits are spread to the bytes of a word of four indices by multiplies; bit by bit 8192 x 28672
// took 108 us, so 92.6.
template <int BITS>
__global__ void __launch_bounds__(kWarps * 32) dequant_table_kernel(const uint32_t* __restrict__ packed,
                                                                    const uint16_t* __restrict__ cb,
                                                                    uint16_t* __restrict__ W, int64_t N, int64_t K,
                                                                    int shares) {
  constexpr int Q = 1 << BITS;
  const uint8_t* bytes = reinterpret_cast<const uint8_t*>(packed);
  const int gpr = (int)(K >> 3);
  const int64_t chunks = table_chunks(K);
  for_each_share(N, shares, [&](int64_t n, int first) {
    const uint16_t* row_cb = cb + n * Q;
    Dec2 dec;
    uint32_t c0, c1;
    if constexpr (BITS == 2) dec.init(row_cb);
    else load_codebook<BITS>(row_cb, c0, c1);
    uint4* const out = reinterpret_cast<uint4*>(W + n * K);
    const int g_lane = first + (threadIdx.x & 31);
    uint32_t plane[kBatch][BITS];
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
#pragma unroll
      for (int p = 0; p < BITS; ++p)
        plane[i][p] = g_lane + 32 * i < gpr ? __ldg(bytes + table_byte_offset(n, g_lane + 32 * i, p, chunks, BITS)) : 0;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      const int g = g_lane + 32 * i;
      if (g >= gpr) break;
      if constexpr (BITS == 2) {
        uint4 o;
        dec.pair((spread(plane[i][0]) & 0x01010101u) | (spread(plane[i][1]) << 1 & 0x02020202u), 0, o.x, o.y);
        dec.pair((spread(plane[i][0] >> 4) & 0x01010101u) | (spread(plane[i][1] >> 4) << 1 & 0x02020202u), 0, o.z, o.w);
        stg_stream_u4(out + g, o);
      } else {
        stg_stream_u4(out + g, decode8<BITS>(plane[i][0], c0, c1, row_cb));
      }
    }
  });
}

}  // namespace

cudaError_t launch_dequant(const uint32_t* packed, const uint16_t* cb, uint16_t* W, int64_t N, int64_t K, int bits,
                           int layout, cudaStream_t s) {
  const bool tuned = layout != KMQ_LAYOUT_CANONICAL;
  const int shares = row_shares(K);
  const unsigned grid = share_grid(N, K);
  constexpr int kThreads = kWarps * 32;
  if (layout == KMQ_LAYOUT_TABLE && bits != 4) {
    if (bits == 1) dequant_table_kernel<1><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
    else dequant_table_kernel<2><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
    return cudaGetLastError();
  }
  if (bits == 1 && tuned) dequant_rows_kernel<1, true><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  else if (bits == 1) dequant_rows_kernel<1, false><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  else if (bits == 2 && tuned) dequant_rows_kernel<2, true><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  else if (bits == 2) dequant_rows_kernel<2, false><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  else if (tuned) dequant_rows_kernel<4, true><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  else dequant_rows_kernel<4, false><<<grid, kThreads, 0, s>>>(packed, cb, W, N, K, shares);
  return cudaGetLastError();
}

}  // namespace kmq
