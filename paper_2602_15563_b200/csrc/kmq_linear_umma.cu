// kmq_linear on the tuned (tile-major) layout for large batches: the 5th-generation tensor core (tcgen05.mma)
// multiplies dequantised bf16 weights, held in tensor memory, with the activations in shared memory; the accumulator
// lives in tensor memory too.
//
// One CTA owns 128 output rows (8 tiles of 16) and walks its share of K in stages of 128 weights per row.  Its 16
// decoder warps, one MMA warp and one TMA producer warp meet only through mbarriers:
//   * the decoder threads copy the packed words of the CTA's 8 tiles, one 1 KB step per tile at a time, global ->
//     shared with coalesced cp.async (ring of kWRing steps, rows padded to 80 bytes; one named barrier per step).
//     Decoder thread (warp w, lane l) owns output row 32 (w % 4) + l of the CTA -- the tensor-memory lane a warp may
//     write is fixed by its index -- and quarter w / 4 of each stage's weights of that row: it reads its 4..16 bytes
//     from the ring, rebuilds the 32 weights as bf16 pairs in registers and writes them with tcgen05.st into the A
//     operand of the stage (lane = row, 32-bit column c = weights 2c, 2c + 1 of the stage; ring of kARing stages).
//     When a warp's part of a stage is in place it arrives on the stage's `full` barrier;
//   * the producer thread copies the activations under a stage (NB batch rows x 128, zero-filled past M and past K)
//     with two TMA tile loads (cp.async.bulk.tensor, 64 columns = 128 bytes wide, 128-byte swizzle) into the B
//     buffer of the stage, up to a whole ring ahead; their bytes complete the same `full` barrier;
//   * the MMA thread waits for `full`, issues 8 tcgen05.mma (128 x NB x 16 each) that add into the accumulator
//     D[128 output rows][NB batch rows], and commits them to the stage's `empty` barrier, which the decoders and the
//     producer wait for before they overwrite the A operand and the B buffer.
// When the 128-row blocks alone would leave half of the SMs idle, K is split over a cluster of 2 CTAs: each
// accumulates its half, CTA 1 writes its accumulator into CTA 0's shared memory (st.shared::cluster between two
// cluster barriers), CTA 0 adds the two in a fixed order.  At the end the decoder warps read the accumulator with
// tcgen05.ld (lane = output row, column = batch row), round to bf16 and store.
//
// Every wait on an mbarrier is bounded; a warp whose wait runs out sets bit 0 of the device error word and goes to
// the end of the kernel (so does, after its own bounded waits, every warp that depended on it); every thread still
// takes part in the cluster barriers and the final CTA barrier, after which the tensor memory is freed.
#include "kmq_umma_common.cuh"

namespace kmq {

using namespace umma;

__device__ unsigned int g_device_error_flags = 0;   // sticky; read and cleared by kmq_device_error_flags()

namespace {

// Stages in flight: A operands in tensor memory (the decoders may run this far ahead of the MMAs) and, one per A
// operand, B buffers in shared memory.  6, or 4 for more than 64 batch rows (128 columns of accumulator, 32 KB per B
// buffer).
template <int NB>
constexpr int ring_depth() {
  return NB > 64 ? 4 : 6;
}
template <int BITS, int NB>
struct USmem {
  static constexpr int kARing = ring_depth<NB>();
  static constexpr int kBRing = kARing;
  static constexpr int kTmemCols = 512;                             // kARing * 64 columns of A + NB columns of D <= 512
  static_assert(kARing * 64 + NB <= 512, "tensor memory has 512 columns");
  static constexpr int kBHalfBytes = NB * 128;                      // NB rows x 64 activations (one TMA box)
  static constexpr int kBStageBytes = 2 * kBHalfBytes;
  static constexpr int kB = 0;
  static constexpr int kWords = kB + kBRing * kBStageBytes;   // ring of packed words: [step][row][80]
  static constexpr int kBars = kWords + kWRing * kWStepBytes;   // full[kARing], empty[kARing]
  static constexpr int kTmemSlot = kBars + 2 * kARing * 8;   // then a word that a failed wait sets
  static constexpr int kTotal = kTmemSlot + 16 + 1024;   // + room to align the base to 1024 bytes (swizzled B buffers)
};

// Instruction descriptor of kind::f16: D fp32, A and B bf16, both K-major, M = kBM, N = NB.
template <int NB>
__device__ __forceinline__ uint32_t instr_desc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

template <int BITS, int NB>
__global__ void __launch_bounds__(kThreads, 1) linear_umma_kernel(const uint32_t* __restrict__ packed,
                                                                  const uint16_t* __restrict__ cb,
                                                                  const __grid_constant__ CUtensorMap xmap,
                                                                  uint16_t* __restrict__ y, int64_t N, int64_t K,
                                                                  int64_t M) {
  using G = UGeo<BITS>;
  using SM = USmem<BITS, NB>;
  constexpr int SPS = G::kStagesPerStep;
  constexpr int NW = G::kThreadBytes / 4;   // packed words per thread and stage: 4, 2, 1
  constexpr int kARing = SM::kARing;
  constexpr int kReaders = NB % 32 == 0 ? 4 : 2;   // warps per lane quarter that read the accumulator
  constexpr int kReadCols = NB / kReaders;         // columns each of them reads (a multiple of 8)
  extern __shared__ __align__(1024) unsigned char smem_unaligned[];
  unsigned char* const smem_raw =
      smem_unaligned + ((1024u - ((uint32_t)__cvta_generic_to_shared(smem_unaligned) & 1023u)) & 1023u);
  const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t b_addr = smem_base + SM::kB;
  const uint32_t full_bar = smem_base + SM::kBars, empty_bar = full_bar + 8 * kARing;
  volatile uint32_t* const tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t block_row0 = (int64_t)blockIdx.x * kBM;
  const int64_t m0 = (int64_t)blockIdx.z * NB;   // first batch row of this CTA's tile
  const int steps = (int)tuned_row_steps(K, BITS);
  // K is split over the gridDim.y CTAs of a cluster (same output rows): rank r takes steps [s_begin, s_end)
  const int ksplit = gridDim.y, rank = blockIdx.y;
  const int s_begin = (int)((int64_t)steps * rank / ksplit), s_end = (int)((int64_t)steps * (rank + 1) / ksplit);
  const int my_steps = s_end - s_begin;
  const int total = my_steps * SPS;             // stages of this CTA

  // ---- set-up: mbarriers, tensor memory ----
  if (threadIdx.x == 0) {
    *reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot + 4) = 0;
#pragma unroll
    for (int i = 0; i < kARing; ++i) {
      // decoder warps + the producer's arrive-and-expect; the TMA bytes complete the same phase
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full_bar + 8 * i), "r"(kDecodeWarps + 1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty_bar + 8 * i) : "memory");
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kDecodeWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_base + SM::kTmemSlot),
                 "r"((uint32_t)SM::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_d = tmem_base + kARing * G::kCols;   // the accumulator follows the A operands
  bool ok = true;

  if (warp < kDecodeWarps) {
    // ================= decoder warps =================
    const int q = warp & 3, kh = warp >> 2;   // tensor-memory lane quarter; which quarter of a stage's weights
    const int rho = 32 * q + lane;            // output row inside the CTA = tensor-memory lane
    const int64_t tiles = (N + kTileRows - 1) / kTileRows;
    // row rho % 16 of a tile owns bytes [64 (rho % 16), +64) of each 1 KB step; rows of a tile past N decode zeros
    // and are never stored
    RowState<BITS> st;
    st.d.init(cb + min(block_row0 + rho, N - 1) * (1 << BITS));
    // packed words: whole 1 KB steps of the CTA's 8 tiles, global -> shared, coalesced (thread j copies 16-byte piece
    // j % 64 of tile j / 64 = piece j % 4 of row j / 4), one cp.async group per step, kWRing - 1 steps in flight
    const unsigned char* const w_row = smem_raw + SM::kWords + rho * kWRowStride + kh * G::kThreadBytes;
    const int cj = threadIdx.x;
    const int64_t c_tile = (int64_t)blockIdx.x * (kBM / 16) + (cj >> 6);
    const unsigned char* const c_src =
        reinterpret_cast<const unsigned char*>(packed) + ((c_tile < tiles ? c_tile : 0) * (int64_t)steps + s_begin) * 1024 +
        (cj & 63) * 16;
    const uint32_t c_dst = smem_base + SM::kWords + (cj >> 2) * kWRowStride + (cj & 3) * 16;
    auto copy_step = [&](int s) {
      if (s < my_steps) cp_async16(c_dst + (s % kWRing) * kWStepBytes, c_src + (int64_t)s * 1024, c_tile < tiles);
      cp_async_commit();
    };
    volatile uint32_t* const fail_word = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot + 4);
#pragma unroll 1
    for (int d = 0; d < kWRing - 1; ++d) copy_step(d);
    int i = 0;   // stage
    for (int s = 0; s < my_steps; ++s) {
      cp_async_wait<kWRing - 2>();   // this thread's piece of step s has landed
      // every decoder thread's piece of step s has landed, and every one is done with step s - 1
      asm volatile("bar.sync 1, %0;" ::"n"(kDecodeThreads) : "memory");
      if (*fail_word) {   // some warp's wait ran out: all decoders leave together
        ok = false;
        break;
      }
      copy_step(s + kWRing - 1);     // into the slot of step s - 1
      const unsigned char* const w_step = w_row + (s % kWRing) * kWStepBytes;
#pragma unroll
      for (int u = 0; u < SPS; ++u, ++i) {
        const int abuf = i % kARing;
        // the stage's bytes of the row: [u * 64 / SPS, +64 / SPS) of its 64 bytes in the step; this thread's quarter
        uint32_t wv[NW];
        if constexpr (NW == 4) {
          const uint4 t4 = *reinterpret_cast<const uint4*>(w_step + u * (64 / SPS));
          wv[0] = t4.x; wv[1] = t4.y; wv[2] = t4.z; wv[3] = t4.w;
        } else if constexpr (NW == 2) {
          const uint2 t2 = *reinterpret_cast<const uint2*>(w_step + u * (64 / SPS));
          wv[0] = t2.x; wv[1] = t2.y;
        } else {
          wv[0] = *reinterpret_cast<const uint32_t*>(w_step + u * (64 / SPS));
        }
        if (ok && i >= kARing) {
          // the MMAs of stage i - kARing are done: A operand i % kARing may be overwritten
          ok = mbar_wait(empty_bar + 8 * abuf, ((i / kARing) - 1) & 1);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) *fail_word = 1;
          tc_fence_after_sync();
        }
        if (!ok) continue;   // up to the next barrier, where all decoders leave
        // this thread's quarter of the stage's weights of its row -> columns kh * kCols / 4 ... of the A operand
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + abuf * G::kCols + kh * (G::kCols / 4);
        decode_to_tmem<BITS, NW>(wv, st, taddr);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar + 8 * abuf);
      }
    }
    // ---- wait until all MMAs of this CTA are done ----
    if (ok && total > 0) {
      const int last = total - 1;
      ok = mbar_wait(empty_bar + 8 * (last % kARing), (last / kARing) & 1);
      ok = __all_sync(0xFFFFFFFFu, ok);
    }
    if (!ok && lane == 0) atomicOr(&g_device_error_flags, 1u);
  } else if (warp == kDecodeWarps && lane == 0) {
    // ================= MMA warp (one thread) =================
    // The issuing thread is blocked for about 70 clocks per tcgen05.mma and runs everything in between serially, so
    // the per-instruction work is kept to one add: descriptors differ only in their low word.
    const uint32_t idesc = instr_desc<NB>();
    const uint64_t desc0 = smem_desc_sw128(b_addr);
    const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
    uint32_t desc_lo = (uint32_t)desc0, a_tmem = tmem_base, bar_off = 0;   // of the current stage's buffer
    int abuf = 0;
    uint32_t parity = 0;
    for (int i = 0; i < total; ++i) {
      if (!mbar_wait(full_bar + bar_off, parity)) {
        ok = false;
        break;
      }
      tc_fence_after_sync();
#pragma unroll
      for (int ks = 0; ks < G::kKSlices; ++ks) {   // 16 activations = 32 bytes further inside a 128-byte row
        const uint32_t lo = desc_lo + (ks >> 2) * (SM::kBHalfBytes >> 4) + (ks & 3) * 2;
        const uint64_t b_desc = ((uint64_t)desc_hi << 32) | lo;
        if (ks == 0) umma_bf16(tmem_d, a_tmem, b_desc, idesc, i != 0);
        else umma_bf16_acc(tmem_d, a_tmem + ks * 8, b_desc, idesc);
      }
      umma_commit(empty_bar + bar_off);
      if (++abuf == kARing) {
        abuf = 0;
        parity ^= 1;
        desc_lo = (uint32_t)desc0;
        a_tmem = tmem_base;
        bar_off = 0;
      } else {
        desc_lo += SM::kBStageBytes >> 4;
        a_tmem += G::kCols;
        bar_off += 8;
      }
    }
    if (!ok) atomicOr(&g_device_error_flags, 1u);
  } else if (warp == kDecodeWarps + 1 && lane == 0) {
    // ================= TMA producer (one thread) =================
    for (int j = 0; j < total; ++j) {
      const int buf = j % kARing;
      if (j >= kARing && !mbar_wait(empty_bar + 8 * buf, ((j / kARing) - 1) & 1)) {   // the MMAs that read the buffer
        ok = false;
        break;
      }
      mbar_expect_tx(full_bar + 8 * buf, SM::kBStageBytes);
      const int k0 = (s_begin * SPS + j) * G::kStageK;
      tma_load_2d(b_addr + buf * SM::kBStageBytes, &xmap, k0, (int)m0, full_bar + 8 * buf);
      tma_load_2d(b_addr + buf * SM::kBStageBytes + SM::kBHalfBytes, &xmap, k0 + 64, (int)m0, full_bar + 8 * buf);
    }
    if (!ok) atomicOr(&g_device_error_flags, 1u);
  }
  // ---- accumulators of the cluster -> rank 0 -> bf16 ----
  // Rank r > 0 hands its accumulator to rank 0 through rank 0's shared memory (the B buffers, free once every CTA of
  // the cluster has seen its last MMA complete): [r - 1][batch row][output row] floats.
  __syncwarp();
  if (ksplit > 1) cluster_sync();
  const bool reader = warp < kDecodeWarps && (warp >> 2) < kReaders && ok;   // the warps of a lane quarter split the columns
  if (reader) {
    const int q = warp & 3, kh = warp >> 2, rho = 32 * q + lane;
    tc_fence_after_sync();
    if (rank != 0) {
      const uint32_t remote = map_to_rank0(smem_base + SM::kB) + (uint32_t)(rank - 1) * (NB * kBM * 4);
      const int col0 = kh * kReadCols;
      uint32_t w[kReadCols];
      load_acc<kReadCols>(w, tmem_d + ((uint32_t)(q * 32) << 16) + col0, total > 0);
#pragma unroll
      for (int j = 0; j < kReadCols; ++j)
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(remote + ((col0 + j) * kBM + rho) * 4), "r"(w[j]) : "memory");
    }
  }
  __syncwarp();
  if (ksplit > 1) cluster_sync();
  if (reader && rank == 0) {
    const int q = warp & 3, kh = warp >> 2, rho = 32 * q + lane;
    const int64_t n = block_row0 + rho;
    const float* const partial = reinterpret_cast<const float*>(smem_raw + SM::kB);
    const int col0 = kh * kReadCols;
    uint32_t w[kReadCols];
    load_acc<kReadCols>(w, tmem_d + ((uint32_t)(q * 32) << 16) + col0, total > 0);
#pragma unroll
    for (int j = 0; j < kReadCols; ++j) {
      float v = __uint_as_float(w[j]);
      for (int r = 1; r < ksplit; ++r) v += partial[((r - 1) * NB + col0 + j) * kBM + rho];   // fixed order
      if (m0 + col0 + j < M && n < N) y[(m0 + col0 + j) * N + n] = (uint16_t)float_to_bf16_bits(v);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  // The tensor memory is given back on every path, also after a wait ran out: a CTA that left without freeing its
  // columns would block every later CTA on this SM in tcgen05.alloc for good.  A wait only runs out after 100 ms,
  // five orders of magnitude beyond the life of any instruction this kernel issues, so nothing of this CTA can
  // still be using the columns then.
  if (warp == kDecodeWarps)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)SM::kTmemCols)
                 : "memory");
}

}  // namespace

namespace {

template <int BITS, int NB>
cudaError_t launch_nb(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N, int64_t K,
                      int64_t M, int ksplit, cudaStream_t s) {
  // Every CTA takes all 512 tensor-memory columns with a blocking tcgen05.alloc and frees them only at its end, after
  // cluster barriers: two such CTAs on one SM (of one cluster or of two) could wait for each other for ever.  The
  // launch therefore asks for more than half of the SM's shared memory whatever the kernel needs, so that a second
  // CTA can never become resident on the same SM.
  const DeviceInfo* di = device_info();
  if (!di) return cudaErrorInvalidDevice;
  const int smem = umma_launch_smem(USmem<BITS, NB>::kTotal, di->max_smem_optin);
  if (smem > di->max_smem_optin || 2 * (smem + 1024) <= di->max_smem_optin + 1024) return cudaErrorInvalidConfiguration;
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    cudaError_t e = cudaFuncSetAttribute(linear_umma_kernel<BITS, NB>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  CUtensorMap xmap;
  if (!make_x_map(&xmap, x, K, M, NB)) return cudaErrorInvalidValue;
  const unsigned blocks = (unsigned)((N + kBM - 1) / kBM);
  if ((ksplit - 1) * NB * kBM * 4 > USmem<BITS, NB>::kBRing * USmem<BITS, NB>::kBStageBytes)
    return cudaErrorInvalidValue;   // the partial accumulators of the other CTAs must fit the B buffers
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, (unsigned)ksplit, (unsigned)((M + NB - 1) / NB));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = (unsigned)ksplit;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ksplit > 1 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, linear_umma_kernel<BITS, NB>, packed, cb, xmap, y, N, K, M);
}

template <int BITS>
cudaError_t launch_bits(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N,
                        int64_t K, int64_t M, int ksplit, cudaStream_t s) {
  if (M <= 16) return launch_nb<BITS, 16>(packed, cb, x, y, N, K, M, ksplit, s);
  if (M <= 32) return launch_nb<BITS, 32>(packed, cb, x, y, N, K, M, ksplit, s);
  if (M <= 48) return launch_nb<BITS, 48>(packed, cb, x, y, N, K, M, ksplit, s);
  if (M <= 64) return launch_nb<BITS, 64>(packed, cb, x, y, N, K, M, ksplit, s);
  if (M <= 96) return launch_nb<BITS, 96>(packed, cb, x, y, N, K, M, ksplit, s);
  return launch_nb<BITS, 128>(packed, cb, x, y, N, K, M, ksplit, s);
}

}  // namespace
}  // namespace kmq

#include "kmq_linear_umma_pair.cuh"

namespace kmq {

// Batch rows per launch (the grid's limits; in earnest one launch).
constexpr int64_t kSingleMaxRows = 128, kRowsPerLaunch = int64_t(1) << 20;
int64_t linear_umma_rows_per_launch() { return kRowsPerLaunch; }

// CTAs per 128-row block: K is split over a cluster of 2 or 4 (partial sums meet in CTA 0's shared memory) while the
// blocks alone would leave at least half (three quarters) of the SMs idle and each part still has a few steps.
// `batch` = rows of one launch; 4 CTAs only up to 64 rows (three partial accumulators must fit the B buffers).
int linear_umma_ksplit(int64_t N, int64_t K, int bits, int64_t batch) {
  const DeviceInfo* di = device_info();
  if (!di) return 1;
  const int64_t blocks = (N + kBM - 1) / kBM * ((batch + kSingleMaxRows - 1) / kSingleMaxRows);
  const int64_t steps = tuned_row_steps(K, bits);
  if (blocks * 4 <= di->sm_count && steps >= 32 && batch <= 64) return 4;   // measured: no gain with fewer than 8 steps per CTA
  return (blocks * 2 <= di->sm_count && steps >= 8) ? 2 : 1;
}

// The tensor core issues one tcgen05.mma (2048 weights) per 70-100 clocks whatever the batch, so the kernel's time
// does not depend on M up to 128 rows, but a CTA covers 128 output rows: it pays when the batch is large and there
// are enough 128-row blocks to occupy most SMs.  Measured: 16384 x 3072, b = 2: 18.5 us for any M <= 64 against
// 18.5 / 28.5 / 31.6 us of the multi-tile kernel at M = 32 / 40 / 64; 12288 x 4096, M = 64: 22.7 against 38.9 us;
// 8192 x 8192 (64 blocks), M = 64: 38.9 against 36.0 us.
bool linear_umma_selected(int64_t N, int64_t K, int bits, int64_t M) {
  const DeviceInfo* di = device_info();
  // b = 1: the multi-tile kernel has no 16-warp form beyond 16 rows (its x buffers are twice as large) and takes
  // 80 us at 8192 x 28672 for M = 17..32 against 60 us here
  if (!di || M <= (bits == 1 ? 16 : 32)) return false;
  if (!encode_tiled()) return false;   // no tensor-map encoder in this driver: stay on the mma.sync kernels
  if (M > kSingleMaxRows) return true;
  const int64_t ctas = (N + kBM - 1) / kBM * linear_umma_ksplit(N, K, bits, M);
  // with fewer CTAs it still wins where the multi-tile kernel is weakest: more than 48 rows, or b = 1 (which that
  // kernel serves 32 rows at a time): 4096 x 4096, 64 CTAs, M = 64: b = 2 18.4 against 20.7 us, b = 1 17.6 against 32.8 us
  const int64_t need = (M > 48 || bits == 1) ? (int64_t)di->sm_count * 3 / 8 : (int64_t)di->sm_count * 5 / 8;
  return ctas >= need;
}

// Whether more than 128 batch rows go to the CTA pairs.  Clocks, from in-kernel timelines and sweeps: a pair spends 136
// per 16 weights whatever its batch rows up to 256 (150 at b = 4), 3000 per tile and 8000 per launch besides; a single
// CTA (up to 128 rows) 115 (190) and 14000, or 24000 where K is split over a cluster, but there are twice as many of
// them.  The pairs win as soon as their 256 x 256 tiles fill the machine: 16384 x 3072, b = 2, M = 1024: 95 against
// 164 us; 4096 x 4096, M = 256 (16 tiles): 27 against 20 us.
static bool pair_pays(int64_t N, int64_t K, int bits, int64_t M) {
  const DeviceInfo* di = device_info();
  if (!di || M <= kSingleMaxRows) return false;
  const int64_t sms = di->sm_count, k16 = K / 16;
  const int64_t tiles = (N + 2 * kBM - 1) / (2 * kBM) * ((M + kPairMaxRows - 1) / kPairMaxRows);
  const int64_t rounds = (2 * tiles + sms - 1) / sms;
  const int64_t pair = 8000 + rounds * (3000 + k16 * (bits == 4 ? 150 : 136));
  const int64_t ks = linear_umma_ksplit(N, K, bits, M);
  const int64_t ctas = (N + kBM - 1) / kBM * ((M + kSingleMaxRows - 1) / kSingleMaxRows) * ks;
  const int64_t single = (ctas + sms - 1) / sms * ((ks > 1 ? 24000 : 14000) + k16 * (bits == 4 ? 190 : 115) / ks);
  return pair < single;
}

cudaError_t launch_linear_umma(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N,
                               int64_t K, int bits, int64_t M, cudaStream_t s) {
  for (int64_t m0 = 0; m0 < M; m0 += kRowsPerLaunch) {
    const int64_t mc = M - m0 < kRowsPerLaunch ? M - m0 : kRowsPerLaunch;
    const uint16_t* xp = x + m0 * K;
    uint16_t* yp = y + m0 * N;
    cudaError_t e;
    if (pair_pays(N, K, bits, mc)) {
      if (bits == 1) e = launch_umma_pair<1>(packed, cb, xp, yp, N, K, mc, s);
      else if (bits == 2) e = launch_umma_pair<2>(packed, cb, xp, yp, N, K, mc, s);
      else e = launch_umma_pair<4>(packed, cb, xp, yp, N, K, mc, s);
    } else {
      const int ks = linear_umma_ksplit(N, K, bits, mc);
      if (bits == 1) e = launch_bits<1>(packed, cb, xp, yp, N, K, mc, ks, s);
      else if (bits == 2) e = launch_bits<2>(packed, cb, xp, yp, N, K, mc, ks, s);
      else e = launch_bits<4>(packed, cb, xp, yp, N, K, mc, ks, s);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Reads and clears the device error word (synchronises the device).
cudaError_t read_device_error_flags(unsigned int* flags) {
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return e;
  e = cudaMemcpyFromSymbol(flags, g_device_error_flags, sizeof(unsigned int));
  if (e != cudaSuccess) return e;
  if (*flags) {
    const unsigned int zero = 0;
    e = cudaMemcpyToSymbol(g_device_error_flags, &zero, sizeof(unsigned int));
    if (e != cudaSuccess) return e;
  }
  unsigned int lut = 0;
  e = read_lut_error_flags(&lut);
  *flags |= lut;
  return e;
}


}  // namespace kmq
