// kmq_linear on the tuned layout for prefill batches (M > 128): tcgen05.mma over a pair of CTAs.  Included by
// kmq_linear_umma.cu, whose single-CTA kernel does the same for up to 128 batch rows; the roles of the warps are that kernel's.
// Here all 16 decoder warps rebuild every stage together, from packed words that a ring of cp.async copies brings to shared
// memory, with a barrier of theirs per step (up to 256 batch rows per decode: the tensor core is what the others wait for).
//
// What bounds it: one SM multiplies 128 x 256 x 16 in 128 clocks, and the 256 activations rows of that step are 8 KB, so
// a CTA on its own would draw 64 bytes per clock from L2, more than L2 gives 148 SMs at once; with 128 batch rows per
// CTA the tensor core is fed at half rate besides, because reading the 128-row A operand takes 64 clocks whatever the
// batch.  So two CTAs (two SMs, cta_group::2) share one 256 x 256 tile: each decodes 128 output rows into its own
// tensor memory (256 columns of A in a ring of 4 stages, 256 columns of accumulator) and brings half of the batch rows
// under a stage into its shared memory; the leader's MMA thread issues for both.  16384 x 3072, b = 2, M = 1024:
// 164 us as 8 passes of 128 rows.
//
// Meeting points, per stage of 128 weights: `full` of each CTA (its 16 decoder warps, its TMA bytes); the peer's relay
// thread passes its `full` on to the leader's `peer` barrier; the leader's MMA thread waits for both and commits to the
// `empty` barriers of both CTAs.  Per tile: `done` of each CTA (a commit behind the last stage) releases the eight
// epilogue warps, which read the accumulator; when those of both CTAs have it in registers (`drained`, at the leader) the
// MMA thread starts the next tile.
//
// The pairs are persistent: each takes every (number of pairs)-th tile, and everybody but the epilogue and the MMA thread
// runs on into the next tile, so that its first four stages wait in the rings while the accumulator is read.  One tile
// per cluster instead cost 8 us of start, fill and end against 16 us of multiplying (16384 x 3072, M = 256 and 1024:
// 24 and 105 us; now 24 and 96 us, 91 us at the clocks a colder card allows: the card's 1000 W bind, cuBLAS takes
// 86 us for the same product of bf16 matrices under the same cap).
#include <cuda_bf16.h>

namespace kmq {
namespace {

constexpr int kPairRing = 4;
constexpr int kPairMaxRows = 256;                         // batch rows of a tile
constexpr int kEpilogueWarps = 8;                         // 4 tensor-memory lane quarters x 2 halves of the batch rows
constexpr int kPairThreads = kThreads + kEpilogueWarps * 32;
constexpr int kEpilogueWarp0 = kDecodeWarps + 2;

template <int BITS>
struct PSmem {
  static constexpr int kBHalfBytes = (kPairMaxRows / 2) * 128;   // 128 batch rows x 64 activations
  static constexpr int kBStageBytes = 2 * kBHalfBytes;
  static constexpr int kB = 0;
  static constexpr int kWords = kB + kPairRing * kBStageBytes;
  static constexpr int kBars = kWords + kWRing * kWStepBytes;
  // full, empty, peer: [kPairRing] each; done, drained
  static constexpr int kTmemSlot = kBars + (3 * kPairRing + 2) * 8;   // then a word that a failed wait sets
  static constexpr int kTotal = kTmemSlot + 16 + 1024;
};

__device__ __forceinline__ void umma_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// arrives at the barrier of this offset in both CTAs of the pair
__device__ __forceinline__ void umma_pair_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_rank0(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(map_to_rank(bar, 0)) : "memory");
}

// 16 columns of this warp's lanes of the accumulator; the registers hold them after tmem_wait_load()
__device__ __forceinline__ void tmem_load16(uint32_t (&w)[16], uint32_t taddr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]),
        "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_load(uint32_t (&w)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7]),
                 "+r"(w[8]), "+r"(w[9]), "+r"(w[10]), "+r"(w[11]), "+r"(w[12]), "+r"(w[13]), "+r"(w[14]), "+r"(w[15])
               :
               : "memory");
}

template <int BITS>
__global__ void __launch_bounds__(kPairThreads, 1) linear_umma_pair_kernel(const uint32_t* __restrict__ packed,
                                                                           const uint16_t* __restrict__ cb,
                                                                           const __grid_constant__ CUtensorMap xmap,
                                                                           uint16_t* __restrict__ y, int64_t N,
                                                                           int64_t K, int64_t M, int NB) {
  using G = UGeo<BITS>;
  using SM = PSmem<BITS>;
  constexpr int SPS = G::kStagesPerStep;
  constexpr int NW = G::kThreadBytes / 4;   // packed words per thread and stage: 4, 2, 1
  extern __shared__ __align__(1024) unsigned char smem_unaligned[];
  unsigned char* const smem_raw =
      smem_unaligned + ((1024u - ((uint32_t)__cvta_generic_to_shared(smem_unaligned) & 1023u)) & 1023u);
  const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t b_addr = smem_base + SM::kB;
  const uint32_t full_bar = smem_base + SM::kBars, empty_bar = full_bar + 8 * kPairRing;
  const uint32_t peer_bar = empty_bar + 8 * kPairRing, done_bar = peer_bar + 8 * kPairRing, drained_bar = done_bar + 8;
  volatile uint32_t* const tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x & 1;                       // the pair = two neighbouring 128-row blocks
  const int steps = (int)tuned_row_steps(K, BITS);
  const int total = steps * SPS;                         // stages per tile
  // tile t: row pair t % pairs, batch tile t / pairs; this pair of CTAs takes tiles first, first + stride, ...
  const int64_t pairs = (N + 2 * kBM - 1) / (2 * kBM), tiles = pairs * ((M + NB - 1) / NB);
  const int64_t first = blockIdx.x >> 1, stride = gridDim.x >> 1;
  auto row_block = [&](int64_t t) { return 2 * (t % pairs) + rank; };   // this CTA's 128-row block of tile t

  // ---- set-up: mbarriers, tensor memory ----
  if (threadIdx.x == 0) {
    *reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot + 4) = 0;
    auto init = [](uint32_t bar, uint32_t count) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    };
#pragma unroll
    for (int i = 0; i < kPairRing; ++i) {
      init(full_bar + 8 * i, kDecodeWarps + 1);   // decoder warps + the producer's arrive-and-expect; TMA bytes besides
      init(empty_bar + 8 * i, 1);
      init(peer_bar + 8 * i, 1);
    }
    init(done_bar, 1);
    init(drained_bar, 2 * kEpilogueWarps);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kDecodeWarps) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_base + SM::kTmemSlot)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();          // the peer's barriers are set up before anything arrives there
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_d = tmem_base + kPairRing * G::kCols;   // the accumulator follows the A operands
  bool ok = true;

  if (warp < kDecodeWarps) {
    // ================= decoder warps, on from tile to tile =================
    const int q = warp & 3, kh = warp >> 2;
    const int rho = 32 * q + lane;
    const int64_t row_tiles = (N + kTileRows - 1) / kTileRows;
    const unsigned char* const w_row = smem_raw + SM::kWords + rho * kWRowStride + kh * G::kThreadBytes;
    const int cj = threadIdx.x;
    const uint32_t c_dst = smem_base + SM::kWords + (cj >> 2) * kWRowStride + (cj & 3) * 16;
    // the copies run kWRing - 1 steps ahead, into the next tile: step c_step of tile c_tile into slot c_slot
    int64_t c_tile = first;
    int c_step = 0, c_slot = 0;
    const unsigned char* c_src = nullptr;
    bool c_real = false;
    auto copy_step = [&]() {
      if (c_tile < tiles) {
        if (c_step == 0) {
          const int64_t t16 = row_block(c_tile) * (kBM / 16) + (cj >> 6);
          c_real = t16 < row_tiles;
          c_src = reinterpret_cast<const unsigned char*>(packed) + (c_real ? t16 : 0) * (int64_t)steps * 1024 +
                  (cj & 63) * 16;
        }
        cp_async16(c_dst + c_slot * kWStepBytes, c_src + (int64_t)c_step * 1024, c_real);
        if (++c_step == steps) {
          c_step = 0;
          c_tile += stride;
        }
        c_slot = c_slot + 1 == kWRing ? 0 : c_slot + 1;
      }
      cp_async_commit();
    };
    volatile uint32_t* const fail_word = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot + 4);
#pragma unroll 1
    for (int d = 0; d < kWRing - 1; ++d) copy_step();
    int slot = 0, abuf = 0;
    uint32_t parity = 1;   // of the wait for an empty stage: the first round finds all of them empty
    for (int64_t tile = first; tile < tiles && ok; tile += stride) {
      RowState<BITS> st;
      st.d.init(cb + min(row_block(tile) * kBM + rho, N - 1) * (1 << BITS));
      for (int s = 0; s < steps; ++s) {
        cp_async_wait<kWRing - 2>();   // this thread's piece of the step has landed
        // every decoder thread's piece has landed, and every one is done with the step before
        asm volatile("bar.sync 1, %0;" ::"n"(kDecodeThreads) : "memory");
        if (*fail_word) {   // some warp's wait ran out: all decoders leave together
          ok = false;
          break;
        }
        copy_step();                   // into the slot of the step before
        const unsigned char* const w_step = w_row + slot * kWStepBytes;
        slot = slot + 1 == kWRing ? 0 : slot + 1;
#pragma unroll
        for (int u = 0; u < SPS; ++u) {
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
          if (ok) {
            ok = mbar_wait(empty_bar + 8 * abuf, parity);
            ok = __all_sync(0xFFFFFFFFu, ok);
            if (!ok) *fail_word = 1;
            tc_fence_after_sync();
          }
          if (!ok) continue;   // up to the next barrier, where all decoders leave
          const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + abuf * G::kCols + kh * (G::kCols / 4);
          decode_to_tmem<BITS, NW>(wv, st, taddr);
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(full_bar + 8 * abuf);
          if (++abuf == kPairRing) {
            abuf = 0;
            parity ^= 1;
          }
        }
      }
    }
    if (!ok && lane == 0) atomicOr(&g_device_error_flags, 1u);
  } else if (warp == kDecodeWarps && lane == 0) {
    int buf = 0;
    uint32_t parity = 0, drained_parity = 1;
    if (rank == 0) {
      // ================= MMA thread of the pair =================
      // D fp32, A and B bf16, both K-major, M = 256, N = NB
      const uint32_t idesc =
          (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)((2 * kBM) >> 4) << 24);
      const uint64_t desc0 = smem_desc_sw128(b_addr);
      const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
      for (int64_t tile = first; tile < tiles && ok; tile += stride) {
        ok = mbar_wait_cluster(drained_bar, drained_parity);   // the accumulator of the tile before (none: passes)
        drained_parity ^= 1;
        for (int i = 0; i < total && ok; ++i) {
          ok = mbar_wait(full_bar + 8 * buf, parity) && mbar_wait_cluster(peer_bar + 8 * buf, parity);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t desc_lo = (uint32_t)desc0 + buf * (SM::kBStageBytes >> 4), a_tmem = tmem_base + buf * G::kCols;
#pragma unroll
          for (int ks = 0; ks < G::kKSlices; ++ks) {   // 16 activations = 32 bytes further inside a 128-byte row
            const uint32_t lo = desc_lo + (ks >> 2) * (SM::kBHalfBytes >> 4) + (ks & 3) * 2;
            umma_pair(tmem_d, a_tmem + ks * 8, ((uint64_t)desc_hi << 32) | lo, idesc, (i | ks) != 0);
          }
          umma_pair_commit(empty_bar + 8 * buf);
          if (++buf == kPairRing) {
            buf = 0;
            parity ^= 1;
          }
        }
        if (ok) umma_pair_commit(done_bar);
      }
    } else {
      // ================= relay: this CTA's part of a stage is in place =================
      for (int64_t tile = first; tile < tiles && ok; tile += stride) {
        for (int i = 0; i < total; ++i) {
          ok = mbar_wait(full_bar + 8 * buf, parity);
          if (!ok) break;
          tc_fence_after_sync();
          tc_fence_before_sync();
          mbar_arrive_rank0(peer_bar + 8 * buf);
          if (++buf == kPairRing) {
            buf = 0;
            parity ^= 1;
          }
        }
      }
    }
    if (!ok) atomicOr(&g_device_error_flags, 1u);
  } else if (warp == kDecodeWarps + 1 && lane == 0) {
    // ================= TMA producer: this CTA's half of a tile's batch rows =================
    const int rows = NB / 2;
    int buf = 0;
    uint32_t parity = 1;
    for (int64_t tile = first; tile < tiles && ok; tile += stride) {
      const int row0 = (int)(tile / pairs) * NB + rank * rows;
      for (int j = 0; j < total; ++j) {
        ok = mbar_wait(empty_bar + 8 * buf, parity);   // the MMAs that read the buffer
        if (!ok) break;
        mbar_expect_tx(full_bar + 8 * buf, rows * 256);
        const int k0 = j * G::kStageK;
        tma_load_2d(b_addr + buf * SM::kBStageBytes, &xmap, k0, row0, full_bar + 8 * buf);
        tma_load_2d(b_addr + buf * SM::kBStageBytes + SM::kBHalfBytes, &xmap, k0 + 64, row0, full_bar + 8 * buf);
        if (++buf == kPairRing) {
          buf = 0;
          parity ^= 1;
        }
      }
    }
    if (!ok) atomicOr(&g_device_error_flags, 1u);
  } else if (warp >= kEpilogueWarp0) {
    // ================= epilogue: accumulator -> bf16 =================
    // A warp reads the lane quarter that its index allows and half of the batch rows, 16 at a time.
    const int q = warp & 3, c0 = ((warp - kEpilogueWarp0) >> 2) * (NB / 2), c1 = c0 + NB / 2;
    uint32_t parity = 0;
    // a whole tile may be under way: 100 ms and 10 us for every stage of it
    const uint64_t limit = kWaitLimitNs + (uint64_t)total * 10000u;
    for (int64_t tile = first; tile < tiles; tile += stride) {
      ok = mbar_wait(done_bar, parity, limit);
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (!ok) break;
      parity ^= 1;
      tc_fence_after_sync();
      const int64_t n = row_block(tile) * kBM + 32 * q + lane, m0 = tile / pairs * NB;
      const uint32_t taddr = tmem_d + ((uint32_t)(q * 32) << 16);
      const int rows = n < N ? (int)(M - m0 < NB ? M - m0 : NB) : 0;   // columns of this lane that are stored
      uint16_t* out = y + (m0 + c0) * N + n;
      uint32_t w[16];
      tmem_load16(w, taddr + c0);
      for (int c = c0; c < c1; c += 16) {
        tmem_wait_load(w);
        uint32_t p[8];                 // bf16 pairs of columns c + 2 j, c + 2 j + 1
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const __nv_bfloat162 v =
              __floats2bfloat162_rn(__uint_as_float(w[2 * j]), __uint_as_float(w[2 * j + 1]));
          p[j] = *reinterpret_cast<const uint32_t*>(&v);
        }
        if (c + 16 < c1) {
          tmem_load16(w, taddr + c + 16);   // under way while these are stored
        } else {                       // all of this warp's part is in registers: the accumulator may be overwritten
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_rank0(drained_bar);
        }
        if (c + 16 <= rows) {
#pragma unroll
          for (int j = 0; j < 16; ++j, out += N) *out = (uint16_t)(j & 1 ? p[j >> 1] >> 16 : p[j >> 1]);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j, out += N)
            if (c + j < rows) *out = (uint16_t)(j & 1 ? p[j >> 1] >> 16 : p[j >> 1]);
        }
      }
    }
    if (!ok && lane == 0) atomicOr(&g_device_error_flags, 1u);
  }
  __syncwarp();
  tc_fence_before_sync();
  __syncthreads();
  cluster_sync();          // neither CTA gives its tensor memory back, or leaves, while the other still uses the pair's
  if (warp == kDecodeWarps)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
}

// Batch rows per tile: the fewest tiles of at most 256 rows (an MMA takes 136 clocks for any number of them, measured at
// 64, 160 and 256), evenly filled, in steps of 32.
inline int pair_tile_rows(int64_t M) {
  const int64_t t = (M + kPairMaxRows - 1) / kPairMaxRows;
  return (int)((M + 32 * t - 1) / (32 * t)) * 32;
}

template <int BITS>
cudaError_t launch_umma_pair(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N,
                             int64_t K, int64_t M, cudaStream_t s) {
  const DeviceInfo* di = device_info();
  if (!di) return cudaErrorInvalidDevice;
  constexpr int smem = PSmem<BITS>::kTotal;   // more than half of an SM's: the CTAs take all of its tensor memory
  if (smem > di->max_smem_optin || 2 * (smem + 1024) <= di->max_smem_optin + 1024) return cudaErrorInvalidConfiguration;
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {
    cudaError_t e =
        cudaFuncSetAttribute(linear_umma_pair_kernel<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  const int64_t slots = di->sm_count / 2 > 0 ? di->sm_count / 2 : 1;
  const int nb = pair_tile_rows(M);
  const int64_t tiles = (N + 2 * kBM - 1) / (2 * kBM) * ((M + nb - 1) / nb);
  CUtensorMap xmap;
  if (!make_x_map(&xmap, x, K, M, nb / 2)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * (tiles < slots ? tiles : slots)));
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, linear_umma_pair_kernel<BITS>, packed, cb, xmap, y, N, K, M, nb);
}

}  // namespace
}  // namespace kmq
