// kmq_linear on the tuned (tile-major) layout for large batches: the 5th-generation tensor core (tcgen05.mma)
// multiplies dequantised bf16 weights, held in tensor memory, with the activations in shared memory; the accumulator
// lives in tensor memory too.
//
// One CTA owns 128 output rows (8 tiles of 16) and walks its share of K in stages of 128 weights per row.  Its 16
// decoder warps, one MMA warp and one TMA producer warp meet only through mbarriers:
//   * the decoder warps are 4 groups of 4; group j rebuilds stages j, j + 4, ... on its own, so that four stages are in
//     flight and no barrier of the CTA stands in the loop.  Thread (warp w, lane l) owns output row 32 (w % 4) + l -- the
//     tensor-memory lane a warp may write is fixed by its index.  It loads the row's 64, 32 or 16 bytes of a stage
//     straight into registers (a few stages ahead; a lane's bytes are whole 32-byte sectors at b = 4, 2), rebuilds the 128
//     weights as bf16 pairs and writes them with tcgen05.st into the A operand of the stage (lane = row, 32-bit column
//     c = weights 2c, 2c + 1 of the stage; ring of kRing stages), then arrives on the slot's `full` barrier;
//   * the producer thread copies the activations under a stage (NB batch rows x 128, zero-filled past M and past K)
//     with two TMA tile loads (cp.async.bulk.tensor, 64 columns = 128 bytes wide, 128-byte swizzle) into a ring of B
//     buffers with barriers of its own;
//   * the MMA thread waits for both, issues 8 tcgen05.mma (128 x NB x 16 each) that add into the accumulators
//     D[128 output rows][NB batch rows], and commits them to the slots' `empty` barriers, which the decoders and the
//     producer wait for before they overwrite the A operand and the B buffer.
// A tcgen05.mma cuts its sum off instead of rounding it, so the error of a result grows with the number of MMAs that add into
// one accumulator.  The slices of K therefore take turns on 2 to 8 accumulators (kAccs), which the epilogue adds: what fits
// tensor memory beside enough A operands.  Share of results that are not the rounded exact ones, one accumulator / now
// (mma.sync with its four or more chains, for comparison): 8192 x 28672, b = 4, M = 16 0.0080 / 0.0012 (0.0031); 12288 x 8192,
// b = 4, M = 24 0.0042 / 0.0011 (0.0014); 4096 x 4096, b = 2, M = 40 0.00056 / 0.00030 (0.00037); 4096 x 2048, b = 2,
// M = 128 0.00065 / 0.00032 (0.00039).  It costs up to 3 % up to 64 batch rows (8192 x 28672, b = 1, M = 16 28.15 -> 28.28 us;
// 14000 x 1024, b = 4, M = 16 4.63 -> 4.78), 4 % up to 96 and up to 6 % with 128 (8192 x 28672, b = 1, M = 128 44.5 -> 46.1,
// 4096 x 1024, b = 4 6.5 -> 6.9), where it leaves 4 stages in flight instead of 5.
// b = 4, up to 64 batch rows: a row's 256 (centroid, centroid) pairs sit in shared memory, one bank per row, so that two
// weights cost one PRMT and one conflict-free load (in registers: 5 integer instructions).  A tcgen05.mma of up to 64
// batch rows takes 45 clocks, its 2048 weights 32 clocks of the load port, 16 of the integer pipe.
// When the 128-row blocks alone would leave SMs idle, K is split over a cluster of CTAs: each accumulates its share and
// hands its sums over through the owners' shared memory (st.shared::cluster), every CTA adds those of its share of the
// batch rows in a fixed order.  At the end the decoder warps read the accumulator with tcgen05.ld (lane = output row,
// column = batch row), round to bf16 and store.
//
// Every wait on an mbarrier is bounded; a warp whose wait runs out sets bit 0 of the device error word and goes to
// the end of the kernel (so does, after its own bounded waits, every warp that depended on it); every thread still
// takes part in the cluster barriers and the final CTA barrier, after which the tensor memory is freed.  Under
// programmatic dependent launch packed words and codebooks are read ahead of the previous kernel's end; no bounded wait
// that depends on the activations starts before it.
#include <algorithm>
#include <atomic>

#include "kmq_umma_common.cuh"

namespace kmq {

using namespace umma;

__device__ unsigned int g_device_error_flags = 0;   // sticky; read and cleared by kmq_device_error_flags()

namespace {

constexpr int kGroups = kDecodeWarps / 4;
constexpr int kMaxSplit = 8;                             // CTAs of a cluster
// Columns of sums that a CTA of a cluster of any size takes in at most: its share of the NB, from every CTA.
constexpr int exchange_columns(int nb) {
  int most = 0;
  for (int ks = 2; ks <= kMaxSplit; ++ks) most = most > ks * ((nb + ks - 1) / ks) ? most : ks * ((nb + ks - 1) / ks);
  return most;
}

template <int BITS, int NB>
struct USmem {
  static constexpr bool kTab = BITS == 4 && NB <= 64;               // pair tables in shared memory
  static constexpr int kAccs = NB <= 16 ? 8 : NB <= 32 ? 4 : 2;     // accumulators of NB columns ...
  static constexpr int kAccStride = NB == 48 ? 64 : NB;             // ... that many columns apart
  // stages in flight: A operands in tensor memory beside the accumulators (and so B buffers in shared memory)
  static constexpr int kRing = NB <= 64 ? 6 : NB <= 96 ? 5 : 4;
  static constexpr int kTmemCols = 512;
  static_assert(kRing * 64 + kAccs * kAccStride <= 512, "tensor memory has 512 columns");
  static_assert(UGeo<BITS>::kKSlices % kAccs == 0, "every stage adds to all accumulators");
  static_assert(kRing >= kGroups, "a slot belongs to one group at a time");
  static constexpr int kBHalfBytes = NB * 128;                      // NB rows x 64 activations (one TMA box)
  static constexpr int kBStageBytes = 2 * kBHalfBytes;
  static constexpr int kB = 0;
  static constexpr int kTables = kB + kRing * kBStageBytes;         // 4 quarters of 32 rows, see `bank`
  static constexpr int kBars = kTables + (kTab ? 2 * 65536 : 0);    // full[kRing], empty[kRing], done
  static constexpr int kTmemSlot = kBars + (2 * kRing + 2) * 8;
  // Sums that the CTAs of a cluster hand over, columns of 128 floats.  Where they do not fit beside the rest they lie over
  // the B buffers; with 128 batch rows too, where that is faster (1024 x 3072, b = 1, M = 128 8.1 us, beside the rest 8.6).
  static constexpr int kExchangeBytes = exchange_columns(NB) * kBM * 4;
  static constexpr bool kOwnExchange = NB <= 96 && kTmemSlot + 16 + kExchangeBytes + 1024 <= 227 * 1024;
  static constexpr int kExchange = kOwnExchange ? kTmemSlot + 16 : kB;
  static_assert(kOwnExchange || kExchangeBytes <= kBars, "the exchange lies over buffers that are free by then");
  static constexpr int kTotal = kTmemSlot + 16 + (kOwnExchange ? kExchangeBytes : 0) + 1024;   // + room to align the base
};

// Instruction descriptor of kind::f16: D fp32, A and B bf16, both K-major, M = kBM, N = NB.
template <int NB>
__device__ __forceinline__ uint32_t instr_desc() {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NB >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);
}

// Packed words of a row in a stage: 64, 32, 16 bytes for b = 4, 2, 1.  32 bytes at a time where the array is aligned to
// that (`wide`): a lane's load is then a whole sector.
template <int NW>
__device__ __forceinline__ void load_words(uint32_t (&w)[NW], const unsigned char* p, bool wide) {
  if constexpr (NW >= 8) {
    if (wide) {
#pragma unroll
      for (int i = 0; i < NW; i += 8)
        asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(w[i]), "=r"(w[i + 1]), "=r"(w[i + 2]), "=r"(w[i + 3]), "=r"(w[i + 4]), "=r"(w[i + 5]),
                       "=r"(w[i + 6]), "=r"(w[i + 7])
                     : "l"(p + 4 * i));
      return;
    }
  }
#pragma unroll
  for (int i = 0; i < NW; i += 4) {
    const uint4 v = __ldg(reinterpret_cast<const uint4*>(p + 4 * i));
    w[i] = v.x;
    w[i + 1] = v.y;
    w[i + 2] = v.z;
    w[i + 3] = v.w;
  }
}
__device__ __forceinline__ void tmem_store16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(
          taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
// The loads of w are waited for here.
template <int NW>
__device__ __forceinline__ void arrived(uint32_t (&w)[NW]) {
#pragma unroll
  for (int i = 0; i < NW; i += 4) asm volatile("" : "+r"(w[i]), "+r"(w[i + 1]), "+r"(w[i + 2]), "+r"(w[i + 3]));
}
// Word(s) number `c` of a stage -> 32 weights as bf16 pairs in the order of k.  `bank`: this lane's place in the pair
// tables, byte 1 open for an index byte.
template <int BITS, int NW, bool TAB>
__device__ __forceinline__ void decode32(uint32_t (&a)[16], const uint32_t (&w)[NW], int c, const RowState<BITS>& st,
                                         const unsigned char* tables, uint32_t bank) {
  if constexpr (BITS == 4 && TAB) {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t at = prmt(w[4 * c + (i >> 2)], bank, 0x7604u | ((i & 3) << 4));
      a[i] = *reinterpret_cast<const uint32_t*>(tables + at);
    }
  } else if constexpr (BITS == 4) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t v[4];
      st.d.word(w[4 * c + j], v);
#pragma unroll
      for (int i = 0; i < 4; ++i) a[4 * j + i] = v[i];
    }
  } else if constexpr (BITS == 2) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) st.d.pair(w[2 * c + j], q, a[8 * j + 2 * q], a[8 * j + 2 * q + 1]);
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = st.d.select(w[c] * kPow2[i]);
  }
}

template <int BITS, int NB>
__global__ void __launch_bounds__(kThreads, 1) linear_umma_kernel(const uint32_t* __restrict__ packed,
                                                                  const uint16_t* __restrict__ cb,
                                                                  const __grid_constant__ CUtensorMap xmap,
                                                                  uint16_t* __restrict__ y, int64_t N, int64_t K,
                                                                  int64_t M) {
  using G = UGeo<BITS>;
  using SM = USmem<BITS, NB>;
  constexpr int NW = 4 * BITS;              // packed words of a row in a stage
  constexpr int kAhead = 32 / NW;           // stages of a group whose words are in registers or on their way there
  constexpr int kRing = SM::kRing;
  extern __shared__ __align__(1024) unsigned char smem_unaligned[];
  unsigned char* const smem_raw =
      smem_unaligned + ((1024u - ((uint32_t)__cvta_generic_to_shared(smem_unaligned) & 1023u)) & 1023u);
  const uint32_t smem_base = (uint32_t)__cvta_generic_to_shared(smem_raw);
  const uint32_t b_addr = smem_base + SM::kB;
  const uint32_t full_bar = smem_base + SM::kBars, empty_bar = full_bar + 8 * kRing, done_bar = empty_bar + 8 * kRing;
  volatile uint32_t* const tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::kTmemSlot);

  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform for the compiler
  const int64_t block_row0 = (int64_t)blockIdx.x * kBM;
  const int64_t m0 = (int64_t)blockIdx.z * NB;   // first batch row of this CTA's tile
  // K is split over the gridDim.y CTAs of a cluster (same output rows): rank r takes stages [begin, begin + total)
  const int ksplit = gridDim.y, rank = blockIdx.y;
  const int stages = (int)((K + G::kStageK - 1) / G::kStageK);
  const int begin = (int)((int64_t)stages * rank / ksplit), total = (int)((int64_t)stages * (rank + 1) / ksplit) - begin;

  // ---- decoder threads: the first packed words and the row's codebook are on their way before anything else ----
  const int q = warp & 3, group = warp >> 2;   // tensor-memory lane quarter; which stages
  const int rho = 32 * q + lane;               // output row inside the CTA = tensor-memory lane
  const bool wide = (reinterpret_cast<uintptr_t>(packed) & 31) == 0;
  const unsigned char* w_src = nullptr;
  uint32_t words[kAhead][NW];
  RowState<BITS> st;
  auto load_stage = [&](uint32_t (&w)[NW], int i) {   // a row's stages lie in steps of 64 bytes, 1 KB apart
    const int k = begin + i;
    load_words<NW>(w, w_src + (int64_t)(k / G::kStagesPerStep) * 1024 + (k % G::kStagesPerStep) * (4 * NW), wide);
  };
  if (warp < kDecodeWarps) {
    // rows past N read the last row of the last tile (their results are never stored)
    const int64_t n = min(block_row0 + rho, N - 1);
    w_src = reinterpret_cast<const unsigned char*>(packed) + (n >> 4) * tuned_row_steps(K, BITS) * 1024 + (n & 15) * 64;
#pragma unroll
    for (int p = 0; p < kAhead; ++p)
      if (group + p * kGroups < total) load_stage(words[p], group + p * kGroups);
    if constexpr (!SM::kTab) st.d.init(cb + n * (1 << BITS));
  }

  // ---- set-up: mbarriers, tensor memory, tables ----
  if (threadIdx.x == kDecodeThreads + 32) {
#pragma unroll
    for (int i = 0; i < kRing; ++i) {
      // a group's warps + the producer's arrive-and-expect; the TMA bytes complete the same phase
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(full_bar + 8 * i), "r"(4 + 1) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(empty_bar + 8 * i) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(done_bar), "r"(1) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kDecodeWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_base + SM::kTmemSlot),
                 "r"((uint32_t)SM::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  bool ok = true;
  unsigned char* const tables = smem_raw + SM::kTables;
  uint32_t bank = 0;
  if constexpr (SM::kTab) {
    // entry e of the 32 rows of quarter q at (q / 2) * 64 KB + e * 256 + (q % 2) * 128 + 4 * lane
    bank = (q >> 1) * 65536 + (q & 1) * 128 + lane * 4;
    if (warp < kDecodeWarps) {
      // group j builds the entries whose second index is 4 j .. 4 j + 3
      const uint16_t* const crow = cb + min(block_row0 + rho, N - 1) * 16;
      const uint4 c0 = __ldg(reinterpret_cast<const uint4*>(crow)), c1 = __ldg(reinterpret_cast<const uint4*>(crow) + 1);
      const uint2 second = __ldg(reinterpret_cast<const uint2*>(crow) + group);
      const uint32_t first[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
      for (int hi = 0; hi < 4; ++hi) {
        const uint32_t s = hi < 2 ? second.x : second.y;
#pragma unroll
        for (int lo = 0; lo < 16; ++lo) {
          const uint32_t v = prmt(first[lo >> 1], s, ((hi & 1) ? 0x7600u : 0x5400u) | ((lo & 1) ? 0x32u : 0x10u));
          *reinterpret_cast<uint32_t*>(tables + bank + ((4 * group + hi) * 16 + lo) * 256) = v;
        }
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t tmem_d = tmem_base + kRing * G::kCols;   // the accumulators follow the A operands
  asm volatile("griddepcontrol.launch_dependents;");
  if (SM::kOwnExchange && ksplit > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

  if (warp < kDecodeWarps) {
    // ================= decoder warps =================
    int slot = group, round = 0;   // slot of the ring, how often the group's stages have gone round it
    for (int i0 = group; i0 < total && ok; i0 += kAhead * kGroups) {
#pragma unroll
      for (int p = 0; p < kAhead; ++p) {
        const int i = i0 + p * kGroups;
        if (i >= total) break;
        if (round > 0) {
          // The MMAs of stage i - kRing are done: the slot may be overwritten.  (A wait by parity needs the phase before
          // to be complete: that of stage i - 2 kRing, and this group has waited for stage i - 4 - kRing, no earlier one.)
          asm volatile("griddepcontrol.wait;" ::: "memory");
          ok = mbar_wait(empty_bar + 8 * slot, (round - 1) & 1);
          ok = __all_sync(0xFFFFFFFFu, ok);
          if (!ok) break;
          tc_fence_after_sync();
        }
        // The words of the stage before are loaded anew only now that this stage's have arrived: a wait for registers of a load
        // is a wait for later loads too, where they share one of a warp's few counters, and behind the stage's decode each
        // round ended with the latency of the load just issued.  us in a graph, before / now: 8192 x 28672, M = 16, b = 4 29.6 / 28.3,
        // b = 2 32.2 / 30.5; at b = 1, with eight loads of one word each in flight, it gained nothing (28.4 as before).
        if constexpr (BITS >= 2) {
          arrived<NW>(words[p]);
          if (i != group && i + (kAhead - 1) * kGroups < total)
            load_stage(words[(p + kAhead - 1) % kAhead], i + (kAhead - 1) * kGroups);
        }
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + slot * G::kCols;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t a[16];
          decode32<BITS, NW, SM::kTab>(a, words[p], c, st, tables, bank);
          tmem_store16(taddr + 16 * c, a);
        }
        if constexpr (BITS == 1)
          if (i + kAhead * kGroups < total) load_stage(words[p], i + kAhead * kGroups);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar + 8 * slot);
        slot += kGroups;
        if (slot >= kRing) {
          slot -= kRing;
          ++round;
        }
      }
    }
    // ---- wait until all MMAs of this CTA are done ----
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ok && total > 0) {
      ok = mbar_wait(done_bar, 0);
      ok = __all_sync(0xFFFFFFFFu, ok);
    }
    if (!ok && lane == 0) atomicOr(&g_device_error_flags, 1u);
  } else if (warp == kDecodeWarps) {
    // ================= MMA warp =================
    // The whole warp runs the loop and one elected lane issues: descriptors and addresses are then warp-uniform for the
    // compiler, and a tcgen05.mma of 16 batch rows goes out every 10 clocks (26 with a stage's wait and commit).  With
    // the loop inside a branch on the lane number each took 45 (72) clocks, more than the decoders need.
    asm volatile("griddepcontrol.wait;" ::: "memory");   // what follows waits for activations
    const uint32_t idesc = instr_desc<NB>();
    const uint64_t desc0 = smem_desc_sw128(b_addr);
    const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
    uint32_t slot = 0, parity = 0;
    for (int i = 0; i < total; ++i) {
      ok = __all_sync(0xFFFFFFFFu, mbar_wait(full_bar + 8 * slot, parity));   // the warp goes on, or gives up, as one
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t desc_lo = (uint32_t)desc0 + slot * (SM::kBStageBytes >> 4), a_tmem = tmem_base + slot * G::kCols;
#pragma unroll
      for (int ks = 0; ks < G::kKSlices; ++ks) {   // 16 activations = 32 bytes further inside a 128-byte row
        const uint32_t lo = desc_lo + (ks >> 2) * (SM::kBHalfBytes >> 4) + (ks & 3) * 2;
        umma_bf16_elect(tmem_d + ks % SM::kAccs * SM::kAccStride, a_tmem + ks * 8, ((uint64_t)desc_hi << 32) | lo, idesc,
                        ks >= SM::kAccs || i > 0);
      }
      umma_commit_elect(empty_bar + 8 * slot);
      if (++slot == kRing) {
        slot = 0;
        parity ^= 1;
      }
    }
    if (ok) umma_commit_elect(done_bar);
    else if (lane == 0) atomicOr(&g_device_error_flags, 1u);
  } else {
    // ================= TMA producer warp =================
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the activations may come from the previous kernel
    uint32_t slot = 0, parity = 1;
    for (int j = 0; j < total; ++j) {
      if (j >= kRing) {   // the MMAs that read the buffer
        ok = __all_sync(0xFFFFFFFFu, mbar_wait(empty_bar + 8 * slot, parity));
        if (!ok) break;
      }
      const uint32_t bar = full_bar + 8 * slot, dst = b_addr + slot * SM::kBStageBytes;
      const int k0 = (begin + j) * G::kStageK;
      tma_load_pair_elect(dst, dst + SM::kBHalfBytes, SM::kBStageBytes, &xmap, k0, k0 + 64, (int)m0, bar);
      if (++slot == kRing) {
        slot = 0;
        parity ^= 1;
      }
    }
    if (!ok && lane == 0) atomicOr(&g_device_error_flags, 1u);
  }
  // ---- accumulators of the cluster -> their columns' owners -> bf16 ----
  // This code runs once a launch and mostly waits for its own instructions: the loops stay rolled up (unrolled over 32
  // columns it took 15 us for 128 batch rows).
  __syncwarp();
  if (ksplit > 1) {
    if constexpr (SM::kOwnExchange) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // all have started
    else cluster_sync();                                     // all are done with the buffers below the exchange
  }
  // CTA r of the cluster owns `share` batch rows: every CTA writes its sums of them into r's shared memory ([CTA][batch row of
  // the share][output row] floats), and r adds them in the order of the ranks.
  const int share = (NB + ksplit - 1) / ksplit;
  if (warp < kDecodeWarps && ok) {
    tc_fence_after_sync();
    const int64_t n = block_row0 + rho;
#pragma unroll 1
    for (int c = 8 * group; c < NB; c += 8 * kGroups) {
      uint32_t w[8];
      load_acc<SM::kAccs>(w, tmem_d + ((uint32_t)(q * 32) << 16) + c, SM::kAccStride, total > 0);
      if (ksplit > 1) {
        int owner = c / share, mine = c % share;
        const uint32_t here = smem_base + SM::kExchange + (rank * share * kBM + rho) * 4;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(map_to_rank(here + mine * (kBM * 4), owner)), "r"(w[j]) : "memory");
          if (++mine == share) {
            mine = 0;
            ++owner;
          }
        }
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (m0 + c + j < M && n < N) y[(m0 + c + j) * N + n] = (uint16_t)float_to_bf16_bits(__uint_as_float(w[j]));
      }
    }
  }
  __syncwarp();
  if (ksplit > 1) {
    cluster_sync();
    if (warp < kDecodeWarps && ok) {
      const float* sums = reinterpret_cast<const float*>(smem_raw + SM::kExchange) + rho;
      const int64_t n = block_row0 + rho;
#pragma unroll 1
      for (int c = group; c < share; c += kGroups) {
        const int64_t m = m0 + rank * share + c;
        if (rank * share + c >= NB || m >= M || n >= N) break;
        float v = sums[c * kBM];
#pragma unroll 1
        for (int r = 1; r < ksplit; ++r) v += sums[(r * share + c) * kBM];   // fixed order
        y[m * N + n] = (uint16_t)float_to_bf16_bits(v);
      }
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
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, (unsigned)ksplit, (unsigned)((M + NB - 1) / NB));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = (unsigned)ksplit;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = ksplit > 1 ? 2 : 1;
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

// Clusters of `size` CTAs of this kernel (one per SM) that fit the device at once: a cluster lies within one group of SMs,
// so that fewer than sm_count / size may.  Asked for once per device and size.
static int resident_clusters(int size) {
  static std::atomic<int> known[64][kMaxSplit + 1] = {};   // + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || size < 2 || size > kMaxSplit) return 0;
  int n = known[dev][size].load(std::memory_order_relaxed);
  if (n == 0) {
    const DeviceInfo* di = device_info();
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1, (unsigned)size, 1);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = umma_launch_smem(USmem<1, 16>::kTotal, di ? di->max_smem_optin : 0);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = (unsigned)size;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (!di ||
        cudaFuncSetAttribute(linear_umma_kernel<1, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, linear_umma_kernel<1, 16>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    known[dev][size].store(++n, std::memory_order_relaxed);
  }
  return n - 1;
}

// Time of a call of the single-CTA kernel with K split over clusters of ks CTAs, in ns: a model fitted to 3000 calls (N 128 to
// 18000, K 256 to 28672, M 16 to 1024; 12 % standard deviation, which the choices below can bear: they are 1 % from the
// best of what was measured).  A stage of a CTA, start and end of every wave of CTAs, the cluster's exchange, and what
// CTAs beyond 40 cost at the start (shared paths to L2; fewer of the next call's can set up beside them).
static int64_t single_ns(int64_t blocks, int64_t stages, int64_t nb, int bits, int ks, int64_t sms) {
  const int64_t ctas = blocks * ks, waves = (ctas + sms - 1) / sms;
  const int64_t stage = 156 + nb * 6 / 5 + (bits == 4 && nb > 64 ? 110 : 0);
  const int64_t exchange = ks > 1 ? (900 + 100 * ks + (ks > 6 ? 500 : 0)) * (64 + nb) / 80 : 0;
  return waves * ((stages + ks - 1) / ks * stage + 3900) + exchange + 20 * std::max<int64_t>(0, std::min(ctas, sms) - 40);
}

// CTAs per 128-row block: K split over a cluster of up to 8.  Measured, b = 4, M = 16, us per call with 1 / 2 / 3 / 4 / 5 / 6 /
// 8 CTAs: 1024 x 3072 6.2 / 4.5 / 4.0 / 3.7 / 3.6 / 3.6 / 4.2, 3072 x 3072 6.4 / 4.8 / 5.1 / 5.1 / 5.5 / 8.2 / - (6 x 24: more
// clusters than fit), 3072 x 8192 15.7 / 9.3 / 8.3 / 7.7 / 7.8, 8192 x 3072 7.0 / 7.3; M = 128, 1024 x 3072 13.0 / 10.6 / 8.7 /
// 8.3 / 8.0 / 7.9 / 8.0.
static int best_split(int64_t N, int64_t K, int bits, int64_t batch, int64_t* ns) {
  const DeviceInfo* di = device_info();
  *ns = 0;
  if (!di) return 1;
  const int64_t sms = di->sm_count, tiles = (batch + kSingleMaxRows - 1) / kSingleMaxRows;
  const int64_t blocks = (N + kBM - 1) / kBM * tiles, stages = (K + UGeo<4>::kStageK - 1) / UGeo<4>::kStageK;
  const int64_t nb = (std::min(batch, kSingleMaxRows) + 15) / 16 * 16;
  int best = 1;
  *ns = single_ns(blocks, stages, nb, bits, 1, sms);
  for (int ks = 2; ks <= kMaxSplit; ++ks) {
    if (blocks * ks > sms || stages < 3 * ks || blocks > resident_clusters(ks)) continue;
    const int64_t t = single_ns(blocks, stages, nb, bits, ks, sms);
    if (t < *ns) {
      *ns = t;
      best = ks;
    }
  }
  return best;
}
int linear_umma_ksplit(int64_t N, int64_t K, int bits, int64_t batch) {
  int64_t ns;
  return best_split(N, K, bits, batch, &ns);
}

// Which calls come here (tuned layout): from 9 batch rows on, unless rows are short and the 128-row blocks few.  Lines from
// sweeps of this and the multi-tile kernel over 1200 shapes (100 to 20000 rows of 256 to 28672 weights) at 9 to 64 batch
// rows; us per call, multi-tile / this:
//   9 to 16   rows from K = 2048 (b = 4: 1536) on: 3072 x 3072, M = 16, b = 2 5.1 / 4.7, b = 4 6.9 / 4.8, 8192 x 28672, b = 4
//             51.4 / 31.5.  Shorter ones with many of them: from 4096 (b = 4: from K = 1024 on; else 9472) on: 12288 x 1024,
//             b = 4 7.3 / 5.0, but 4096 x 512 4.0 / 4.3.  At b = 1 also up to K = 512, where both are one start of a CTA
//             (1227 x 256 2.9 / 2.4; 1024 x 1024 10 % slower here).
//             Not at b = 1 with half to three quarters as many blocks as SMs, which no cluster fills up, from K = 8192 on
//             (9600 x 16384, M = 16 17 % slower than the balanced form of the multi-tile kernel).
//   17 to 32  b = 1 always (512 x 1024, M = 20 14 % faster); b = 2, 4 from K = 1536 or 4096 rows on (512 x 1024, b = 4 4 % slower)
//   33 on     always
bool linear_umma_selected(int64_t N, int64_t K, int bits, int64_t M) {
  const DeviceInfo* di = device_info();
  if (!di || M <= 8) return false;
  if (!encode_tiled()) return false;   // no tensor-map encoder in this driver: stay on the mma.sync kernels
  if (M > 32) return true;
  if (M > 16) return bits == 1 || K >= 1536 || N >= 4096;
  const int64_t blocks = (N + kBM - 1) / kBM;
  if (bits == 1 && K >= 8192 && 2 * blocks > di->sm_count && 4 * blocks < 3 * di->sm_count) return false;
  if (bits == 4) return K >= 1536 || N >= (K >= 1024 ? 4096 : 9472);
  return K >= 2048 || N >= 4096 || (bits == 1 && K <= 512);
}

// Which calls of up to 8 batch rows come here, of those that no balanced pair of kernels takes.  What decides is how the 128-row
// blocks fill the machine and how the 16-row tiles do: the GEMV kernel at b = 4 has room for three tiles an SM (444, 7104 rows),
// and is bound by its table port where this kernel decodes a quarter faster; rows must be long enough to pay for this kernel's
// start.  Lines from a sweep of 16 x 13 shapes (256 to 16384 rows of 256 to 28672 weights) at 1, 2, 4 and 8 batch rows; us per
// call, GEMV or multi-tile / this: b = 4, M = 1 8192 x 8192 15.2 / 11.9, 16384 x 8192 25.4 / 19.4, but 6144 x 6144 7.9 / 8.7 and
// (blocks that fill 58 % of the machine and can not be split) 11008 x 4096 9.6 / 10.2; M = 8 14336 x 4096 17.9 / 11.3,
// 3072 x 8192 8.9 / 7.2; b = 2, M = 8 16384 x 8192 23.4 / 19.3.
// Between kernels of the other kind a call here costs some 2.4 us more (neither can set up beside the other): a decode step of
// 3072 / 8192, b = 4, M = 1 took 345.7 us with its 16384 x 3072 layers here (11.7 / 9.4 by themselves) against 339.2.  Where the
// gain is of that size a call stays where it was, hence the lines at 2^26 weights and at K = 2048 to 4096 (steps of 2048 / 5376,
// b = 4, M = 4 233.7 us, with the 10752 x 2048 layers here 241.4; of 3072 / 8192, M = 4 260.7 / 227.4).
bool linear_umma_few_rows(int64_t N, int64_t K, int bits, int64_t M) {
  const DeviceInfo* di = device_info();
  if (!di || M > 8 || !encode_tiled()) return false;
  const int64_t sms = di->sm_count, blocks = (N + kBM - 1) / kBM, waves = (blocks + sms - 1) / sms;
  const int64_t part = 1000 * blocks / sms;                // thousandths of the SMs that have a block
  if (part < 50) return false;                             // the GEMV kernel's clusters fill the machine with so few
  const int64_t filled = 100 * blocks / (waves * sms);     // % of the machine, one CTA a block
  const bool half = 2 * blocks <= sms;                     // room for two CTAs a block
  if (bits == 4 && M > 2) {
    if (!half) return filled >= 64 ? K >= 2048 : filled >= 55 && K >= 4096;
    if (part >= 355) return K >= (M <= 5 ? 6144 : 4096);
    if (part >= 267) return K >= 3072;
    return K >= (M <= 5 ? 8192 : 6144);
  }
  if (bits == 1 || N * K < (int64_t(1) << 26)) return false;
  if (bits == 4) return !half ? filled >= 64 : part >= 375 || part <= 272;   // between: a cluster of two leaves too many SMs empty
  return M >= 6 && filled >= 75;
}

// Whether more than 128 batch rows go to the CTA pairs (256 x 256 tiles, persistent).  Fitted as above, 5 % standard
// deviation: us per call, pairs / batch tiles of 128 rows: 16384 x 3072, b = 2, M = 1024 95 / 164 (at the time the pairs
// were written); 512 x 1280, b = 1, M = 256 15.3 / 7.2; 13184 x 6528, b = 4, M = 512 95.5 / 82.7.
static bool pair_pays(int64_t N, int64_t K, int bits, int64_t M) {
  const DeviceInfo* di = device_info();
  if (!di || M <= kSingleMaxRows) return false;
  const int64_t sms = di->sm_count;
  const int64_t ctas = 2 * ((N + 2 * kBM - 1) / (2 * kBM) * ((M + kPairMaxRows - 1) / kPairMaxRows));
  const int64_t rounds = (ctas + sms - 1) / sms;
  const int64_t pair = 4700 + rounds * (3100 + K / 16 * (bits == 4 ? 99 : 81)) + 10 * std::min(ctas, sms);
  int64_t single;
  best_split(N, K, bits, M, &single);
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
