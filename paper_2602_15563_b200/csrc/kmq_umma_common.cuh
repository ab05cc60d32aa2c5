// Pieces shared by the tcgen05 kernels of kmq_linear (kmq_linear_umma.cu, kmq_linear_umma_pair.cuh): mbarriers with
// bounded waits, TMA tile loads of the activations, the tcgen05 instructions, the decode of packed words into tensor
// memory.
#pragma once
#include <cuda.h>

#include "kmq_common.cuh"
#include "kmq_linear_variants.cuh"
#include "kmq_mma_common.cuh"

namespace kmq {
namespace umma {

constexpr int kBM = 128;                                 // output rows per CTA (rows of the MMA)
constexpr int kDecodeWarps = 16;                         // 4 tensor-memory lane quarters x 4 quarters of a stage's weights
constexpr int kDecodeThreads = kDecodeWarps * 32;
constexpr int kThreads = kDecodeThreads + 64;            // + the MMA warp + the TMA producer warp
constexpr int kWRing = 6;                   // ring of 1 KB steps of packed words per tile (cp.async), kWRing - 1 in flight
constexpr int kWRowStride = 80;                          // a row's 64 bytes of a step, padded: lanes read consecutive rows
constexpr int kWStepBytes = kBM * kWRowStride;
constexpr uint32_t kWaitHintNs = 20000;                  // one try_wait on an mbarrier may park the thread this long
constexpr uint64_t kWaitLimitNs = 100ull * 1000 * 1000;  // a wait gives up after this much time on the global timer

template <int BITS>
struct UGeo {
  static constexpr int kStageK = 128;                            // weights of a row per stage
  static constexpr int kStagesPerStep = (512 / BITS) / kStageK;  // 1, 2, 4 for b = 4, 2, 1
  static constexpr int kThreadBytes = kStageK * BITS / 32;       // packed bytes a thread decodes per stage: 16, 8, 4
  static constexpr int kCols = kStageK / 2;                      // 32-bit columns of the A operand of a stage
  static constexpr int kKSlices = kStageK / 16;                  // MMAs per stage
};

// Shared-memory matrix descriptor of a K-major operand in the 128-byte-swizzle layout TMA writes: rows of 128 bytes,
// 8-row groups 1024 bytes apart (stride byte offset), descriptor version of sm_100, layout type 2 = 128-byte swizzle.
// The buffer is 1024-byte aligned; 16 weights further along K = 32 bytes further in the start address.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// TMA tile load of the box at (c0, c1) of a 2-D tensor map into shared memory; its bytes complete on `bar`.
__device__ __forceinline__ void tma_load_2d(uint32_t smem_dst, const CUtensorMap* map, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

// D (tensor memory) (+)= A (tensor memory) x B (shared memory descriptor), issued by one elected lane of a converged warp.
__device__ __forceinline__ void umma_bf16_elect(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                                uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, one;\n\telect.sync _|one, 0xFFFFFFFF;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "@one tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      :
      : "r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit_elect(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred one;\n\telect.sync _|one, 0xFFFFFFFF;\n\t"
      "@one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
      : "memory");
}
// Announces `bytes` on `bar` and loads the boxes at (ca, c1) and (cb, c1) of a 2-D tensor map to two places.
__device__ __forceinline__ void tma_load_pair_elect(uint32_t dst_a, uint32_t dst_b, uint32_t bytes, const CUtensorMap* map,
                                                    int ca, int cb, int c1, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred one;\n\telect.sync _|one, 0xFFFFFFFF;\n\t"
      "@one mbarrier.arrive.expect_tx.shared::cta.b64 _, [%7], %2;\n\t"
      "@one cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%3, {%4, %6}], [%7];\n\t"
      "@one cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%1], [%3, {%5, %6}], [%7];\n\t}"
      ::"r"(dst_a), "r"(dst_b), "r"(bytes), "l"(reinterpret_cast<uint64_t>(map)), "r"(ca), "r"(cb), "r"(c1), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tmem_store8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void cp_async16(uint32_t smem_dst, const void* gmem_src, bool valid) {
  const int bytes = valid ? 16 : 0;   // 0 source bytes: the 16 destination bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gmem_src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// All threads of all CTAs of the cluster.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The shared::cluster address of CTA `rank`'s copy of this CTA's shared-memory address `saddr`.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t saddr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// This thread's lane of 8 columns from `taddr` on, added up over ACCS accumulators that lie `stride` columns apart (zeros when
// nothing was accumulated).  All loads are issued before the one wait; their registers pass through an empty statement behind
// it, so that no use of them is moved ahead of it.
template <int ACCS>
__device__ __forceinline__ void load_acc(uint32_t (&w)[8], uint32_t taddr, int stride, bool valid) {
  if (valid) {
    uint32_t r[ACCS][8];
#pragma unroll
    for (int a = 0; a < ACCS; ++a)
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(r[a][0]), "=r"(r[a][1]), "=r"(r[a][2]), "=r"(r[a][3]), "=r"(r[a][4]), "=r"(r[a][5]), "=r"(r[a][6]),
                     "=r"(r[a][7])
                   : "r"(taddr + a * stride));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int a = 0; a < ACCS; ++a)
      asm volatile("" : "+r"(r[a][0]), "+r"(r[a][1]), "+r"(r[a][2]), "+r"(r[a][3]), "+r"(r[a][4]), "+r"(r[a][5]),
                        "+r"(r[a][6]), "+r"(r[a][7])::"memory");
#pragma unroll
    for (int j = 0; j < 8; ++j) {
#pragma unroll
      for (int n = ACCS; n > 1; n /= 2)
#pragma unroll
        for (int a = 0; a < n / 2; ++a) r[a][j] = __float_as_uint(__uint_as_float(r[a][j]) + __uint_as_float(r[a + n / 2][j]));
      w[j] = r[0][j];
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = 0;
  }
}

// Bounded wait for the phase of parity `parity` of an mbarrier.  try_wait parks the thread in hardware for up to the
// hinted time instead of spinning, so waiting warps do not take issue slots from the ones that decode.  The hint is
// only a hint (a try may come back early), so the bound is taken on the global timer, not on the number of tries.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns = kWaitLimitNs) {
  uint64_t t0 = 0;
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(kWaitHintNs)
        : "memory");
    if (done) return true;
    uint64_t now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (t0 == 0) t0 = now;
    else if (now - t0 > limit_ns) return false;
  }
}

// The same for a barrier at which a thread of another CTA of the cluster arrives.
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity) {
  uint64_t t0 = 0;
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(kWaitHintNs)
        : "memory");
    if (done) return true;
    uint64_t now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (t0 == 0) t0 = now;
    else if (now - t0 > kWaitLimitNs) return false;
  }
}

// Decode state of a thread's output row.
template <int BITS>
struct RowState;
template <>
struct RowState<1> {
  Dec1 d;
};
template <>
struct RowState<2> {
  Dec2 d;
};
template <>
struct RowState<4> {
  Dec4 d;
};

// The packed words of a row in a stage -> bf16 pairs in the order of k, written to consecutive columns of the row's
// tensor-memory lane starting at `taddr`.
template <int BITS, int NW>
__device__ __forceinline__ void decode_to_tmem(const uint32_t (&w)[NW], const RowState<BITS>& st, uint32_t taddr) {
  constexpr int kRegs = 16 / BITS * NW;   // 16 per thread and stage
#pragma unroll
  for (int c = 0; c < kRegs; c += 8) {
    uint32_t a[8];
    if constexpr (BITS == 4) {
      uint32_t x[4], y[4];
      st.d.word(w[c / 4], x);
      st.d.word(w[c / 4 + 1], y);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = x[i];
        a[4 + i] = y[i];
      }
    } else if constexpr (BITS == 2) {
#pragma unroll
      for (int q = 0; q < 4; ++q) st.d.pair(w[c / 8], q, a[2 * q], a[2 * q + 1]);   // weights 4q .. 4q + 3
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = st.d.select(w[0] * kPow2[c + i]);   // weights 2 (c + i), 2 (c + i) + 1
    }
    tmem_store8(taddr + c, a);
  }
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once through the runtime (no link against the driver library).
inline EncodeTiledFn encode_tiled() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// x as a 2-D tensor [M rows][K] of bf16; boxes of `rows` x 64 columns (128 bytes) land in shared memory with the
// 128-byte swizzle; rows past M and columns past K read as zero.
inline bool make_x_map(CUtensorMap* map, const uint16_t* x, int64_t K, int64_t M, int rows) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)rows};
  const cuuint32_t elem[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(x), dims, strides, box, elem,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Dynamic shared memory to launch with: what the kernel uses, but more than half of what an SM offers (the opt-in
// maximum per CTA is the SM's shared memory minus the 1 KB the system keeps per CTA).
inline int umma_launch_smem(int kernel_bytes, int max_smem_optin) {
  const int more_than_half = max_smem_optin / 2 + 1024;
  return kernel_bytes > more_than_half ? kernel_bytes : more_than_half;
}

}  // namespace umma
}  // namespace kmq
