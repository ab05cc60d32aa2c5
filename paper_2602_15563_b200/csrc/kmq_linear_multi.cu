// kmq_linear on the tuned (tile-major) layout for batches of up to 32 rows (chosen from 2 to 9 rows on, see
// linear_multi_min_rows, up to where linear_umma_selected takes over): the tiles of a CTA share the staged
// activations, and the decode of a weight fragment is paid once and reused by up to 4 MMAs (one per group of 8 batch rows).
//
// One CTA owns TPC = 4 (or 2) tiles of 16 output rows.  Its 8 warps are 8 / TPC K-groups of TPC warps; warp
// (group, i) owns tile i and the steps s = group, group + 8 / TPC, ... of it.  The warps of a K-group walk the
// same steps together and share the activations under a step: they are copied global -> shared with cp.async, double buffered, one named barrier per
// step.  Per step a warp decodes its 1 KB of packed indices (two 128-bit loads issued one step earlier) into
// mma.sync.m16n8k16 A fragments and multiplies each fragment with the NT B fragments (batch rows 8 nt .. 8 nt + 7)
// read from shared memory.  At the end the other K-groups hand their accumulators to the first through shared
// memory, which adds them, applies the b = 1 codebook and stores bf16.
//
// The weights are rebuilt in registers (Dec1, Dec2, Dec4).  At b = 4 that costs 2.6 integer instructions a weight, and up
// to 16 batch rows the integer pipe bounded the kernel: there the upper 8 rows of a tile come from tables of all 256
// (centroid, centroid) pairs in shared memory, half an instruction and half a load a weight, and the lower 8 from
// registers, so that both pipes carry a part (8192 x 28672, M = 4, us per call before / after: 57.3 / 47.1).
// With more batch rows the port is taken by the activations' fragments.
#include <atomic>

#include "kmq_common.cuh"
#include "kmq_linear_variants.cuh"
#include "kmq_mma_common.cuh"

namespace kmq {
namespace {

constexpr int kMaxSmem = 200 * 1024;                  // dynamic shared memory a variant may ask for
// Pair table of 8 rows: entry e, lane l (the 4 lanes of a row get a bank each) at e * 256 + l * 4; two tables interleave.
constexpr int kEntryStride = 256;
constexpr int kHalfTableBytes = 256 * kEntryStride / 2;

template <int BITS>
struct MGeo {
  static constexpr int kMmaPerWord = 8 / BITS;
  static constexpr int kStepK = 512 / BITS;
  static constexpr int kWordK = 32 / BITS;
  static constexpr int kChunkXBytes = 4 * kWordK * 2;     // activations under one 16-byte chunk of a row
  static constexpr int kChunkStride = kChunkXBytes + 16;  // +16 bytes: conflict-free 16-byte B-fragment loads
  static constexpr int kRowStride = 4 * kChunkStride;     // one batch row of one step
  static constexpr int kPiecesPerRow = kStepK / 8;        // 16-byte pieces per batch row and step
};

// TPC tiles per CTA (2 or 4), W warps -> W / TPC K-groups of TPC warps
template <int BITS, int NT, int TPC, int W = 8>
struct MSmem {
  using G = MGeo<BITS>;
  static constexpr int kGroups = W / TPC;
  static constexpr int kBuf = 8 * NT * G::kRowStride;                 // one x buffer: 8 NT batch rows of one step
  static constexpr int kX = kGroups * 2 * kBuf;                       // double buffered, per K-group
  static constexpr int kRed = (kGroups - 1) * TPC * 32 * NT * 4 * 4;  // accumulators of K-groups 1.. (aliases x)
  static constexpr bool kTab = BITS == 4 && NT <= 2;                   // pair tables of the tiles' upper 8 rows
  static constexpr int kTables = kTab ? TPC * kHalfTableBytes : 0;
  static constexpr int kTotal = kTables + (kX > kRed ? kX : kRed);
};

template <int BITS>
__device__ __forceinline__ int piece_offset(int w) {
  using G = MGeo<BITS>;
  constexpr int kPiecesPerChunk = G::kChunkXBytes / 16;
  return (w / kPiecesPerChunk) * G::kChunkStride + (w % kPiecesPerChunk) * 16;
}

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src, bool valid) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
  const int bytes = valid ? 16 : 0;   // 0 source bytes: the 16 destination bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gmem_src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void group_barrier(int group, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "r"(threads) : "memory");
}

// This lane's four sums of 8 batch rows from `m0` on -> y (rows row0 + g, + 8; batch rows m0 + 2 t, + 1).
__device__ __forceinline__ void store_sums(const float (&v)[4], uint16_t* __restrict__ y, int64_t N, int M, int64_t row0,
                                           int m0, int lane) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int m = m0 + 2 * (lane & 3) + (r & 1);
    const int64_t n = row0 + (lane >> 2) + 8 * (r >> 1);
    if (m < M && n < N) y[(int64_t)m * N + n] = (uint16_t)float_to_bf16_bits(v[r]);
  }
}

// Resident CTAs per SM that the register budget is for (two of 8 warps fit up to 16 batch rows, but only the balanced form,
// whose loop over the groups makes the compiler generous, needs to be told with 4 tiles).
template <int NT, int TPC, int W, bool SPLIT>
constexpr int multi_ctas_per_sm() {
  return W == 8 && (SPLIT || (NT <= 2 && TPC == 2)) ? 2 : 1;
}

// SPLIT: the balanced form.  The (group of TPC tiles, step) units, group by group, are cut into gridDim.x equal ranges,
// one per resident CTA; a group that several CTAs share leaves its sums in scratch for linear_multi_sum_kernel.
template <int BITS, int NT, int TPC, int W, bool SPLIT>
__global__ void __launch_bounds__(W * 32, (multi_ctas_per_sm<NT, TPC, W, SPLIT>())) linear_multi_kernel(
    const uint32_t* __restrict__ packed, const uint16_t* __restrict__ cb, const uint16_t* x,
    uint16_t* __restrict__ y, int64_t N, int64_t K, int M, float* __restrict__ scratch) {
  using G = MGeo<BITS>;
  using SM = MSmem<BITS, NT, TPC, W>;
  constexpr int kThreads = W * 32;
  constexpr int Q = G::kMmaPerWord;
  constexpr int kGroups = SM::kGroups, kGroupThreads = TPC * 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* const xbase = smem_raw + SM::kTables;
  float* const red = reinterpret_cast<float*>(xbase);                       // reused after the main loop

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;
  const int wt = warp % TPC, group = warp / TPC;       // tile inside the CTA, K-group
  const int gtid = threadIdx.x - group * kGroupThreads;  // thread inside the K-group
  const int64_t tiles = (N + kTileRows - 1) / kTileRows;
  const int steps = (int)tuned_row_steps(K, BITS);
  int64_t u0 = 0, u1 = 0, tg = blockIdx.x;   // SPLIT: units of this CTA; group of tiles
  if constexpr (SPLIT) {
    const int64_t units = (tiles + TPC - 1) / TPC * steps;
    u0 = units * blockIdx.x / gridDim.x;
    u1 = units * (blockIdx.x + 1) / gridDim.x;
    tg = u0 / steps;
  }
  unsigned char* const xgroup = xbase + group * 2 * SM::kBuf;

  // copy the activations under step s into buffer `buf` of this K-group (zeros past K; rows >= M are not touched:
  // their MMA columns are never stored)
  auto stage = [&](int s, int buf) {
    unsigned char* dst = xgroup + buf * SM::kBuf;
    const int total = M * G::kPiecesPerRow;
    for (int p = gtid; p < total; p += kGroupThreads) {
      const int m = p / G::kPiecesPerRow, w = p % G::kPiecesPerRow;
      const int64_t k = (int64_t)s * G::kStepK + w * 8;
      const bool ok = k < K;
      cp_async16(dst + m * G::kRowStride + piece_offset<BITS>(w), x + (int64_t)m * K + (ok ? k : 0), ok);
    }
    cp_async_commit();
  };

 do {   // one pass unless SPLIT
  const int64_t base = tg * steps;
  const int sa = SPLIT && u0 > base ? (int)(u0 - base) : 0, sb = SPLIT && u1 - base < steps ? (int)(u1 - base) : steps;
  const int64_t tile_id = tg * TPC + wt;
  const bool has_tile = tile_id < tiles;               // warp-uniform; such a warp still stages x and joins barriers
  const int64_t row0 = tile_id * kTileRows;
  const uint4* __restrict__ tile =
      reinterpret_cast<const uint4*>(packed) + (has_tile ? tile_id : 0) * (int64_t)steps * 64 + lane;
  // ---- first loads: weights of this warp's first two steps, activations of the group's first step ----
  uint4 qa[2], qb[2];
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    const int s = sa + group + d * kGroups;
    qa[d] = qb[d] = make_uint4(0, 0, 0, 0);
    if (has_tile && s < sb) {
      qa[d] = ldg_stream_u4(tile + (int64_t)s * 64);
      qb[d] = ldg_stream_u4(tile + (int64_t)s * 64 + 32);
    }
  }
  // ---- per-row decode state ----
  Dec1 sg, sh;
  if constexpr (BITS == 1) {
    sg.init(cb + min(row0 + g, N - 1) * 2);
    sh.init(cb + min(row0 + g + 8, N - 1) * 2);
  }
  Dec2 dg, dh;
  if constexpr (BITS == 2) {
    dg.init(cb + min(row0 + g, N - 1) * 4);
    dh.init(cb + min(row0 + g + 8, N - 1) * 4);
  }
  Dec4 fg, fh;
  if constexpr (BITS == 4) {
    if constexpr (!SM::kTab) fg.init(cb + min(row0 + g, N - 1) * 16);
    fh.init(cb + min(row0 + g + 8, N - 1) * 16);
  }
  if (SPLIT && base > u0) __syncthreads();   // the previous group's sums are read (they lie over the activations)
  if constexpr (SM::kTab) {
    // a thread takes a row and a low index: one fetch of the row's centroids, the 16 entries low + 16 high
    for (int it = threadIdx.x; it < TPC * 128; it += kThreads) {
      const int r8 = it & 7, low = (it >> 3) & 15, i = it >> 7;
      const int64_t row = min((tg * TPC + i) * kTileRows + r8, N - 1);
      const uint16_t* const crow = cb + row * 16;
      const uint4 ca = __ldg(reinterpret_cast<const uint4*>(crow)), cc = __ldg(reinterpret_cast<const uint4*>(crow) + 1);
      const uint32_t lo = __ldg(crow + low);
      const uint32_t c2[8] = {ca.x, ca.y, ca.z, ca.w, cc.x, cc.y, cc.z, cc.w};
      unsigned char* const dst = smem_raw + (i >> 1) * (2 * kHalfTableBytes) + (i & 1) * 128 + low * kEntryStride + r8 * 16;
#pragma unroll
      for (int hi = 0; hi < 16; ++hi) {
        const uint32_t v = prmt(lo, c2[hi >> 1], (hi & 1) ? 0x7610u : 0x5410u);
        *reinterpret_cast<uint4*>(dst + hi * 16 * kEntryStride) = make_uint4(v, v, v, v);
      }
    }
    __syncthreads();
  }
  // this lane's bank of the tile's table; byte 1 is the entry's place
  const uint32_t bank = (wt >> 1) * (2 * kHalfTableBytes) + (wt & 1) * 128 + lane * 4;
  // Programmatic dependent launch: up to here only the packed indices and the codebooks were read (constants of the
  // layer); the activations may come from the previous kernel on the stream and are read only once it has completed.
  // At b = 4, where the set-up of a CTA is long (its tables), the next kernel is released at once so that its CTAs
  // set up under this grid's MMAs; otherwise just before the partial sums are exchanged (measured, 4096 x 4096 M = 16:
  // b = 4 9.7 -> 8.3 us early, 8.7 late; b = 2 6.4 -> 6.3 / 6.5; 8192 x 8192 b = 2 M = 32 20.1 -> 20.1 / 19.5).
  if (!SPLIT || base <= u0) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if constexpr (BITS == 4) asm volatile("griddepcontrol.launch_dependents;");
  }
  if (sa + group < sb) stage(sa + group, 0);

  float acc[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;

  for (int s0 = sa + group; s0 < sb; s0 += 2 * kGroups) {   // uniform over the K-group
#pragma unroll
   for (int buf = 0; buf < 2; ++buf) {                     // buffer index = parity of the group's step count
    const int s = s0 + buf * kGroups;
    if (s >= sb) break;
    cp_async_wait_all();
    group_barrier(group, kGroupThreads);   // x of step s is in place, and every warp of the group is done with step s - 2
    if (s + kGroups < sb) stage(s + kGroups, buf ^ 1);
    const unsigned char* const xs = xgroup + buf * SM::kBuf;
    if (has_tile) {
      const uint4 va = qa[buf], vb = qb[buf];
      const uint32_t wa[4] = {va.x, va.y, va.z, va.w};
      const uint32_t wb[4] = {vb.x, vb.y, vb.z, vb.w};
      if (s + 2 * kGroups < sb) {   // refill for the step after next
        qa[buf] = ldg_stream_u4(tile + (int64_t)(s + 2 * kGroups) * 64);
        qb[buf] = ldg_stream_u4(tile + (int64_t)(s + 2 * kGroups) * 64 + 32);
      }
      const unsigned char* const xb = xs + g * G::kRowStride + t * G::kChunkStride;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        uint32_t dg4[4], dh4[4];
        if constexpr (BITS == 4) {
          if constexpr (!SM::kTab) fg.word(wa[j], dg4);
          fh.word(wb[j], dh4);
        }
#pragma unroll
        for (int q2 = 0; q2 < Q; q2 += 2) {
          uint4 xv[NT];   // 16 bytes of x per batch row = the k-slots of two consecutive MMAs
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            xv[nt] = *reinterpret_cast<const uint4*>(xb + nt * 8 * G::kRowStride + (j * Q + q2) * 8);
#pragma unroll
          for (int qq = 0; qq < 2; ++qq) {
            const int q = q2 + qq;
            uint32_t a0, a1, a2, a3;
            if constexpr (BITS == 2) {
              dg.pair(wa[j], q, a0, a2);
              dh.pair(wb[j], q, a1, a3);
            } else if constexpr (BITS == 4) {
              if constexpr (SM::kTab) {
                // index byte k of the word in byte 1 of `bank`
                const uint32_t o0 = prmt(wa[j], bank, 0x7604u | ((2 * q) << 4));
                const uint32_t o1 = prmt(wa[j], bank, 0x7604u | ((2 * q + 1) << 4));
                a0 = *reinterpret_cast<const uint32_t*>(smem_raw + o0);
                a2 = *reinterpret_cast<const uint32_t*>(smem_raw + o1);
              } else {
                a0 = dg4[2 * q];
                a2 = dg4[2 * q + 1];
              }
              a1 = dh4[2 * q];
              a3 = dh4[2 * q + 1];
            } else {
              const uint32_t m0 = kPow2[2 * q], m1 = kPow2[2 * q + 1];
              a0 = sg.select(wa[j] * m0);
              a2 = sg.select(wa[j] * m1);
              a1 = sh.select(wb[j] * m0);
              a3 = sh.select(wb[j] * m1);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
              mma_bf16_16816(acc[nt], a0, a1, a2, a3, qq ? xv[nt].z : xv[nt].x, qq ? xv[nt].w : xv[nt].y);
          }
        }
      }
    }
   }
  }

  // ---- K-groups 1.. hand their partial sums to K-group 0, which adds and stores ----
  if (!SPLIT || base + steps >= u1) asm volatile("griddepcontrol.launch_dependents;");
  __syncthreads();   // every warp is done with the x buffers; `red` aliases them
  if (group > 0) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
      *reinterpret_cast<float4*>(red + ((((group - 1) * TPC + wt) * NT + nt) * 32 + lane) * 4) =
          make_float4(acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]);
  }
  __syncthreads();
  if (group == 0 && has_tile) {
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float v[4] = {acc[nt][0], acc[nt][1], acc[nt][2], acc[nt][3]};
#pragma unroll
      for (int gq = 1; gq < kGroups; ++gq) {
        const float4 o =
            *reinterpret_cast<const float4*>(red + ((((gq - 1) * TPC + wt) * NT + nt) * 32 + lane) * 4);
        v[0] += o.x; v[1] += o.y; v[2] += o.z; v[3] += o.w;
      }
      if (!SPLIT || (sa == 0 && sb == steps)) store_sums(v, y, N, M, row0, nt * 8, lane);
      else
        reinterpret_cast<float4*>(scratch)[(((int64_t)blockIdx.x * 2 + (sa == 0 ? 1 : 0)) * (TPC * NT) + wt * NT + nt) * 32 +
                                           lane] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
 } while (SPLIT && ++tg * steps < u1);
}

// Block (c, tile of the group) adds the shares of group c where more than one CTA worked on it: slot [.][1] of the CTA
// that started it, slot [.][0] of every later one, in that order.
template <int BITS, int NT, int TPC>
__global__ void __launch_bounds__(32 * NT) linear_multi_sum_kernel(const float* scratch,
                                                                   uint16_t* __restrict__ y, int64_t N, int64_t K, int M,
                                                                   int ctas) {
  const int64_t steps = tuned_row_steps(K, BITS), groups = (N + TPC * kTileRows - 1) / (TPC * kTileRows);
  const int64_t units = groups * steps;
  // CTA c works on units [units c / ctas, units (c + 1) / ctas): unit u belongs to CTA ((u + 1) ctas - 1) / units
  const int64_t first = (int64_t)blockIdx.x * steps, last = first + steps - 1;
  const int64_t c0 = ((first + 1) * ctas - 1) / units, c1 = ((last + 1) * ctas - 1) / units;
  // At b = 4 the next call's CTAs set up (tables) under the first kernel's MMAs, as they do without this kernel: it releases
  // them before its own wait (8192 x 28672, M = 3 45.6 -> 44.9 us; 8192 x 16384 29.1 -> 28.6).  With more than 8 batch rows
  // and at b = 1, 2, where the set-up is short, that gave nothing or cost up to 1 %.
  constexpr bool kEarly = BITS == 4 && NT == 1;
  if constexpr (kEarly) asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");   // every block: this grid must not be complete before the first is
  if constexpr (!kEarly) asm volatile("griddepcontrol.launch_dependents;");
  if (c0 == c1) return;
  const float4* const src = reinterpret_cast<const float4*>(scratch) + (int64_t)blockIdx.y * NT * 32 + threadIdx.x;
  constexpr int kSlot = TPC * NT * 32;
  float v[4];
  const uint4 a = ld_input_u4(src + (c0 * 2 + 1) * kSlot);
  v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
  for (int64_t c = c0 + 1; c <= c1; ++c) {
    const uint4 b = ld_input_u4(src + c * 2 * kSlot);
    v[0] += __uint_as_float(b.x); v[1] += __uint_as_float(b.y); v[2] += __uint_as_float(b.z); v[3] += __uint_as_float(b.w);
  }
  store_sums(v, y, N, M, ((int64_t)blockIdx.x * TPC + blockIdx.y) * kTileRows, (threadIdx.x >> 5) * 8, threadIdx.x & 31);
}

// CTAs of the balanced form that fit an SM, asked from the runtime once per device.
template <int BITS, int NT, int TPC, int W>
int resident_ctas() {
  static std::atomic<int> cached[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = cached[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    constexpr int smem = MSmem<BITS, NT, TPC, W>::kTotal;
    if (cudaFuncSetAttribute(linear_multi_kernel<BITS, NT, TPC, W, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, linear_multi_kernel<BITS, NT, TPC, W, true>, W * 32, smem) !=
            cudaSuccess)
      return 0;
    cached[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

// A call; with `plan` set nothing is launched, and the shape of its CTA is put there.
struct MultiCall {
  const uint32_t* packed;
  const uint16_t *cb, *x;
  uint16_t* y;
  int64_t N, K;
  int M;
  float* scratch;   // not null: the balanced form
  MultiSplit* plan;
  cudaStream_t s;
};

// BALANCED: this shape of CTA has a balanced form.
template <int BITS, int NT, int TPC, int W = 8, bool BALANCED = true>
cudaError_t launch_nt(const MultiCall& c) {
  constexpr int smem = MSmem<BITS, NT, TPC, W>::kTotal;
  const int64_t tiles = (c.N + kTileRows - 1) / kTileRows, groups = (tiles + TPC - 1) / TPC;
  int slots = 0;
  if constexpr (BALANCED) {
    const DeviceInfo* di = device_info();
    if (!di) return cudaErrorInvalidDevice;
    slots = di->sm_count * resident_ctas<BITS, NT, TPC, W>();
    if (slots <= 0) return cudaErrorInvalidConfiguration;
  }
  if (c.plan) {
    c.plan->ctas = slots;
    c.plan->tiles = TPC;
    c.plan->groups = groups;
    c.plan->scratch = (size_t)slots * 2 * TPC * NT * 512;
    return cudaSuccess;
  }
  static bool configured[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !configured[dev]) {   // (the balanced form: resident_ctas())
    cudaError_t e = cudaFuncSetAttribute(linear_multi_kernel<BITS, NT, TPC, W, false>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    configured[dev] = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)groups);
  cfg.blockDim = dim3(W * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c.s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (BALANCED) {
    if (c.scratch) {
      cfg.gridDim = dim3((unsigned)slots);
      cudaError_t e = cudaLaunchKernelEx(&cfg, linear_multi_kernel<BITS, NT, TPC, W, true>, c.packed, c.cb, c.x, c.y, c.N, c.K,
                                         c.M, c.scratch);
      if (e != cudaSuccess) return e;
      cfg.gridDim = dim3((unsigned)groups, TPC);
      cfg.blockDim = dim3(32 * NT);
      cfg.dynamicSmemBytes = 0;
      return cudaLaunchKernelEx(&cfg, linear_multi_sum_kernel<BITS, NT, TPC>, (const float*)c.scratch, c.y, c.N, c.K, c.M,
                                slots);
    }
  }
  return cudaLaunchKernelEx(&cfg, linear_multi_kernel<BITS, NT, TPC, W, false>, c.packed, c.cb, c.x, c.y, c.N, c.K, c.M,
                            (float*)nullptr);
}

template <int BITS>
cudaError_t launch_bits(const MultiCall& c) {
  const int64_t N = c.N, K = c.K;
  const int M = c.M;
  // Tiles per CTA: 4 share the staged activations among more warps, 2 give twice as many CTAs.  Measured: 2 wins
  // when 4 would leave more than half of the SMs without a CTA, and for b = 2, 4 (two CTAs then fit an SM).
  const DeviceInfo* di = device_info();
  const int64_t tiles = (N + kTileRows - 1) / kTileRows;
  const bool few = (tiles + 3) / 4 <= (di ? di->sm_count : 148) / 2;
  const bool fits_one_wave = (tiles + 3) / 4 <= (di ? di->sm_count : 148);   // CTAs of 4 tiles <= SMs
  // few tiles and a long K: 2 tiles x 8 K-groups (16 warps) while each K-group still gets 4 steps or more
  // (4096 x 11008, b = 2, M = 6: 13.4 -> 9.0 us; 4160 x 4096, b = 4, M = 7 7.8 -> 5.9; 4096 x 11008, b = 1, M = 8 12.1, 12.2)
  const bool few16 = few && (tiles + 1) / 2 <= (di ? di->sm_count : 148) && tuned_row_steps(K, BITS) >= 32;
  if (M <= 8) {
    // same shape of CTA for up to 8 batch rows (8192 x 28672, b = 1, M = 4: 35.0 -> 23.5 us; 8192 x 8192, b = 2,
    // M = 8: 12.7 -> 11.7 us)
    if (!few && fits_one_wave) return launch_nt<BITS, 1, 4, 16>(c);
    if constexpr (MSmem<BITS, 1, 2, 16>::kTotal <= kMaxSmem) {
      if (few16) return launch_nt<BITS, 1, 2, 16>(c);
    }
    if (few || BITS != 1) return launch_nt<BITS, 1, 2>(c);
    return launch_nt<BITS, 1, 4>(c);
  }
  // More rows: what linear_umma_selected leaves.  Where a driver has no tensor-map encoder, all calls of more rows are made with
  // these forms, which serve any shape.
  if (M <= 16) {
    if constexpr (BITS == 1) {
      if (!few) return launch_nt<BITS, 2, 4>(c);
    } else if constexpr (BITS == 4) {   // 6000 x 768, M = 12 4.0 -> 3.2 us, 9000 x 896, M = 16 5.1 -> 3.9
      if (!few && fits_one_wave) return launch_nt<BITS, 2, 4, 16, false>(c);
    }
    return launch_nt<BITS, 2, 2, 8, false>(c);
  }
  // b = 1 (only without the encoder): 4 K-groups of 2 tiles would need 278 KB for their activations
  if (M <= 32) return launch_nt<BITS, 4, BITS == 1 ? 4 : 2, 8, false>(c);
  return cudaErrorInvalidValue;   // unreachable: launched in passes of linear_multi_rows_per_launch() rows
}

}  // namespace

// Batch rows per launch of the multi-tile kernel (more than that come here only where the tcgen05 kernel can not run).
int linear_multi_rows_per_launch() { return 32; }

// Smallest batch that goes to the multi-tile kernel.  The GEMV kernel stages the activations once per tile, here the tiles
// of a CTA share them; but its grid is finer, and it shares K among a cluster.  The lines below are from a sweep of 20 to
// 1024 tiles by 4 to 224 steps at every batch up to 8, both kernels on all of it; us per call, GEMV / multi-tile:
//   More than three tiles per SM.  The multi-tile kernel has the better of it up to four, where its groups are one wave;
//   with up to six the second wave is nearly empty, and on short rows the finer grid wins.
//     b = 1  2 rows on (8192 x 4096, M = 2 5.6 / 6.0, M = 3 6.3 / 6.0).  Beyond four tiles per SM 3 with 4 to 32 steps, of
//            more than six tiles 8 to 32 (9600 x 4096, M = 2 6.3 / 9.2), and 5 with 4 to 12 steps of up to five tiles
//            (11008 x 4096, M = 3 7.6 / 9.6).  Not on shorter rows (9600 x 1024, M = 2 and 3 13 and 25 % faster here).
//     b = 2  5 rows on (8192 x 4096, M = 5 7.7 / 6.6; M = 4 6.8 / 6.6, but 9600 x 4096, M = 4 7.8 / 9.2), on long rows 2
//            (7200 x 24576, M = 2 28.6 / 24.1).
//     b = 4  from two tiles per SM on, where the GEMV kernel's tables leave room for two CTAs per SM from 3 rows on: 3
//            (8192 x 4096, M = 3 9.4 / 8.4), 5 with 13 to 32 steps of four to six tiles (12288 x 4096, M = 3 13.7 / 15.2;
//            11008 x 2048, M = 3 7.5 / 8.6; 11008 x 8192 23.6 / 21.9).
//   Fewer tiles.
//     b = 1  5 (1024 x 8192, M = 3 3.5 / 5.4; 6144 x 8192, M = 4 8.4 / 9.8), on long rows 3 (4160 x 24576, M = 3
//            15.1 / 14.1), and with an even number of steps below 8 on one to one and a half tiles per SM (3072 x 3072,
//            M = 3 3.6 / 3.4; an odd number is slower by 2 to 11 % on nine widths, 3072 x 2560 3.1 / 3.4).
//     b = 2  9.  On long rows 2 with one and a half to two tiles per SM (4160 x 10240, M = 3 9.8 / 7.9); 5 below that, where
//            the GEMV kernel uses clusters (2976 x 16384, M = 4 9.6 / 10.5, M = 8 11.5 / 11.0), with less than a tile per SM
//            from 64 steps on (1600 x 16384, M = 8 9.4 / 8.6, but 2336 x 10240, M = 4 5.4 / 7.7) and 2 from 81 on
//            (1600 x 24576, M = 4 10.9 / 9.7).
//     b = 4  9.  With one to two tiles per SM 3 on long rows (2976 x 16384, M = 3 15.4 / 14.3) and 7 on medium ones
//            (4160 x 8192, M = 8 10.5 / 9.0).
int linear_multi_min_rows(int bits, int64_t N, int64_t K) {
  const DeviceInfo* di = device_info();
  const int64_t sms = di ? di->sm_count : 148, tiles = (N + kTileRows - 1) / kTileRows, steps = tuned_row_steps(K, bits);
  const bool second_wave = tiles > 4 * sms && tiles <= 6 * sms;
  if (bits == 1) {
    if (tiles > 4 * sms && steps >= (second_wave ? 4 : 8) && steps <= 32) return steps <= 12 && tiles <= 5 * sms ? 5 : 3;
    if (tiles > 3 * sms) return 2;
    return steps > 32 || (steps < 8 && steps % 2 == 0 && tiles > sms && 2 * tiles <= 3 * sms) ? 3 : 5;
  }
  if (bits == 2) {
    if (tiles > 3 * sms) return steps > 64 ? 2 : 5;
    if (steps <= 32 || 2 * tiles <= sms || tiles > 2 * sms) return 9;
    if (2 * tiles > 3 * sms) return 2;
    if (tiles > sms) return 5;
    return steps > 80 ? 2 : steps >= 64 ? 5 : 9;
  }
  if (tiles > 2 * sms) return second_wave && steps > 12 && steps <= 32 ? 5 : 3;
  if (tiles <= sms || steps < 32) return 9;
  return steps > 64 ? 3 : 7;
}

static cudaError_t launch_multi(int bits, const MultiCall& c) {
  return bits == 1 ? launch_bits<1>(c) : bits == 2 ? launch_bits<2>(c) : launch_bits<4>(c);
}

// Whether the balanced form is used (ctas > 0), and its scratch.  It saves the steps in which the last wave leaves CTA
// slots empty and costs the second kernel and a CTA's start on one or two more groups.  us per call, without / with:
//   up to 8 batch rows, from sweeps of 20 to 1300 groups by 8 to 224 steps: the cost, in thousands of weights on an SM, which
//          the weights of the steps saved have to exceed, is 190 at b = 1 (12288 x 4096, 184, M = 3 9.8 / 10.3;
//          16384 x 12288, 213, M = 8 27.1 / 26.0), 172 at b = 2 (8192 x 16384, 142, M = 3 19.4 / 19.5; 5120 x 8192, 241,
//          M = 8 10.9 / 9.5), but 340 there in two waves or more: the CTAs of a last wave have an SM to themselves and finish
//          early (12288 x 4096, 184, M = 8 10.8 / 11.7; 9600 x 6144, 387, 13.3 / 12.5).  At b = 4 165 (5632 x 6144, 159,
//          M = 8 12.0 / 12.2; 6400 x 8192, 170, 15.5 / 15.3), 140 where the groups nearly fill the SMs, so that few are
//          shared by more than two CTAs (8192 x 16384, 142, M = 3 28.4 / 28.6, M = 8 29.5 / 29.4; 8192 x 20480, 177,
//          M = 8 36.0 / 35.0).
//   more   at b = 1, 4 tiles a CTA, the only calls of more rows here that leave slots empty on long rows: 180 (14080 x 8192,
//          M = 16 23.4 / 21.2; 9600 x 16384 42.6 / 26.9).
MultiSplit linear_multi_split(int64_t N, int64_t K, int bits, int64_t M) {
  MultiSplit sp = {};
  const DeviceInfo* di = device_info();
  if (!di || M > linear_multi_rows_per_launch()) return sp;
  if (launch_multi(bits, {nullptr, nullptr, nullptr, nullptr, N, K, (int)M, nullptr, &sp, nullptr}) != cudaSuccess || sp.ctas == 0)
    return {};
  const int64_t steps = tuned_row_steps(K, bits), sms = di->sm_count;
  // CTAs that have an SM to themselves run as fast as the SM lets them: then it is the SMs that are empty, not the slots
  const int64_t slots = sp.groups <= sms ? sms : sp.ctas, waves = (sp.groups + slots - 1) / slots;
  const double saved = (double)(waves * slots - sp.groups) / slots * (double)steps;
  const double weights = saved * (double)(slots / sms) * sp.tiles * (kTileRows * 512 / bits);   // of one SM
  double cost;
  if (M > 8) cost = 180e3;
  else if (bits == 4) cost = sp.groups <= sms && 6 * sp.groups >= 5 * sms ? 140e3 : 165e3;
  else cost = bits == 1 ? 190e3 : waves > 1 ? 340e3 : 172e3;
  return weights > cost && sp.groups * steps >= sp.ctas ? sp : MultiSplit{};
}

cudaError_t launch_linear_multi(const uint32_t* packed, const uint16_t* cb, const uint16_t* x, uint16_t* y, int64_t N,
                                int64_t K, int bits, int64_t M, void* scratch, cudaStream_t s) {
  const int64_t per = linear_multi_rows_per_launch();
  for (int64_t m0 = 0; m0 < M; m0 += per) {
    const int mc = (int)(M - m0 < per ? M - m0 : per);
    const uint16_t* xp = x + m0 * K;
    uint16_t* yp = y + m0 * N;
    cudaError_t e;
    if (mc < linear_multi_min_rows(bits, N, K)) e = launch_linear_tiled(packed, cb, xp, yp, N, K, bits, mc, s);   // a short tail
    else e = launch_multi(bits, {packed, cb, xp, yp, N, K, mc, static_cast<float*>(scratch), nullptr, s});
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace kmq
