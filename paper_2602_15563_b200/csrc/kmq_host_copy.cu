// Small copies between pinned host memory and the device by a kernel, for kmq_linear_host: a call of the layer is a few
// microseconds, and each cudaMemcpyAsync around it costs the hand-over between the compute and the copy engine besides
// its own start (4096 x 4096, b = 1, M = 1, 8 KB each way: 21.7 us with two copies, 13 us of it not the layer).  The
// kernels read or write the pinned memory over the bus directly; under programmatic dependent launch the layer's own
// kernel sets up (packed indices, tables) while the activations arrive.
#include <cuda.h>

#include "kmq_common.cuh"

namespace kmq {
namespace {

constexpr int kCopyThreads = 256;

// 16 bytes per thread and round; the last bytes two at a time (bf16 values)
__global__ void __launch_bounds__(kCopyThreads) host_copy_kernel(void* dst, const void* src, int64_t bytes) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  const int64_t stride = (int64_t)gridDim.x * kCopyThreads, first = (int64_t)blockIdx.x * kCopyThreads + threadIdx.x;
  for (int64_t i = first; i < bytes / 16; i += stride)
    static_cast<uint4*>(dst)[i] = ld_input_u4(static_cast<const uint4*>(src) + i);
  const int64_t tail = bytes / 16 * 8;
  if (tail + first < bytes / 2) static_cast<uint16_t*>(dst)[tail + first] = ld_input_u16(static_cast<const uint16_t*>(src) + tail + first);
}

}  // namespace

// The device's address of pinned host memory that a kernel can copy with 16-byte accesses; nullptr where the memory is
// pageable or unaligned, or the copy is large enough for the copy engine's bandwidth to matter.  The whole copy has to lie
// in one allocation or registration: of a buffer that is pinned in part a kernel would touch unmapped addresses, while
// cudaMemcpyAsync sees the range and refuses.  (One driver call, 35 ns; cudaPointerGetAttributes, which knows no ranges,
// takes 56.)
void* host_copy_address(const void* host, size_t bytes) {
  constexpr size_t kMost = 256 * 1024;
  if (bytes > kMost || (reinterpret_cast<uintptr_t>(host) & 15u) != 0) return nullptr;
  static const auto get_attributes = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPoint("cuPointerGetAttributes", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<CUresult (*)(unsigned int, CUpointer_attribute*, void**, CUdeviceptr)>(p);
  }();
  if (!get_attributes) return nullptr;
  CUmemorytype type = (CUmemorytype)0;   // all of these stay 0 for memory that is not pinned
  CUdeviceptr device = 0, start = 0;
  size_t size = 0;
  CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_POINTER,
                                CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, CU_POINTER_ATTRIBUTE_RANGE_SIZE};
  void* where[] = {&type, &device, &start, &size};
  if (get_attributes(4, what, where, reinterpret_cast<CUdeviceptr>(host)) != CUDA_SUCCESS) return nullptr;
  const bool inside = device >= start && device - start <= size && bytes <= size - (device - start);
  return type == CU_MEMORYTYPE_HOST && inside ? reinterpret_cast<void*>(device) : nullptr;
}

cudaError_t launch_host_copy(void* dst, const void* src, size_t bytes, cudaStream_t s) {
  size_t blocks = (bytes / 16 + kCopyThreads - 1) / kCopyThreads;
  if (blocks < 1) blocks = 1;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kCopyThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, host_copy_kernel, dst, src, (int64_t)bytes);
}

}  // namespace kmq
