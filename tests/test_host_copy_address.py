"""Which host buffers kmq_linear_host lets a kernel copy: only those that lie whole inside one pinned allocation or
registration.  The rule is host code; it is compiled here against a stand-in for the driver's and the runtime's pointer
queries (one pinned range of 8 KB, a second one right behind a page that is not pinned), so no GPU is involved."""
import os
import subprocess

import pytest

from paper_2602_15563_b200 import build as kb

HARNESS = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

struct Range { uintptr_t start; size_t size; };
static const Range kPinned[] = {{0x100000, 8192}, {0x103000, 4096}};
static const Range* find(uintptr_t p) {
  for (const Range& r : kPinned) if (p >= r.start && p - r.start < r.size) return &r;
  return nullptr;
}
static CUresult fake_attributes(unsigned int n, CUpointer_attribute* what, void** where, CUdeviceptr p) {
  const Range* const r = find(p);
  for (unsigned int i = 0; i < n; ++i) {
    if (what[i] == CU_POINTER_ATTRIBUTE_MEMORY_TYPE) *(unsigned int*)where[i] = r ? CU_MEMORYTYPE_HOST : 0;
    if (what[i] == CU_POINTER_ATTRIBUTE_DEVICE_POINTER) *(CUdeviceptr*)where[i] = r ? p : 0;
    if (what[i] == CU_POINTER_ATTRIBUTE_RANGE_START_ADDR) *(CUdeviceptr*)where[i] = r ? r->start : 0;
    if (what[i] == CU_POINTER_ATTRIBUTE_RANGE_SIZE) *(size_t*)where[i] = r ? r->size : 0;
  }
  return CUDA_SUCCESS;
}
static cudaError_t fake_entry_point(const char* name, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  const bool known = strcmp(name, "cuPointerGetAttributes") == 0;
  *fn = known ? (void*)fake_attributes : nullptr;
  *q = known ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
static cudaError_t fake_runtime_attributes(cudaPointerAttributes* a, const void* p) {
  const bool pinned = find((uintptr_t)p) != nullptr;
  memset(a, 0, sizeof *a);
  a->type = pinned ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  a->devicePointer = pinned ? const_cast<void*>(p) : nullptr;
  return cudaSuccess;
}
#define cudaGetDriverEntryPoint fake_entry_point
#define cudaPointerGetAttributes fake_runtime_attributes
#include "kmq_host_copy.cu"

int main() {
  unsigned long long p, bytes;
  while (scanf("%llx %llu", &p, &bytes) == 2) printf("%llx\n", (unsigned long long)(uintptr_t)kmq::host_copy_address((void*)p, bytes));
}
"""

CASES = [
    (0x100000, 8192, True),             # the whole range
    (0x100010, 8176, True),             # up to its last byte
    (0x101ff0, 16, True),
    (0x100000, 8194, False),            # two bytes past its end
    (0x101ff0, 18, False),
    (0x100000, 0x4000, False),          # first and last byte pinned, the page between the ranges not
    (0x0ffff0, 32, False),              # begins before the range
    (0x102000, 16, False),              # pageable
    (0x100008, 16, False),              # not on a 16-byte boundary
    (0x103000, 4096, True),
]


@pytest.fixture(scope="module")
def answers(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_copy")
    src, exe = d / "harness.cu", d / "harness"
    src.write_text(HARNESS)
    subprocess.run([kb._nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", kb.CSRC, "-I",
                    os.path.join(kb.ROOT, "include"), str(src), "-o", str(exe)], check=True, capture_output=True)
    text = "".join(f"{p:x} {n}\n" for p, n, _ in CASES)
    out = subprocess.run([str(exe)], input=text, check=True, capture_output=True, text=True).stdout
    return [int(line, 16) for line in out.split()]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_only_buffers_inside_one_pinned_range(answers, i):
    address, _, inside = CASES[i]
    assert answers[i] == (address if inside else 0)
