"""A fake of the CUDA runtime to link the library's object files with (test infrastructure
only): it records launches and shared-memory attributes and fails the launch it is told
to, so what the host side does after an error runs without a GPU and without a fault.
"""
import ctypes
import os
import subprocess

from paper_1702_01530_gb300 import build

LAUNCH_ERROR = 701          # cudaErrorLaunchOutOfResources

_COMMON = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <map>
#include <utility>
#include "rt_internal.cuh"

static int g_launches, g_fail_at, g_device;
static cudaError_t g_last;
static unsigned g_word[16];
static std::map<std::pair<int, const void*>, int> g_smem;     // dynamic shared memory allowed, by device and kernel

static cudaError_t launch(const void* kernel, size_t smem) {
  const int at = g_launches++;
  const auto it = g_smem.find({g_device, kernel});
  const size_t most = it == g_smem.end() ? 48u * 1024u : (size_t)it->second;
  const cudaError_t e = at == g_fail_at ? cudaErrorLaunchOutOfResources : smem > most ? cudaErrorInvalidValue : cudaSuccess;
  if (e != cudaSuccess) g_last = e;
  return e;
}
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void*) { *smem = 0; return cudaSuccess; }
cudaError_t __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void* k, dim3, dim3, void**, size_t smem, cudaStream_t) { return launch(k, smem); }
cudaError_t CUDARTAPI cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->dynamicSmemBytes);
}
cudaError_t CUDARTAPI cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = v;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
cudaError_t CUDARTAPI cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                                       cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t CUDARTAPI cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t CUDARTAPI cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* b, const void*, int, size_t, unsigned) {
  *b = 9;
  return cudaSuccess;
}
cudaError_t CUDARTAPI cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
// a download brings words of g_word
cudaError_t CUDARTAPI cudaMemcpyAsync(void* to, const void*, size_t n, cudaMemcpyKind k, cudaStream_t) {
  if (k == cudaMemcpyDeviceToHost)
    for (size_t i = 0; i < n / 4; ++i) static_cast<unsigned*>(to)[i] = g_word[i];
  return cudaSuccess;
}
static void* at(size_t i) { return reinterpret_cast<void*>(4096 * (i + 1)); }
void fake_begin(int device, int fail_at) { g_device = device; g_fail_at = fail_at; g_launches = 0; }
int fake_launches() { return g_launches; }
"""


def load(tmp, objects, entry):
    """The named object files and the C++ text ``entry`` (inside extern "C") as a library:
    fake_begin(device, launch to fail or -1) and fake_launches() besides its own functions."""
    build.build()
    objs = [os.path.join(build.OUT_DIR, o) for o in objects]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    src, lib = str(tmp / "fake.cpp"), str(tmp / "libfake.so")
    with open(src, "w") as f:
        f.write(_COMMON + entry + "}\n")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-I", build.CSRC,
                    "-I", build.INCLUDE, src, *objs, "-o", lib], check=True, capture_output=True)
    return ctypes.CDLL(lib)
