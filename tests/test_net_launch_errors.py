"""The host side of the network's kernels against a fake of the CUDA runtime (no GPU).

The library's object file is linked with a runtime that records launches and
attributes, and fails the launch it is told to: what the host does then is what it
would do with the real one.
"""
import ctypes
import os
import subprocess

import pytest

from paper_1702_01530_gb300 import build

FAKE = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <map>
#include <utility>
#include "rt_internal.cuh"

static int g_launches, g_fail_at, g_device;
static cudaError_t g_last;
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

namespace rt { int num_sms() { return 152; } }

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
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

static void* at(size_t i) { return reinterpret_cast<void*>(4096 * (i + 1)); }
void fake_begin(int device, int fail_at) { g_device = device; g_fail_at = fail_at; g_launches = 0; }
int fake_launches() { return g_launches; }
int fake_train(unsigned W, unsigned H) {
  rt::nn::TrainBuffers t = {};
  size_t i = 0;
  t.params = (float*)at(i++); t.m = (float*)at(i++); t.v = (float*)at(i++);
  for (int l = 0; l < 4; ++l) { t.wf[l] = (__nv_bfloat16*)at(i++); t.wb[l] = (__nv_bfloat16*)at(i++); }
  for (int l = 0; l < 3; ++l) { t.act[l] = (__nv_bfloat16*)at(i++); t.dz[l] = (__nv_bfloat16*)at(i++); }
  t.g8 = (__nv_bfloat16*)at(i++); t.mask = (uint32_t*)at(i++);
  t.wpart = (float*)at(i++); t.loss_part = (float*)at(i++); t.loss = (float*)at(i++);
  return rt::nn::train_step((__nv_bfloat16*)at(i), (float*)at(i + 1), t, W, H, 1e-3f, 1u, nullptr, (uint32_t*)at(i + 2), 0);
}
int fake_forward(int fp8, unsigned W, unsigned H) {
  __nv_bfloat16* wf[4];
  uint8_t* w8[3];
  float* inv[3];
  const float scale[3] = {1.f, 1.f, 1.f};
  for (int l = 0; l < 4; ++l) wf[l] = (__nv_bfloat16*)at(l);
  for (int l = 0; l < 3; ++l) { w8[l] = (uint8_t*)at(4 + l); inv[l] = (float*)at(7 + l); }
  __nv_bfloat16* feat = (__nv_bfloat16*)at(10);
  float *params = (float*)at(11), *prob = (float*)at(12);
  uint32_t* err = (uint32_t*)at(13);
  if (fp8) return rt::nn::forward_fp8(feat, params, wf, w8, inv, scale, prob, W, H, err, 0, 1);
  return rt::nn::forward(feat, params, wf, nullptr, prob, W, H, err, 0, 1);
}
}
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    build.build()
    obj = os.path.join(build.OUT_DIR, "nn.o")
    if not os.path.exists(obj):
        build.build(force=True)
    d = tmp_path_factory.mktemp("fake")
    src, lib = str(d / "fake.cpp"), str(d / "libfake.so")
    with open(src, "w") as f:
        f.write(FAKE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-I", build.CSRC,
                    "-I", build.INCLUDE, src, obj, "-o", lib], check=True, capture_output=True)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("W,H", [(960, 540), (33, 9)])
def test_a_step_ends_at_its_first_failed_launch(fake, W, H):
    fake.fake_begin(0, -1)
    assert fake.fake_train(W, H) == 0
    steps = fake.fake_launches()
    assert steps == 4
    for at in range(steps):
        fake.fake_begin(0, at)
        assert fake.fake_train(W, H) == 701          # cudaErrorLaunchOutOfResources
        assert fake.fake_launches() == at + 1, "a kernel was launched on what the failed one did not make"
        fake.fake_begin(0, -1)
        assert fake.fake_train(W, H) == 0, "the failure is reported once"


@pytest.mark.parametrize("W,H", [(960, 540), (33, 9)])     # either weight-gradient kernel
def test_a_second_device_allows_the_shared_memory_too(fake, W, H):
    for device in (0, 1, 0, 2):
        fake.fake_begin(device, -1)
        assert fake.fake_forward(0, W, H) == 0, device
        assert fake.fake_forward(1, W, H) == 0, device
        assert fake.fake_train(W, H) == 0, device
