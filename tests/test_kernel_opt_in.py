"""Opt-ins of a kernel belong to one device: launches of one process on several devices, and a launch after a
failed opt-in.  The translation unit of the projections is linked with a stand-in for the CUDA runtime
that keeps each device's limit on dynamic shared memory and refuses launches above it, as the runtime
does; no GPU is used."""
import ctypes
import os
import subprocess

import pytest

from paper_2508_13867_gb300 import build

FAKE = r"""
#include <cuda_runtime.h>
#include <map>
#include <utility>
#include "uqlb_internal.h"
static int device = 0, fail_next = 0, launches = 0;
static std::map<std::pair<int, const void*>, size_t> limit;
extern "C" {
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (fail_next) { fail_next = 0; return cudaErrorInvalidDevice; }
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[{device, f}] = (size_t)v;
    return cudaSuccess;
}
static cudaError_t last = cudaSuccess;
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t) { return ""; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static dim3 g_, b_;
static size_t s_;
static void* st_;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) { g_ = g; b_ = b; s_ = s; st_ = st; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
    *g = g_; *b = b_; *s = s_; *(void**)st = st_; return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
static cudaError_t launch(const void* f, size_t smem) {
    const auto it = limit.find({device, f});
    last = smem <= (it == limit.end() ? 48u * 1024u : it->second) ? cudaSuccess : cudaErrorInvalidValue;
    launches += last == cudaSuccess;
    return last;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
    return launch((const void*)k, smem);
}
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) { return launch(f, smem); }

// one reflected projection of K terms on `dev`; the status of its launch
int reflect_on(int dev, int fail, int dtype, int K, int max_m) {
    cudaSetDevice(dev);
    fail_next = fail;
    const uqlb::ReflPlanView v{nullptr, nullptr, nullptr, 1, max_m};
    const int rc = uqlb::launch_reflect(v, K, nullptr, dtype, 100, 100, nullptr, nullptr);
    fail_next = 0;
    return rc;
}
}
namespace uqlb {
int ctx_fail(uqlb_ctx*, int s, const char*) { return s; }
int ctx_projection_view(uqlb_ctx*, const double**, int*, int64_t*, int*) { return 1; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("optin"))
    with open(os.path.join(d, "fake.cpp"), "w") as f:
        f.write(FAKE)
    out = os.path.join(d, "fake.so")
    inc = ["-I", build.INCLUDE, "-I", build.CSRC]
    obj = os.path.join(d, "p.o")
    for cmd in ([build.nvcc(), "-std=c++17", "-O1", "-Xcompiler", "-fPIC", *build.ARCH, "--expt-relaxed-constexpr", *inc,
                 "-c", os.path.join(build.CSRC, "project_kernels.cu"), "-o", obj],
                [build.nvcc(), "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", *inc,
                 os.path.join(d, "fake.cpp"), obj, "-o", out]):
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
    return ctypes.CDLL(out)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("K,max_m", [(35, 4), (112, 4), (10, 2)])
def test_reflected_projection_on_several_devices(lib, dtype, K, max_m):
    """The 137-point grid's 35 terms take 51 KB per block, 112 terms the most of the plan (128 KB)."""
    lib.reflect_on(0, 1, dtype, K, max_m)  # a failed opt-in is not kept
    for dev in (0, 1, 0, 2):
        assert lib.reflect_on(dev, 0, dtype, K, max_m) == 0, dev
