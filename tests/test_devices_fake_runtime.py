"""Two devices in one process, on the CPU: the library's own objects linked against a
stand-in for the CUDA runtime that, like the real one, keeps a kernel's shared-memory
limit per device and refuses a launch above it.  Nothing runs; what is checked is
which limits the host code has raised, for how many SMs it sizes a grid, and whose
status word it reads, on the device that a call is made on."""
import glob
import os
import shutil
import subprocess

import pytest

from paper_2407_11698_gb300 import binding as nb
from paper_2407_11698_gb300 import build as nbuild

FAKE = r'''
#include <cuda.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <utility>
#include "nitro.h"

static int g_dev = 0, g_launches = 0, g_refused = 0, g_most_ctas = 0;
static cudaError_t g_error = cudaSuccess;
static const int kSms[2] = {152, 20};
static std::map<std::pair<int, const void*>, int> g_limit;      // device, kernel
static uint32_t* g_symbol[2];      // the library array looked up last on each device: the noalloc words

static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                       const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int d) { *v = kSms[d]; return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
    memset(a, 0, sizeof(*a));
    a->maxThreadsPerBlock = 1024;
    a->numRegs = 96;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
    g_limit[{g_dev, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    ++g_launches;
    const auto it = g_limit.find({g_dev, f});
    const int limit = it == g_limit.end() ? 48 * 1024 : it->second;
    if ((int)c->dynamicSmemBytes > limit) { ++g_refused; return g_error = cudaErrorInvalidValue; }
    if (c->dynamicSmemBytes > 48 * 1024 && (int)c->gridDim.x > g_most_ctas) g_most_ctas = (int)c->gridDim.x;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = g_symbol[g_dev] = static_cast<uint32_t*>(calloc(1, 1 << 24));
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *p = reinterpret_cast<void*>(&encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_error;
    g_error = cudaSuccess;
    return e;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float*, cudaEvent_t, cudaEvent_t) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void**, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void*, dim3, dim3, void**, size_t, void*) { return cudaSuccess; }
}

int main() {
    static char buf[64];
    for (g_dev = 0; g_dev < 2; ++g_dev) {
        g_launches = g_refused = g_most_ctas = 0;
        // 64 channels in (no im2col), 3 (im2col), and a few tiles with a long K (cluster)
        const int shapes[3][4] = {{16, 64, 128, 64}, {16, 3, 64, 64}, {1, 512, 512, 4}};
        int st = 0;
        for (const auto& q : shapes)
            st |= nitro_conv3x3_forward_noalloc(reinterpret_cast<int8_t*>(buf), reinterpret_cast<int32_t*>(buf), q[0],
                                                q[3] == 64 ? 16 : 4, q[3] == 64 ? 16 : 4, q[1], q[2], 0, 10,
                                                reinterpret_cast<int8_t*>(buf), reinterpret_cast<int8_t*>(buf), nullptr,
                                                nullptr);
        nitro_gemm* g = nullptr;
        st |= nitro_gemm_create(16384, 256, 256, &g);
        if (g) {
            st |= nitro_gemm_run(g, reinterpret_cast<int8_t*>(buf), reinterpret_cast<int32_t*>(buf), 16384, 256, 256,
                                 reinterpret_cast<int64_t*>(buf), nullptr);
            nitro_gemm_destroy(g);
        }
        printf("%d %d %d %d %d\n", g_dev, st, g_launches, g_refused, g_most_ctas);
    }
    // a wait that ran out on the second device: the kernel sets the TIMEOUT bit of words[3]
    g_symbol[1][3] = NITRO_STATUS_BIT_TIMEOUT;
    for (g_dev = 0; g_dev < 2; ++g_dev)
        for (int clear : {0, 1, 0}) printf("%d ", (int)nitro_conv3x3_noalloc_status(clear));
    printf("\n");
    return 0;
}
'''


def test_calls_on_a_second_device(tmp_path):
    cxx = shutil.which("g++")
    include = os.path.join(os.path.dirname(os.path.dirname(nbuild.nvcc())), "include")
    if not cxx or not os.path.exists(os.path.join(include, "cuda.h")):
        pytest.skip("no host compiler or CUDA headers")
    nbuild.build()
    src, exe = tmp_path / "fake.cc", tmp_path / "fake"
    src.write_text(FAKE)
    subprocess.run([cxx, "-std=c++17", "-I", include, "-I", nbuild.INCLUDE, str(src)] +
                   sorted(glob.glob(os.path.join(nbuild.OUT_DIR, "*.o"))) + ["-o", str(exe), "-lpthread"],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == 3
    for line, sms in zip(out, (152, 20)):
        dev, st, launches, refused, ctas = map(int, line.split())
        assert st == 0 and launches > 0 and refused == 0, out
        assert ctas == sms, out                # a persistent grid: one CTA an SM of this device
    # the status of the allocation-free calls: latched, per device, cleared on request
    timeout = nb.NITRO_ERR_TIMEOUT
    assert list(map(int, out[2].split())) == [0, 0, 0, timeout, timeout, 0]
