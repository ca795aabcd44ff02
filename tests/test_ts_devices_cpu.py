"""The eigensolvers' A C product on several devices of one process: tallskinny.cu linked
against a stand-in CUDA runtime that keeps each device's shared-memory limit and refuses a
launch above it, as a GPU does."""
import subprocess

from paper_1602_02864_gb300 import build

RUNTIME = r"""
#include <cuda_runtime.h>
#include <map>
#include <utility>
#include "tallskinny.h"
static int device = 0, launches = 0;
static cudaError_t last = cudaSuccess;
static std::map<std::pair<int, const void*>, int> limit;      // (device, kernel) -> dynamic shared memory
static dim3 g_grid, g_block;
static size_t g_smem;
static cudaStream_t g_stream;
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, cudaStream_t s) {
    g_grid = g; g_block = b; g_smem = m; g_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
    *g = g_grid; *b = g_block; *m = g_smem; *(cudaStream_t*)s = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
    auto it = limit.find({device, (const void*)k});
    if ((int)smem > (it == limit.end() ? 48 * 1024 : it->second)) last = cudaErrorInvalidValue;
    else ++launches;
    return last;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
    return __cudaLaunchKernel((cudaKernel_t)f, g, b, a, m, s);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[{device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
}
int main() {
    for (int round = 0; round < 2; ++round)
        for (device = 0; device < 3; ++device)
            for (int q : {64, 9, 32, 64})
                if (spmm::ts_nn(nullptr, 64, 64, nullptr, q, nullptr, 64, 1000, 1.0, 0.0, 0) != cudaSuccess) return 1;
    return launches == 2 * 3 * 4 ? 0 : 2;
}
"""


def test_shared_memory_limit_is_set_on_every_device(tmp_path):
    main = tmp_path / "main.cpp"
    main.write_text(RUNTIME)
    obj, exe = tmp_path / "ts.o", tmp_path / "main"
    cc = build.nvcc()
    subprocess.check_call([cc, *build.ARCH, *build.NVCC_FLAGS, "-c", f"{build.CSRC}/tallskinny.cu", "-o", str(obj)])
    subprocess.check_call([cc, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-cudart", "none", str(main), str(obj),
                           "-o", str(exe)])
    assert subprocess.run([str(exe)]).returncode == 0
