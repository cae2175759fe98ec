// A stand-in for the CUDA runtime that keeps one thing: how much dynamic shared
// memory each kernel may ask for on each device (48 KB until a function
// attribute says more), and refuses a launch beyond it, as the runtime does.
#include "fake_cudart.h"

#include <cstring>
#include <map>
#include <utility>

#include <cuda_runtime_api.h>

int g_device = 0;
int g_fail_attributes = 0;
void (*g_meanwhile)() = nullptr;
int g_launched = 0;
size_t g_last_smem = 0;
unsigned g_last_blocks = 0;
int g_splits = 0;

namespace {
cudaError_t g_last = cudaSuccess;

std::map<std::pair<const void*, int>, int> g_limit;   // (kernel, device) -> bytes allowed
cudaError_t launch(const void* kernel, dim3 grid, size_t smem) {
    const auto it = g_limit.find({kernel, g_device});
    if (smem > size_t(it == g_limit.end() ? 48 * 1024 : it->second)) return g_last = cudaErrorInvalidValue;
    g_launched++;
    g_last_smem = smem;
    g_last_blocks = grid.x * grid.y;
    return cudaSuccess;
}

dim3 g_grid, g_block;
size_t g_smem;
cudaStream_t g_stream;
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount                ? 152
         : a == cudaDevAttrMaxSharedMemoryPerBlockOptin       ? 227 * 1024
         : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 228 * 1024
                                                              : 0;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* kernel, cudaFuncAttribute a, int v) {
    if (g_fail_attributes > 0) {
        g_fail_attributes--;
        return cudaErrorMemoryAllocation;
    }
    if (a == cudaFuncAttributePreferredSharedMemoryCarveout) g_splits++;
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
        g_limit[{kernel, g_device}] = v;
        if (void (*other)() = g_meanwhile) {
            g_meanwhile = nullptr;
            other();
        }
    }
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* kernel, void**) {
    return launch(kernel, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    memcpy(k, &f, sizeof f);
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t smem, cudaStream_t) {
    return launch(reinterpret_cast<const void*>(k), grid, smem);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
    g_grid = g, g_block = b, g_smem = smem, g_stream = s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = g_grid, *b = g_block, *smem = g_smem, *static_cast<cudaStream_t*>(s) = g_stream;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
}
