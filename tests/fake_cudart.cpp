// A CUDA runtime of the host alone, to link the library's objects with: it records what is asked
// of it and refuses what a device would.  A kernel's attributes belong to the current device.
#include <cuda_runtime_api.h>

#include "fake_cudart.h"

#include <map>
#include <string>
#include <utility>

Fake fake;

namespace {

struct Attrs {
    int smem = 48 << 10;
    bool wide_clusters = false;
};
std::map<std::pair<int, const void*>, Attrs> attrs;
std::map<const void*, std::string> names;
cudaError_t last = cudaSuccess;
struct Config {
    dim3 grid, block;
    size_t smem;
    void* stream;
} config;

cudaError_t result(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}
cudaError_t launch(const void* f, size_t smem, unsigned int cluster, void* stream) {
    const Attrs& a = attrs[{fake.device, f}];
    if (smem > (size_t)a.smem || (cluster > 8 && !a.wide_clusters)) return result(cudaErrorInvalidValue);
    fake.launched.push_back(names[f]);
    fake.streams.push_back(stream);
    return cudaSuccess;
}

}  // namespace

extern "C" {

void** __cudaRegisterFatBinary(void*) {
    static void* handle;
    return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
    names[host] = name;
}
cudaError_t __cudaGetKernel(void** k, const void* f) {
    *k = const_cast<void*>(f);
    return cudaSuccess;
}
unsigned int __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* stream) {
    config = {g, b, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* stream) {
    *g = config.grid;
    *b = config.block;
    *smem = config.smem;
    *(void**)stream = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(void* k, dim3, dim3, void**, size_t smem, void* stream) { return launch(k, smem, 1, stream); }

cudaError_t cudaGetLastError(void) {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t cudaGetDevice(int* d) {
    *d = fake.device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (fake.refuse_attributes) return result(cudaErrorInvalidValue);
    Attrs& x = attrs[{fake.device, f}];
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) x.smem = v;
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed) x.wide_clusters = v != 0;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned int) {
    static char* next = nullptr;
    if (fake.streams_left <= 0) return result(cudaErrorMemoryAllocation);
    --fake.streams_left;
    ++fake.made;
    *s = (cudaStream_t)(next += 16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) {
    --fake.made;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) {
    ++fake.made;
    *e = (cudaEvent_t)&fake;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) {
    --fake.made;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned int) {
    fake.waits.push_back(s);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
    unsigned int cluster = 1;
    for (unsigned int i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    return launch(f, c->dynamicSmemBytes, cluster, c->stream);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t s) {
    return launch(f, smem, 1, s);
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned int) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxPotentialClusterSize(int* n, const void*, const cudaLaunchConfig_t*) {
    *n = 16;
    return cudaSuccess;
}

}  // extern "C"
