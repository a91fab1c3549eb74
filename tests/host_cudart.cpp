// Host stand-in for the CUDA runtime functions the library calls, linked with the
// library's objects by test_buffer_bounds.py: device memory is zeroed host memory,
// copies are memcpy, kernels do not run.  Every launch checks that the particle
// buffers handed to the kernel (Bufs, its first parameter) cover what the filtered
// search writes: 16 bytes to posB and to velB for every particle of a started tile
// of 8, and 32 bytes to key for every started tile.
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>

#include "kmc_internal.h"

namespace {
std::map<const void*, std::string>& names() {   // device name by kernel handle
    static std::map<const void*, std::string> m;
    return m;
}
std::map<const void*, size_t> sizes;   // allocated bytes by address
std::map<std::string, int> launches;
long shortfall;   // largest number of bytes missing
struct Config {
    dim3 grid, block;
    size_t smem;
    void* stream;
} config;

void need(const void* p, size_t bytes) {
    const auto it = sizes.find(p);
    const long missing = (long)bytes - (long)(it == sizes.end() ? 0 : it->second);
    if (missing > shortfall) shortfall = missing;
}
template <typename T>
void check(const kmc::Bufs<T>& b) {
    const size_t tiles = (size_t)(b.n + 7) / 8;
    need(b.posB, tiles * 8 * 16);
    need(b.velB, tiles * 8 * 16);
    need(b.key, tiles * 32);
}
}  // namespace

extern "C" {
long host_shortfall() {   // since the last call
    const long s = shortfall;
    shortfall = 0;
    return s;
}
int host_launches(const char* part) {
    int n = 0;
    for (const auto& l : launches)
        if (l.first.find(part) != std::string::npos) n += l.second;
    return n;
}

void** __cudaRegisterFatBinary(void*) { return (void**)&config; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* fun, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names()[fun] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, CUstream_st* s) {
    config = Config{g, b, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
    *g = config.grid;
    *b = config.block;
    *smem = config.smem;
    *(void**)s = config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
    *k = (cudaKernel_t)fun;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
    const std::string& name = names()[(const void*)k];
    ++launches[name];
    // the kernels of a state take its buffers first
    if (name.find("scatter_kernel") != std::string::npos || name.find("filter_prep") != std::string::npos) {
        if (name.find("kernelIf") != std::string::npos) check(*(const kmc::Bufs<float>*)args[0]);
        else check(*(const kmc::Bufs<double>*)args[0]);
    }
    return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t bytes) {
    *p = aligned_alloc(256, (bytes + 255) / 256 * 256);
    memset(*p, 0, bytes);
    sizes[*p] = bytes;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    sizes.erase(p);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
    memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
    *p = nullptr;
    return cudaErrorNotSupported;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "host stand-in"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = nullptr;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 0.f;
    return cudaSuccess;
}
// no graphs here: the library falls back to plain launches
cudaError_t cudaGraphCreate(cudaGraph_t*, unsigned) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams*) {
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle*, cudaGraph_t, unsigned, unsigned) {
    return cudaErrorNotSupported;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
    return cudaErrorNotSupported;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
}
