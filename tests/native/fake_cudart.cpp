// A CUDA runtime for host tests of the library's bookkeeping: device memory is
// host memory (filled with 1.0, so that solvers find finite non-zero sums),
// copies are memcpy, kernels and graphs do nothing.  Allocations are counted
// and can be made to fail; copies from or to null are counted and refused.
#include "fake_cudart.h"

#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>

FakeCuda fake;

namespace {
char handle_storage[64];
template <typename T>
cudaError_t handle(T* out) {
    *out = reinterpret_cast<T>(handle_storage);
    return cudaSuccess;
}
cudaError_t allocate(void** p, size_t bytes, int* calls, int* fail) {
    ++*calls;
    *p = nullptr;
    if (*fail > 0 && --*fail == 0) return cudaErrorMemoryAllocation;
    const size_t words = bytes / 8 + 1;
    double* d = static_cast<double*>(std::malloc(words * 8));
    for (size_t i = 0; i < words; ++i) d[i] = 1.0;
    *p = d;
    fake.live.insert(d);
    return cudaSuccess;
}
cudaError_t copy(void* dst, const void* src, size_t bytes) {
    if (!dst || !src) {
        ++fake.null_copies;
        return cudaErrorInvalidValue;
    }
    std::memmove(dst, src, bytes);
    if (fake.on_copy) fake.on_copy(dst, bytes);
    return cudaSuccess;
}
CUresult encode(CUtensorMap* m, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    std::memset(m, 0, sizeof(*m));
    return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n, &fake.device_allocs, &fake.fail_device); }
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n, &fake.host_allocs, &fake.fail_host); }
cudaError_t cudaFree(void* p) {
    fake.live.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return copy(d, s, n); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return copy(d, s, n); }
cudaError_t cudaMemset(void* p, int v, size_t n) {
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error of the host test's runtime"; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;   // asked for the number of SMs
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return handle(g); }
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return handle(g); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
    *h = 1;
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
    static cudaGraph_t body[1];
    handle(&body[0]);
    p->conditional.phGraph_out = body;
    return handle(n);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return handle(e); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
    ++fake.graph_launches;
    fake.allocs_at_graph = fake.device_allocs + fake.host_allocs;
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
    a->type = cudaMemoryTypeDevice;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
    *p = const_cast<void*>(symbol);
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *fn = reinterpret_cast<void*>(encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
// what the compiler's launch and registration code calls
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(handle_storage); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 1; }
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { return handle(k); }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
}
