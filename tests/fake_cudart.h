// fake_cudart.h -- a CUDA runtime for host-side checks without a GPU: the
// library's own objects are linked against it in place of cudart.  Kernels do
// nothing but are recorded by name; device memory is host memory.  A copy from
// pageable host memory reads its source at the next synchronisation, the
// latest moment the runtime's contract allows; a source that is freed
// before that is counted.
#pragma once

#include <cuda_runtime.h>
#include <malloc.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

namespace fake {

struct Copy {
    void *dst;
    const void *src;
    size_t bytes;
};
constexpr int kMaxPending = 64;
inline Copy pending[kMaxPending];
inline int npending = 0;
inline int freed_sources = 0;      // sources of pending copies given back to the heap
inline int sms = 152;              // multiprocessors of the device
inline const char *fail_launch = nullptr;  // launches of kernels whose name holds this fail
inline int fail_attribute = 0;     // cudaFuncSetAttribute fails
inline int capturing = 0;          // streams are being captured
inline int ctas_per_sm = 2;        // occupancy of any kernel
inline unsigned grid = 0;          // CTAs of the last cudaLaunchKernelEx
inline int copies = 0;             // copies from host memory
inline int clusters = 1;           // clusters of any size that the device can hold
inline cudaError_t last = cudaSuccess;
inline std::map<const void *, std::string> &names() {
    static std::map<const void *, std::string> m;
    return m;
}
inline std::vector<std::string> &launches() {  // names of the kernels launched
    static std::vector<std::string> v;
    return v;
}
inline std::vector<void *> &pinned() {
    static std::vector<void *> v;
    return v;
}
inline int launched(const char *part) {
    int k = 0;
    for (const std::string &s : launches()) k += s.find(part) != std::string::npos;
    return k;
}
inline cudaError_t launch(const void *f) {
    const std::string &n = names()[f];
    if (fail_launch && n.find(fail_launch) != std::string::npos) return last = cudaErrorLaunchOutOfResources;
    launches().push_back(n);
    return cudaSuccess;
}
inline void run_copies() {
    for (int i = 0; i < npending; ++i) std::memcpy(pending[i].dst, pending[i].src, pending[i].bytes);
    npending = 0;
}
inline void check_free(void *p) {
    const char *b = (const char *)p;
    const size_t n = p ? malloc_usable_size(p) : 0;
    for (int i = 0; i < npending; ++i)
        if (b < (const char *)pending[i].src + pending[i].bytes && (const char *)pending[i].src < b + n) ++freed_sources;
}

}  // namespace fake

void *operator new(size_t n) {
    void *p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void *p) noexcept {
    fake::check_free(p);
    std::free(p);
}
void operator delete(void *p, size_t) noexcept { operator delete(p); }

extern "C" {

void **__cudaRegisterFatBinary(void *) {
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
    fake::names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) {
    *g = *b = dim3(1);
    *s = 0;
    *(cudaStream_t *)st = nullptr;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t, cudaStream_t) {
    return fake::launch((const void *)k);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) {
    fake::grid = c->gridDim.x;
    return fake::launch(f);
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = fake::last;
    fake::last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) {
    return fake::fail_attribute ? fake::last = cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    *a = cudaFuncAttributes{};
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) {
    *p = (void *)s;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = aligned_alloc(256, (n + 255) & ~(size_t)255);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void **p, size_t n) {
    *p = std::calloc(n, 1);
    fake::pinned().push_back(*p);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFreeHost(void *p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t) {
    fake::copies += kind == cudaMemcpyHostToDevice;
    if (kind == cudaMemcpyHostToDevice && fake::npending < fake::kMaxPending) {
        fake::pending[fake::npending++] = fake::Copy{dst, src, n};
        return cudaSuccess;
    }
    fake::run_copies();
    std::memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
    fake::run_copies();
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
    fake::run_copies();
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? fake::sms : 0;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    return *n = fake::ctas_per_sm, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
    return *n = fake::clusters, cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    *st = fake::capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *, cudaGraph_t, unsigned long long) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

}  // extern "C"
