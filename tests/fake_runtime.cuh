// A stand-in for the CUDA runtime calls that the library's host code makes around its
// launches, so that a host check can include a .cu file and drive that code without a GPU:
// devices with multiprocessor counts of their own, recorded attributes and memory calls,
// errors on demand.  (The <<< >>> launches themselves go to the real runtime, which must
// see no device: main starts with no_real_device().)
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <vector>

namespace fake {

inline int device = 0;                               // current device
inline std::vector<int> sm_of_device = {152, 132};   // multiprocessors
inline cudaError_t last_error = cudaSuccess;         // what cudaGetLastError returns (once)
inline cudaError_t launch_error = cudaSuccess;       // what cudaLaunchKernelEx returns
inline std::set<std::pair<const void*, int>> smem_set;   // (kernel, device) with its shared-memory limit raised
inline bool launched_unset = false;                  // a launch over 48 KB on a device without the limit
inline unsigned grid = 0;                            // of the last cudaLaunchKernelEx
struct Set {
    void* p;
    size_t bytes;
};
inline std::vector<Set> sets;                        // cudaMemsetAsync calls

inline size_t live_bytes = 0;                        // device memory held
inline std::map<void*, size_t> blocks;

inline void no_real_device() {
    int n = 0;
    if (cudaGetDeviceCount(&n) == cudaSuccess && n > 0) {
        printf("a GPU is visible: run with CUDA_VISIBLE_DEVICES=\n");
        exit(2);
    }
    (void)cudaGetLastError();
}

inline cudaError_t get_device(int* d) {
    *d = device;
    return cudaSuccess;
}
inline cudaError_t get_attribute(int* v, cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrMultiProcessorCount ? sm_of_device[d] : 0;
    return cudaSuccess;
}
template <class F>
cudaError_t func_set_attribute(F* f, cudaFuncAttribute a, int) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_set.insert({(const void*)f, device});
    return cudaSuccess;
}
template <class F>
cudaError_t occupancy(int* n, F*, int, size_t) {
    *n = 4;
    return cudaSuccess;
}
inline cudaError_t get_last_error() {
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
template <class... A, class... B>
cudaError_t launch_ex(const cudaLaunchConfig_t* c, void (*f)(A...), B&&...) {
    grid = c->gridDim.x;
    if (c->dynamicSmemBytes > 48 * 1024 && !smem_set.count({(const void*)f, device})) launched_unset = true;
    return launch_error;
}
inline cudaError_t memset_async(void* p, int, size_t n, cudaStream_t) {
    sets.push_back({p, n});
    return cudaSuccess;
}

// device memory is host memory, so that copies work; its bytes are counted
template <class T>
cudaError_t device_malloc(T** p, size_t n) {
    *p = (T*)calloc(n ? n : 1, 1);
    blocks[(void*)*p] = n;
    live_bytes += n;
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
inline cudaError_t device_free(void* p) {
    auto b = blocks.find(p);
    if (b == blocks.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
    live_bytes -= b->second;
    blocks.erase(b);
    free(p);
    return cudaSuccess;
}
template <class T>
cudaError_t host_malloc(T** p, size_t n) {
    *p = (T*)calloc(n, 1);
    return cudaSuccess;
}
inline cudaError_t host_free(void* p) {
    free(p);
    return cudaSuccess;
}
inline cudaError_t copy_async(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    memcpy(d, s, n);
    return cudaSuccess;
}

// cudaMemset returns before the fill: unsettled until the host has waited for the stream or device
inline int unsettled = 0;
inline cudaError_t copy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    memcpy(d, s, n);
    return cudaSuccess;
}
// every other call succeeds; handles are numbered
inline size_t handles = 0;
template <class H, class... A>
cudaError_t make_handle(H* h, A...) {
    *h = (H)(uintptr_t)++handles;
    return cudaSuccess;
}
template <class S, class H>
cudaError_t make_second(S, H* h) {
    return make_handle(h);
}
template <class... A>
cudaError_t done(A...) {
    return cudaSuccess;
}
inline cudaError_t priority_range(int* least, int* greatest) {
    *least = *greatest = 0;
    return cudaSuccess;
}
inline float elapsed_ms = 1.f;   // what every pair of events is apart
inline cudaError_t elapsed(float* t, cudaEvent_t, cudaEvent_t) {
    *t = elapsed_ms;
    return cudaSuccess;
}
inline cudaError_t set_bytes(void* p, int v, size_t n) {
    memset(p, v, n);
    ++unsettled;
    return cudaSuccess;
}
inline cudaError_t stream_synchronize(cudaStream_t st) {
    if (st == nullptr || st == cudaStreamLegacy) unsettled = 0;
    return cudaSuccess;
}
inline cudaError_t device_synchronize() {
    unsettled = 0;
    return cudaSuccess;
}

}  // namespace fake

#define cudaGetDevice fake::get_device
#define cudaDeviceGetAttribute fake::get_attribute
#define cudaFuncSetAttribute fake::func_set_attribute
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake::occupancy
#define cudaGetLastError fake::get_last_error
#define cudaLaunchKernelEx fake::launch_ex
#define cudaMemsetAsync fake::memset_async
#define cudaMalloc fake::device_malloc
#define cudaFree fake::device_free
#define cudaMallocHost fake::host_malloc
#define cudaFreeHost fake::host_free
#define cudaMemcpyAsync fake::copy_async
#define cudaMemcpy fake::copy
#define cudaMemset fake::set_bytes
#define cudaSetDevice fake::done
#define cudaDeviceSynchronize fake::device_synchronize
#define cudaStreamSynchronize fake::stream_synchronize
#define cudaStreamCreateWithFlags fake::make_handle
#define cudaStreamCreateWithPriority fake::make_handle
#define cudaStreamDestroy fake::done
#define cudaStreamBeginCapture fake::done
#define cudaStreamEndCapture fake::make_second
#define cudaDeviceGetStreamPriorityRange fake::priority_range
#define cudaEventCreate fake::make_handle
#define cudaEventCreateWithFlags fake::make_handle
#define cudaEventDestroy fake::done
#define cudaEventRecord fake::done
#define cudaEventSynchronize fake::done
#define cudaEventElapsedTime fake::elapsed
#define cudaGraphInstantiate fake::make_handle
#define cudaGraphDestroy fake::done
#define cudaGraphExecDestroy fake::done
#define cudaGraphLaunch fake::done
