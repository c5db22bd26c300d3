// Host emulation of the CUDA features that the decoder's sources use, so that
// its kernels can be run and checked on a CPU.  Tests only.
//
// Every thread of a block is a fiber; the blocks of a launch run one after the
// other.  A lane runs until it reaches a warp or block wide operation and waits
// there for the others, so between two such operations lanes run in any order
// that the test asks for (emu_order), one far ahead of the other if need be: what
// holds on hardware only while a warp happens to be converged fails here.
#pragma once

#include <climits>
#include <cstddef>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <functional>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))
#define __launch_bounds__(...)
#define __grid_constant__
#define __shared__ static   // blocks run one at a time
#define __align__(n) __attribute__((aligned(n)))

struct dim3 { unsigned x = 1, y = 1, z = 1; };
struct int2 { int x, y; } __align__(8);
struct int4 { int x, y, z, w; } __align__(16);
struct uint4 { unsigned x, y, z, w; } __align__(16);
inline int2 make_int2(int x, int y) { return int2{x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return int4{x, y, z, w}; }
inline uint4 make_uint4(unsigned x, unsigned y, unsigned z, unsigned w) { return uint4{x, y, z, w}; }

namespace emu {
extern dim3 thread_idx, block_idx, block_dim, grid_dim;
extern int sms, syncs, fail_alloc;
char *dynamic_shared();
unsigned long long now_ns();
// warp wide: every lane's value, once all lanes of the mask are here
const unsigned long long *exchange(unsigned mask, unsigned long long v);
int lane();
int block_or(int v);   // block wide barrier
void launch(long long grid, int block, size_t smem, const std::function<void()> &kernel);
inline void launch(long long grid, int block, const std::function<void()> &kernel) { launch(grid, block, 0, kernel); }
inline void launch(long long grid, int block, size_t smem, void *, const std::function<void()> &kernel) { launch(grid, block, smem, kernel); }
template <class T> T reduce(unsigned m, T v, T (*f)(T, T)) {
    const unsigned long long *x = exchange(m, (unsigned long long)(unsigned)v);
    bool any = false;
    T r = v;
    for (int l = 0; l < 32; l++)
        if ((m >> l) & 1u) { r = any ? f(r, (T)(unsigned)x[l]) : (T)(unsigned)x[l]; any = true; }
    return r;
}
}  // namespace emu

#define threadIdx (emu::thread_idx)
#define blockIdx (emu::block_idx)
#define blockDim (emu::block_dim)
#define gridDim (emu::grid_dim)

template <class T> T __ldg(const T *p) { return *p; }
inline int __popc(unsigned v) { return __builtin_popcount(v); }
inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
inline unsigned __activemask() { return 1u << emu::lane(); }
inline void __syncwarp(unsigned m = 0xffffffffu) { emu::exchange(m, 0); }
inline void __syncthreads() { emu::block_or(0); }
inline int __syncthreads_or(int v) { return emu::block_or(v); }
inline void __threadfence_block() {}
inline void __threadfence_system() { __atomic_thread_fence(__ATOMIC_SEQ_CST); }
template <class T> T __shfl_sync(unsigned m, T v, int src) { return (T)emu::exchange(m, (unsigned long long)v)[src & 31]; }
template <class T> T __shfl_up_sync(unsigned m, T v, int d) {
    const unsigned long long *x = emu::exchange(m, (unsigned long long)v);
    return emu::lane() >= d ? (T)x[emu::lane() - d] : v;
}
template <class T> T __shfl_xor_sync(unsigned m, T v, int d) { return (T)emu::exchange(m, (unsigned long long)v)[emu::lane() ^ d]; }
inline unsigned __ballot_sync(unsigned m, int p) {
    const unsigned long long *x = emu::exchange(m, p != 0);
    unsigned r = 0;
    for (int l = 0; l < 32; l++)
        if (((m >> l) & 1u) && x[l]) r |= 1u << l;
    return r;
}
inline int __any_sync(unsigned m, int p) { return __ballot_sync(m, p) != 0; }
inline unsigned __reduce_add_sync(unsigned m, unsigned v) { return emu::reduce<unsigned>(m, v, [](unsigned a, unsigned b) { return a + b; }); }
inline unsigned __reduce_min_sync(unsigned m, unsigned v) { return emu::reduce<unsigned>(m, v, [](unsigned a, unsigned b) { return a < b ? a : b; }); }
inline int __reduce_min_sync(unsigned m, int v) { return emu::reduce<int>(m, v, [](int a, int b) { return a < b ? a : b; }); }
inline unsigned __reduce_max_sync(unsigned m, unsigned v) { return emu::reduce<unsigned>(m, v, [](unsigned a, unsigned b) { return a > b ? a : b; }); }
inline int __reduce_max_sync(unsigned m, int v) { return emu::reduce<int>(m, v, [](int a, int b) { return a > b ? a : b; }); }
inline unsigned __reduce_or_sync(unsigned m, unsigned v) { return emu::reduce<unsigned>(m, v, [](unsigned a, unsigned b) { return a | b; }); }
inline unsigned __reduce_xor_sync(unsigned m, unsigned v) { return emu::reduce<unsigned>(m, v, [](unsigned a, unsigned b) { return a ^ b; }); }

template <class T, class U> T atomicAdd(T *p, U v) { T o = *p; *p = (T)(o + (T)v); return o; }
template <class T, class U> T atomicMin(T *p, U v) { T o = *p; if ((T)v < o) *p = (T)v; return o; }
template <class T, class U> T atomicOr(T *p, U v) { T o = *p; *p = o | (T)v; return o; }
template <class T, class U> T atomicAnd(T *p, U v) { T o = *p; *p = o & (T)v; return o; }
template <class T, class U> T atomicXor(T *p, U v) { T o = *p; *p = o ^ (T)v; return o; }
template <class T> T atomicCAS(T *p, T c, T v) { T o = *p; if (o == c) *p = v; return o; }
using std::max;
using std::min;

// ---- runtime calls: one device, every call done when it returns
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2, cudaErrorNotReady = 600 };
typedef void *cudaStream_t;
typedef void *cudaEvent_t;
enum cudaStreamCaptureStatus { cudaStreamCaptureStatusNone = 0 };
enum { cudaMemcpyHostToDevice, cudaMemcpyDeviceToHost, cudaHostAllocDefault, cudaHostAllocMapped, cudaEventDisableTiming,
       cudaStreamNonBlocking, cudaDevAttrMultiProcessorCount, cudaFuncAttributeMaxDynamicSharedMemorySize };
struct cudaFuncAttributes { int maxThreadsPerBlock; };
template <class T> cudaError_t cudaMalloc(T **p, size_t n) {
    if (emu::fail_alloc > 0 && --emu::fail_alloc == 0) return cudaErrorMemoryAllocation;
    *p = (T *)aligned_alloc(256, (n + 256) / 256 * 256);
    if (!*p) return cudaErrorMemoryAllocation;
    if (n < (1u << 20)) memset(*p, 0xa5, n);
    return cudaSuccess;
}
template <class T> cudaError_t cudaHostAlloc(T **p, size_t n, int) { return cudaMalloc(p, n); }
inline cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
inline cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
inline cudaError_t cudaHostGetDevicePointer(void **d, void *h, int) { *d = h; return cudaSuccess; }
inline cudaError_t cudaMemcpy(void *d, const void *s, size_t n, int) { memcpy(d, s, n); return cudaSuccess; }
inline cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, int, cudaStream_t = nullptr) { memcpy(d, s, n); return cudaSuccess; }
inline cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
inline cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t = nullptr) { memset(d, v, n); return cudaSuccess; }
template <class T> cudaError_t cudaGetSymbolAddress(void **p, T &s) { *p = (void *)&s; return cudaSuccess; }
inline cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
inline cudaError_t cudaSetDevice(int) { return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int *v, int, int) { *v = emu::sms; return cudaSuccess; }
inline cudaError_t cudaDeviceSynchronize() { emu::syncs++; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline const char *cudaGetErrorString(cudaError_t) { return "error"; }
inline cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, int) { *e = (void *)1; return cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
inline cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
inline cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t = nullptr) { return cudaSuccess; }
inline cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, int) { *s = (void *)1; return cudaSuccess; }
inline cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) { *s = cudaStreamCaptureStatusNone; return cudaSuccess; }
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, int) { return cudaSuccess; }
template <class F> cudaError_t cudaFuncSetAttribute(F *, int, int) { return cudaSuccess; }
template <class F> cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, F *) { a->maxThreadsPerBlock = 1024; return cudaSuccess; }
template <class F> cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, F *, int, size_t) { *n = 1; return cudaSuccess; }
