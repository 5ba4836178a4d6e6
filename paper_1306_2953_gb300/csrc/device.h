// Device-side helpers shared by the CUDA translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "common.h"

#define RS_CUDA(call)                                                                            \
    do {                                                                                         \
        cudaError_t rs_cuda_e_ = (call);                                                         \
        if (rs_cuda_e_ != cudaSuccess)                                                           \
            return rs::fail(RS_ECUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(rs_cuda_e_), \
                            __FILE__, __LINE__);                                                 \
    } while (0)

#define RS_LAUNCH_CHECK()                                                                        \
    do {                                                                                         \
        cudaError_t rs_cuda_e_ = cudaGetLastError();                                             \
        if (rs_cuda_e_ != cudaSuccess)                                                           \
            return rs::fail(RS_ECUDA, "kernel launch failed: %s (%s:%d)", cudaGetErrorString(rs_cuda_e_), \
                            __FILE__, __LINE__);                                                 \
    } while (0)

namespace rs {

inline bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

// Raises the dynamic shared-memory limit of kernel `fn` on the current
// device to at least `bytes`.  The attribute belongs to a (function, device)
// pair, so the grant is remembered per pair and later calls with a size
// already granted cost one table lookup.
int smem_optin(const void *fn, size_t bytes);

// Device buffer owned by a handle.
struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
    int alloc(size_t n) {
        release();
        if (n == 0) return RS_OK;
        if (cudaMalloc(&p, n) != cudaSuccess) {
            p = nullptr;
            cudaGetLastError();
            return fail(RS_ENOMEM, "cudaMalloc(%zu) failed", n);
        }
        bytes = n;
        return RS_OK;
    }
    int upload(const void *src, size_t n) {
        RS_TRY(alloc(n));
        if (n && cudaMemcpy(p, src, n, cudaMemcpyHostToDevice) != cudaSuccess)
            return fail(RS_ECUDA, "cudaMemcpy H2D failed");
        return RS_OK;
    }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    template <typename T> T *as() const { return (T *)p; }
    ~DevBuf() { release(); }
    DevBuf() = default;
    DevBuf(const DevBuf &) = delete;
    DevBuf &operator=(const DevBuf &) = delete;
};

// Stream-ordered scratch from the library's own pool of the current device:
// freed in stream order, so calls on any number of threads and streams hold
// separate blocks.  The pool keeps at most 256 MB between calls (mapping memory
// anew takes 200 us a call).
int pool_of_device(cudaMemPool_t *out);
struct PoolBuf {
    void *p = nullptr;
    cudaStream_t st = nullptr;
    int alloc(size_t n, cudaStream_t stream) {
        cudaMemPool_t pool;
        RS_TRY(pool_of_device(&pool));
        st = stream;
        if (cudaMallocFromPoolAsync(&p, n, pool, stream) != cudaSuccess) {
            p = nullptr;
            cudaGetLastError();
            return fail(RS_ENOMEM, "scratch allocation of %zu bytes failed", n);
        }
        return RS_OK;
    }
    template <typename T> T *as() const { return (T *)p; }
    ~PoolBuf() {
        if (p) cudaFreeAsync(p, st);
    }
    PoolBuf() = default;
    PoolBuf(const PoolBuf &) = delete;
    PoolBuf &operator=(const PoolBuf &) = delete;
};

// Launch whose start may overlap the end of the kernel before it in the stream:
// the kernel calls pdl_wait() before it reads or writes anything that the
// stream's earlier work touches, and reads what that work wrote by ld_fresh().
template <typename... P, typename... A>
int launch_overlapped(void (*fn)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    RS_CUDA(cudaLaunchKernelEx(&cfg, fn, P(args)...));
    return RS_OK;
}
#ifdef __CUDACC__
// All earlier work of the stream is complete and visible (at once when the
// kernel was launched without overlap).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// Load, behind pdl_wait(), of what an earlier kernel of the stream wrote.  That
// kernel may still be running when this one starts, so such data is not
// read-only for this kernel's life, as the loads that the compiler makes of
// const __restrict__ pointers and of __ldg require; and an ordinary load of such a pointer
// may be moved ahead of the wait.  This one is neither.
template <typename T> __device__ __forceinline__ T ld_fresh(const T *p) {
    static_assert(sizeof(T) == 4 || sizeof(T) == 8 || sizeof(T) == 16, "one access");
    if constexpr (sizeof(T) == 4) {
        uint32_t r;
        asm volatile("ld.global.b32 %0, [%1];\n" : "=r"(r) : "l"(p));
        return *reinterpret_cast<const T *>(&r);
    } else if constexpr (sizeof(T) == 8) {
        unsigned long long r;
        asm volatile("ld.global.b64 %0, [%1];\n" : "=l"(r) : "l"(p));
        return *reinterpret_cast<const T *>(&r);
    } else {
        uint4 r;
        asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
        return *reinterpret_cast<const T *>(&r);
    }
}
// The next kernel of the stream may be started (it waits in pdl_wait).  Only where
// its CTAs fill every SM anyway: a small grid that starts in a tail is packed
// on the few SMs that are free.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
#endif

}  // namespace rs
