// Host-side helpers of device.h that keep state across calls.
#include <map>
#include <mutex>
#include <utility>

#include "device.h"

namespace rs {

int smem_optin(const void *fn, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<const void *, int>, size_t> granted;
    int dev = 0;
    RS_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    size_t &g = granted[{fn, dev}];
    if (g >= bytes) return RS_OK;
    RS_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    g = bytes;
    return RS_OK;
}

int pool_of_device(cudaMemPool_t *out) {
    constexpr int MAXDEV = 64;
    static std::mutex mu;
    static cudaMemPool_t pools[MAXDEV] = {};
    int dev = 0;
    RS_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAXDEV) return fail(RS_ECUDA, "device %d out of range", dev);
    std::lock_guard<std::mutex> lk(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        // the first call may stand in a stream capture, which allows this thread no
        // such call unless it asks (it enqueues nothing, so the graph is not touched)
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
        RS_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
        cudaMemPool_t p = nullptr;
        uint64_t keep = 256ull << 20;
        cudaError_t e = cudaMemPoolCreate(&p, &props);
        if (e == cudaSuccess) e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        RS_CUDA(cudaThreadExchangeStreamCaptureMode(&mode));
        RS_CUDA(e);
        pools[dev] = p;
    }
    *out = pools[dev];
    return RS_OK;
}

}  // namespace rs
