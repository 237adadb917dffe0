// Device memory of the set-up calls (corpus tables, statistics, tokenizer): a bounded pool per device.
//
// A call needs hundreds of megabytes for a few milliseconds.  cudaMalloc and cudaFree of 2 to 512 MB took 0.36 to 0.6 ms
// and 0.29 to 0.76 ms each, in calls whose kernels run for microseconds; a block that the pool still holds takes 2 us.
// A block that the pool has to map first costs about 6.5 us per megabyte, more than cudaMalloc (1 GB: 0.7 ms), so what
// would not be kept anyway does not come from it.
#include "kernels.h"

#include <mutex>

namespace tasc {

namespace {

constexpr int MAX_DEVICES = 64;
constexpr uint64_t KEEP_BYTES = 2ull << 30;          // what a pool may hold beyond the blocks in use
constexpr size_t POOLED_BYTES = 1ull << 30;          // largest block that comes from a pool

std::mutex pool_mu;
cudaMemPool_t pools[MAX_DEVICES] = {nullptr};

// the pool of a device, created at its first use; null when there cannot be one
cudaMemPool_t pool_of(int dev) {
    if (dev < 0 || dev >= MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lk(pool_mu);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        uint64_t keep = KEEP_BYTES;
        cudaMemPool_t p = nullptr;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) { (void)cudaGetLastError(); return nullptr; }
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            (void)cudaGetLastError();
            cudaMemPoolDestroy(p);
            return nullptr;
        }
        pools[dev] = p;
    }
    return pools[dev];
}

}  // namespace

bool scratch_alloc(void** p, size_t bytes, cudaStream_t stream, bool* pooled) {
    *p = nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return false; }
    cudaMemPool_t pool = bytes <= POOLED_BYTES ? pool_of(dev) : nullptr;
    if (pool && cudaMallocFromPoolAsync(p, bytes, pool, stream) == cudaSuccess) { *pooled = true; return true; }
    (void)cudaGetLastError();
    *pooled = false;
    if (cudaMalloc(p, bytes) == cudaSuccess) return true;
    (void)cudaGetLastError();
    (void)scratch_trim();                            // what the pool holds may be what is missing
    if (cudaMalloc(p, bytes) == cudaSuccess) return true;
    (void)cudaGetLastError();
    *p = nullptr;
    return false;
}

void scratch_free(void* p, cudaStream_t stream, bool pooled) {
    if (!p) return;
    if (!(pooled ? cudaFreeAsync(p, stream) == cudaSuccess : cudaFree(p) == cudaSuccess)) (void)cudaGetLastError();
}

tasc_status scratch_trim() {
    int dev = 0;
    TASC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= MAX_DEVICES) return TASC_OK;
    std::lock_guard<std::mutex> lk(pool_mu);
    if (!pools[dev]) return TASC_OK;
    TASC_CUDA_TRY(cudaDeviceSynchronize());          // a block whose turn to be freed has not come is one in use
    TASC_CUDA_TRY(cudaMemPoolTrimTo(pools[dev], 0));
    return TASC_OK;
}

}  // namespace tasc

extern "C" tasc_status tasc_scratch_release(void) { return tasc::scratch_trim(); }
