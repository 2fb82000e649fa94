// The library's device memory pool (one per device, stream-ordered).
//
// Work buffers live for one call or one step, so a pool that hands freed memory back at every
// synchronisation -- the default release threshold is 0 -- maps it again on the next call: a 64-state
// matvec took 510 us after a synchronisation against 170 among other calls.  The pool is the
// library's own, so its threshold touches no other user of the device's default pool -- and no other
// allocator of the process can use what it keeps.  That is up to kIdleBytes between single operations
// (those at the largest bonds take half a gigabyte and more, and free it, each call); everything while
// a context is alive, whose sweeps free and allocate gigabytes per bond step; nothing after the last
// context is destroyed or dmrg_trim is called.  All of it is safe from several host threads and streams
// (the driver's pool is).
#include <mutex>

#include "internal.h"

namespace pd {

namespace {
constexpr unsigned long long kIdleBytes = 2ull << 30;
constexpr int kMaxDevices = 64;
struct DevicePool {
    cudaMemPool_t pool = nullptr;
    int holders = 0;
};
std::mutex g_mu;
DevicePool g_pools[kMaxDevices];

int current_device() {
    int dev = 0;
    PD_CK(cudaGetDevice(&dev));
    PD_REQUIRE(dev >= 0 && dev < kMaxDevices, DMRG_ERR_CAPACITY, "device ordinal beyond 63");
    return dev;
}

cudaMemPool_t pool_of(int dev) {   // g_mu held
    DevicePool& d = g_pools[dev];
    if (!d.pool) {
        cudaMemPoolProps props{};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        PD_CK(cudaMemPoolCreate(&p, &props));
        unsigned long long keep = kIdleBytes;
        const cudaError_t e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) cudaMemPoolDestroy(p);
        PD_CK(e);
        d.pool = p;
    }
    return d.pool;
}
}  // namespace

void* pool_alloc(size_t bytes, cudaStream_t st) {
    static thread_local int last_dev = -1;
    static thread_local cudaMemPool_t last_pool = nullptr;
    const int dev = current_device();
    if (dev != last_dev) {
        std::lock_guard<std::mutex> lk(g_mu);
        last_pool = pool_of(dev);
        last_dev = dev;
    }
    void* p = nullptr;
    PD_CK(cudaMallocFromPoolAsync(&p, bytes, last_pool, st));
    return p;
}

PoolHold::PoolHold() {
    const int d = current_device();
    std::lock_guard<std::mutex> lk(g_mu);
    const cudaMemPool_t p = pool_of(d);
    if (g_pools[d].holders == 0) {
        unsigned long long keep = ~0ull;
        PD_CK(cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep));
    }
    ++g_pools[d].holders;
    dev = d;
}

PoolHold::~PoolHold() {
    std::lock_guard<std::mutex> lk(g_mu);
    if (--g_pools[dev].holders > 0) return;
    unsigned long long keep = kIdleBytes;
    cudaMemPoolSetAttribute(g_pools[dev].pool, cudaMemPoolAttrReleaseThreshold, &keep);
}

cudaError_t pool_trim(bool idle_only) {
    std::lock_guard<std::mutex> lk(g_mu);
    cudaError_t e = cudaSuccess;
    for (const DevicePool& d : g_pools)
        if (d.pool && !(idle_only && d.holders > 0)) {
            const cudaError_t x = cudaMemPoolTrimTo(d.pool, 0);
            if (x != cudaSuccess) e = x;
        }
    return e;
}

static bool pool_in_use() {
    std::lock_guard<std::mutex> lk(g_mu);
    for (const DevicePool& d : g_pools)
        if (d.pool) return true;
    return false;
}

}  // namespace pd

extern "C" dmrg_status dmrg_trim(void) {
    if (!pd::pool_in_use()) return DMRG_OK;          // (nothing allocated yet: no device call)
    if (cudaDeviceSynchronize() != cudaSuccess) return DMRG_ERR_CUDA;
    return pd::pool_trim(false) == cudaSuccess ? DMRG_OK : DMRG_ERR_CUDA;
}
