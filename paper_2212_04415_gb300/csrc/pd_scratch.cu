// pd_scratch.cu -- pool of per-call device scratch. One stream-ordered CUDA
// memory pool per device, made at the first use: allocation and release are
// ordered on the call's stream, so calls on several threads and streams never
// share memory in use, and the pool keeps at most kKeep bytes unused (the
// rest goes back to the device at the next synchronisation; all of it, on every
// device, when the last state or field is destroyed). A pool goes with the
// context that it was made in: after a cudaDeviceReset its handle is dropped,
// never used, and the next call makes another.
#include <cuda.h>

#include <atomic>
#include <mutex>

#include "pd_internal.cuh"

namespace pdi {

namespace {
constexpr uint64_t kKeep = 64ull << 20;
constexpr int kMaxDev = 64;
std::mutex g_mu;
struct Pool {
    cudaMemPool_t pool = nullptr;
    CUcontext context = nullptr;  // the device's primary context, nullptr where it is not the one in use
    unsigned long long id = 0;    // its id when the pool was made, unique in the life of the process
} g_pool[kMaxDev];
std::atomic<long> g_handles{0};  // live states and fields

struct Driver {
    CUresult (*device)(CUdevice *, int) = nullptr;
    CUresult (*state)(CUdevice, unsigned *, int *) = nullptr;
    CUresult (*retain)(CUcontext *, CUdevice) = nullptr;
    CUresult (*release)(CUdevice) = nullptr;
    CUresult (*id)(CUcontext, unsigned long long *) = nullptr;
    template <class F>
    static bool get(const char *name, F &f) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return false;
        }
        f = (F)p;
        return true;
    }
    bool ok;
    Driver()
        : ok(get("cuDeviceGet", device) && get("cuDevicePrimaryCtxGetState", state) &&
             get("cuDevicePrimaryCtxRetain", retain) && get("cuDevicePrimaryCtxRelease", release) &&
             get("cuCtxGetId", id)) {}
};

const Driver &driver() {
    static const Driver d;
    return d;
}

// The device's pool, if the context that it was made in still stands (g_mu
// held). A device's primary context keeps its handle through a reset; its id
// changes, or it has none.
cudaMemPool_t live_pool(int dev) {
    Pool &g = g_pool[dev];
    unsigned long long id = 0;
    if (g.pool && g.context && (driver().id(g.context, &id) != CUDA_SUCCESS || id != g.id)) g = Pool{};
    return g.pool;
}

cudaMemPool_t pool_of(int dev) {
    if (dev < 0 || dev >= kMaxDev) return nullptr;
    std::lock_guard<std::mutex> lock(g_mu);
    if (cudaMemPool_t p = live_pool(dev)) return p;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kKeep;
    if (cudaFree(nullptr) != cudaSuccess || cudaMemPoolCreate(&pool, &props) != cudaSuccess) return nullptr;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return nullptr;
    }
    Pool &g = g_pool[dev];
    g.pool = pool;
    const Driver &d = driver();
    CUdevice cd;
    unsigned flags;
    int active = 0;
    if (d.ok && d.device(&cd, dev) == CUDA_SUCCESS && d.state(cd, &flags, &active) == CUDA_SUCCESS && active &&
        d.retain(&g.context, cd) == CUDA_SUCCESS) {
        if (d.id(g.context, &g.id) != CUDA_SUCCESS) g.context = nullptr;
        d.release(cd);
    }
    return pool;
}
}  // namespace

int scratch_alloc(Scratch &h, size_t bytes, cudaStream_t s) {
    int dev = 0;
    PD_CHECK_CUDA(cudaGetDevice(&dev));
    cudaMemPool_t pool = pool_of(dev);
    cudaError_t e = pool ? cudaMallocFromPoolAsync(&h.p, bytes ? bytes : 1, pool, s) : cudaErrorMemoryAllocation;
    if (e != cudaSuccess) {
        cudaGetLastError();
        h.p = nullptr;
        set_error("scratch of %zu bytes: %s", bytes, cudaGetErrorString(e));
        return PD_ERR_OOM;
    }
    h.s = s;
    return PD_OK;
}

void scratch_hold() { ++g_handles; }

void scratch_release() {
    if (--g_handles > 0) return;
    std::lock_guard<std::mutex> lock(g_mu);
    for (int dev = 0; dev < kMaxDev; ++dev)
        if (g_pool[dev].pool && live_pool(dev)) cudaMemPoolTrimTo(g_pool[dev].pool, 0);
}

}  // namespace pdi
