// scratch.cu -- per-call scratch memory from a pool of the library's own.
//
// The metrics, the adjoint and the payouts take their scratch in stream order
// and release it on the stream. The device's default pool gives released
// memory back to the system whenever the host waits for the device, so a
// caller that reads each result paid the mapping of the same scratch on every
// call (art_metrics on one layer of 1,000,000 trials, each call waited for:
// 293 us, 111 from this pool; not waited for, both 89). This pool keeps up to
// kScratchKeep bytes instead; what it keeps is returned when the process's
// last portfolio is destroyed.
#include <mutex>

#include "art_internal.cuh"

namespace art {

// Id of the current device's context (unique over the process's life, so a
// context recreated after cudaDeviceReset gets a new one); 0 if the driver
// cannot tell. Taken from the driver through the runtime's entry-point
// lookup, without linking the driver library.
unsigned long long current_context_id() {
    typedef int (*GetCurrent)(void**);
    typedef int (*GetId)(void*, unsigned long long*);
    static GetCurrent get_current = nullptr;
    static GetId get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrent>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetId>(f);
    });
    void* ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
    return id;
}

int64_t bytes_behind(const void* p) {
    typedef int (*GetRange)(unsigned long long*, size_t*, unsigned long long);
    static GetRange get_range = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_range = reinterpret_cast<GetRange>(f);
    });
    unsigned long long base = 0;
    size_t bytes = 0;
    const unsigned long long a = reinterpret_cast<uintptr_t>(p);
    if (!get_range || get_range(&base, &bytes, a) != 0 || a < base || a > base + bytes) return INT64_MAX;
    return (int64_t)(base + bytes - a);
}

namespace {

constexpr uint64_t kScratchKeep = 256ULL << 20;  // bytes a device's pool keeps between calls
constexpr int kMaxDevices = 64;

struct DevicePool {
    cudaMemPool_t pool = nullptr;
    unsigned long long ctx_id = 0;  // the context the pool was made in
};
DevicePool g_pools[kMaxDevices];
int64_t g_portfolios = 0;  // live portfolios of the process
std::mutex g_mutex;        // guards both

// The current device's pool; NULL where it cannot be had (the device's
// default pool serves then). A context recreated after a device reset makes
// a new pool.
cudaMemPool_t device_pool() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(g_mutex);
    DevicePool& p = g_pools[dev];
    const unsigned long long ctx = current_context_id();
    if (ctx == 0) return nullptr;
    if (p.pool && p.ctx_id == ctx) return p.pool;
    p.pool = nullptr;
    p.ctx_id = ctx;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = kScratchKeep;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(pool);
        return nullptr;
    }
    p.pool = pool;
    return pool;
}

}  // namespace

cudaError_t scratch_alloc(void** out, size_t bytes, cudaStream_t s) {
    // a captured call's scratch belongs to its graph
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
        return cudaMallocAsync(out, bytes, s);
    cudaMemPool_t pool = device_pool();
    return pool ? cudaMallocFromPoolAsync(out, bytes, pool, s) : cudaMallocAsync(out, bytes, s);
}

void scratch_user(int delta) {
    std::lock_guard<std::mutex> lock(g_mutex);
    g_portfolios += delta;
    if (delta > 0 || g_portfolios > 0) return;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;
    // memory that work in flight still uses stays
    if (g_pools[dev].pool && g_pools[dev].ctx_id == current_context_id()) cudaMemPoolTrimTo(g_pools[dev].pool, 0);
}

}  // namespace art
