// scratch.cu -- per-call scratch memory from a pool of the library's own.
//
// The metrics, the adjoint and the payouts take their scratch in stream order
// and release it on the stream. The device's default pool gives released
// memory back to the system whenever the host waits for the device, so a
// caller that reads each result paid the mapping of the same scratch on every
// call (art_metrics on one layer of 1,000,000 trials, each call waited for:
// 293 us, 111 from this pool; not waited for, both 89). This pool keeps up to
// kScratchKeep bytes instead; what it keeps is returned when the device's last
// portfolio is destroyed, or by art_release_scratch (the metrics need no
// portfolio).
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
int64_t g_portfolios[kMaxDevices];  // live portfolios of each device
std::mutex g_mutex;                 // guards both

// Give back what the current device's pool keeps; memory that work in flight
// still uses stays. With g_mutex held.
cudaError_t trim_current() {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) return e;
    if (!g_pools[dev].pool || g_pools[dev].ctx_id != current_context_id()) return cudaSuccess;
    return cudaMemPoolTrimTo(g_pools[dev].pool, 0);
}

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

void scratch_user(int device, int delta) {
    if (device < 0 || device >= kMaxDevices) return;
    std::lock_guard<std::mutex> lock(g_mutex);
    g_portfolios[device] += delta;
    int current = -1;
    if (delta > 0 || g_portfolios[device] > 0 || cudaGetDevice(&current) != cudaSuccess || current != device) return;
    trim_current();
}

}  // namespace art

extern "C" art_status art_release_scratch(void) {
    std::lock_guard<std::mutex> lock(art::g_mutex);
    const cudaError_t e = art::trim_current();
    if (e) art::set_last_error(e);
    return e ? ART_ECUDA : ART_OK;
}
