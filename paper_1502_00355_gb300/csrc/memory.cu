// memory.cu -- device memory of the library's handles.
//
// Every buffer a mesh, a build or a served job holds comes from one
// stream-ordered memory pool per device that the library owns
// (cudaMemPoolCreate), allocated and freed on the stream that uses it.  The
// pool keeps the memory that destroyed handles return, so a later handle of
// similar size reuses it at once instead of mapping new memory (cudaMalloc)
// and unmapping it again at the device-wide synchronisation of cudaFree.
// sls_trim_memory hands the kept memory back.  The pool is the library's
// own: the device's default pool, which other code in the process may use,
// is left as it is.
#include <mutex>
#include <vector>

#include "api_common.h"

namespace sls {
namespace {

struct DevicePool {
    unsigned long long ctx = 0;  // the context the pool belongs to (0: none yet)
    cudaMemPool_t pool = nullptr;
};

std::mutex g_pool_mu;
DevicePool g_pools[64];

// The pool of the current device, made on first use and again after the
// device's context changed (cudaDeviceReset destroys pools).
cudaError_t current_pool(cudaMemPool_t *out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    const unsigned long long ctx = current_context_id();
    std::lock_guard<std::mutex> lk(g_pool_mu);
    DevicePool &P = g_pools[dev];
    if (P.pool && P.ctx == ctx && ctx != 0) {
        *out = P.pool;
        return cudaSuccess;
    }
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = ~0ull;  // keep freed memory until trimmed
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return e;
    }
    P.pool = pool;
    P.ctx = ctx;
    *out = pool;
    return cudaSuccess;
}

// Kits of destroyed handles, at most kKits of each device: making a stream and
// page-locking memory takes as long as twenty passes of a small mesh (150 x 111
// nodes created, smoothed and destroyed: 463 us a request, 515 without reuse).
constexpr size_t kKits = 16;
struct KitCache {
    unsigned long long ctx = 0;
    std::vector<HandleKit> kits;
};
std::mutex g_kit_mu;
KitCache g_kits[64];

void destroy_kit(const HandleKit &k)
{
    if (k.host) cudaFreeHost(k.host);
    if (k.stream) cudaStreamDestroy(k.stream);
}

}  // namespace

cudaError_t take_kit(HandleKit *kit)
{
    HandleKit k;
    cudaError_t e = cudaGetDevice(&k.device);
    if (e != cudaSuccess) return e;
    k.ctx = current_context_id();
    if (k.ctx != 0 && k.device >= 0 && k.device < 64) {
        std::lock_guard<std::mutex> lk(g_kit_mu);
        KitCache &c = g_kits[k.device];
        if (c.ctx != k.ctx) {  // kits of a context that is gone went with it
            c.kits.clear();
            c.ctx = k.ctx;
        }
        if (!c.kits.empty()) {
            *kit = c.kits.back();
            c.kits.pop_back();
            return cudaSuccess;
        }
    }
    e = cudaStreamCreateWithFlags(&k.stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&k.host, sizeof(PassStats) * kHostStats);
    if (e != cudaSuccess) {
        destroy_kit(k);
        return e;
    }
    *kit = k;
    return cudaSuccess;
}

void give_kit(const HandleKit &kit, bool keep)
{
    if (!kit.stream) return;
    if (keep && kit.ctx != 0 && kit.device >= 0 && kit.device < 64) {
        std::lock_guard<std::mutex> lk(g_kit_mu);
        KitCache &c = g_kits[kit.device];  // the kit's device, whichever is current
        if (c.ctx == kit.ctx && c.kits.size() < kKits) {
            c.kits.push_back(kit);
            return;
        }
    }
    destroy_kit(kit);
}

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = current_pool(&pool);
    if (e != cudaSuccess) return e;
    return cudaMallocFromPoolAsync(p, bytes > 0 ? bytes : 1, pool, s);
}

void pool_free(void *p, cudaStream_t s)
{
    if (p) cudaFreeAsync(p, s);
}

}  // namespace sls

using namespace sls;

extern "C" sls_status sls_trim_memory(size_t keep_bytes)
{
    std::vector<HandleKit> kits;
    int dev = -1;
    const unsigned long long ctx = current_context_id();
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
        std::lock_guard<std::mutex> lk(g_kit_mu);
        if (g_kits[dev].ctx == ctx) kits.swap(g_kits[dev].kits);
    }
    for (const HandleKit &k : kits) destroy_kit(k);
    cudaMemPool_t pool = nullptr;
    cudaError_t e = current_pool(&pool);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();  // frees still queued on streams reach the pool
    if (e == cudaSuccess) e = cudaMemPoolTrimTo(pool, keep_bytes);
    if (e != cudaSuccess) return cuda_fail(e, "sls_trim_memory");
    return SLS_OK;
}
