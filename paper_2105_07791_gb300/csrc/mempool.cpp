// Stream-ordered work space of the library: one memory pool per device whose
// release threshold is unbounded, so memory freed with cudaFreeAsync stays
// mapped for the next call instead of going back to the driver at every
// stream synchronisation (the default pool's threshold of 0 does that, and
// remapping ~100 MB of GMRES work space costs far more than the solve step
// it serves).  The pool is created on first use per device and lives until
// the process exits.
//
// Page-locked staging buffers for small host tables: a copy from pageable
// memory costs the host several microseconds each, and the compression's
// rounds upload a dozen tables per round.  A buffer belongs to one call at a
// time and is handed out again once the copies of the call before have run (an
// event on that call's stream): a call takes an idle one, or a new one while
// the device has fewer than PINNED_MAX, or does without.  It never waits: the
// event may lie behind other work of another thread's stream.
#include <cstdint>
#include <mutex>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "mempool.h"

namespace ndhss {

namespace {
constexpr int MAX_DEVICES = 64;
std::mutex g_pool_mu;
cudaMemPool_t g_pool[MAX_DEVICES] = {};
}  // namespace

cudaError_t pool_malloc_async(void** p, size_t bytes, cudaStream_t st) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaMallocAsync(p, bytes, st);
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_pool_mu);
        if (!g_pool[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.handleTypes = cudaMemHandleTypeNone;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            cudaMemPool_t np = nullptr;
            e = cudaMemPoolCreate(&np, &props);
            if (e != cudaSuccess) return e;
            uint64_t thr = UINT64_MAX;
            e = cudaMemPoolSetAttribute(np, cudaMemPoolAttrReleaseThreshold, &thr);
            if (e != cudaSuccess) {
                cudaMemPoolDestroy(np);
                return e;
            }
            g_pool[dev] = np;
        }
        pool = g_pool[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

namespace {
constexpr int PINNED_MAX = 4;                    // buffers per device, in use or not
std::mutex g_pinned_mu;
int g_pinned_count[MAX_DEVICES] = {};
std::vector<PinnedBuf*>& pinned_free() {
    static std::vector<PinnedBuf*>* v = new std::vector<PinnedBuf*>();     // lives until the process exits
    return *v;
}
void pinned_destroy(PinnedBuf* b) {
    if (b->p) cudaFreeHost(b->p);
    if (b->ev) cudaEventDestroy(b->ev);
    std::lock_guard<std::mutex> lock(g_pinned_mu);
    --g_pinned_count[b->dev];
    delete b;
}
}  // namespace

PinnedBuf* pinned_acquire() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return nullptr;
    {
        std::lock_guard<std::mutex> lock(g_pinned_mu);
        std::vector<PinnedBuf*>& v = pinned_free();
        for (size_t i = v.size(); i-- > 0;) {
            if (v[i]->dev != dev) continue;
            if (cudaEventQuery(v[i]->ev) != cudaSuccess) {
                cudaGetLastError();              // not ready
                continue;
            }
            PinnedBuf* b = v[i];
            v.erase(v.begin() + (std::ptrdiff_t)i);
            return b;
        }
        if (g_pinned_count[dev] >= PINNED_MAX) return nullptr;
        ++g_pinned_count[dev];
    }
    PinnedBuf* b = new (std::nothrow) PinnedBuf();
    if (!b) {
        std::lock_guard<std::mutex> lock(g_pinned_mu);
        --g_pinned_count[dev];
        return nullptr;
    }
    b->dev = dev;
    if (cudaHostAlloc(reinterpret_cast<void**>(&b->p), PINNED_BYTES, cudaHostAllocDefault) != cudaSuccess ||
        cudaEventCreateWithFlags(&b->ev, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        pinned_destroy(b);
        return nullptr;
    }
    return b;
}

void pinned_release(PinnedBuf* b, cudaStream_t st) {
    if (!b) return;
    if (cudaEventRecord(b->ev, st) == cudaSuccess) {
        std::lock_guard<std::mutex> lock(g_pinned_mu);
        pinned_free().push_back(b);
        return;
    }
    cudaStreamSynchronize(st);
    cudaGetLastError();
    pinned_destroy(b);
}

}  // namespace ndhss
