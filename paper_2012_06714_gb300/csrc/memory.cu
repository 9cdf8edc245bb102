#include "memory.cuh"

#include <algorithm>
#include <mutex>
#include <stdexcept>
#include <vector>

namespace adc {

// ---- memory held for speed only ----------------------------------------------------
namespace {
std::mutex g_reclaim_mu;
std::vector<Reclaimable*> g_reclaim;  // those that hold memory
// what the call running on this host thread may give up itself, and its stream
thread_local Reclaimable* tl_own = nullptr;
thread_local cudaStream_t tl_own_stream = nullptr;

void forget(Reclaimable* r) { g_reclaim.erase(std::remove(g_reclaim.begin(), g_reclaim.end(), r), g_reclaim.end()); }
int pins_of(const Reclaimable* r) { return r->pins + (r->call ? r->call->pins : 0); }
}  // namespace

void Reclaimable::hold(void* a, void* b, const ReclaimPin& pin) {
    if (&pin.r != this && &pin.r != call) throw std::logic_error("Reclaimable: held without a pin");
    cudaGetDevice(&device);
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    mem[0] = a;
    mem[1] = b;
    g_reclaim.push_back(this);
}
void Reclaimable::drop(cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    forget(this);
    for (void*& p : mem) {
        dev_free(p, s);
        p = nullptr;
    }
}
bool Reclaimable::held() const {
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    return mem[0] != nullptr;
}
Reclaimable::~Reclaimable() {
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    forget(this);
    for (void* p : mem)
        if (p) cudaFree(p);
}

ReclaimPin::ReclaimPin(Reclaimable& x, cudaStream_t s) : r(x), stream(s) {
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    ++r.pins;
    before = tl_own;
    before_stream = tl_own_stream;
    tl_own = nullptr;
}
void ReclaimPin::give(Reclaimable* x) {
    tl_own = x;
    tl_own_stream = stream;
}
cudaError_t ReclaimPin::wait() {
    const cudaError_t e = cudaStreamSynchronize(stream);
    waited = e == cudaSuccess;
    return e;
}
ReclaimPin::~ReclaimPin() {
    bool last;
    {
        std::lock_guard<std::mutex> lk(g_reclaim_mu);
        last = pins_of(&r) == 1;
    }
    if (last && !waited && cudaStreamSynchronize(stream) != cudaSuccess) cudaGetLastError();
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    --r.pins;
    tl_own = before;
    tl_own_stream = before_stream;
}

// ---- the library's memory pool -------------------------------------------------------
namespace {
struct Pool {
    std::once_flag once;
    cudaMemPool_t pool = nullptr;
};
Pool g_pools[64];
// the current device's pool (NULL: it could not be made, the device's default pool serves)
cudaMemPool_t pool_of(int dev) {
    if (dev < 0 || dev >= 64) return nullptr;
    Pool& q = g_pools[dev];
    std::call_once(q.once, [&q, dev] {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        size_t fr = 0, tot = 0;
        if (cudaMemGetInfo(&fr, &tot) != cudaSuccess || cudaMemPoolCreate(&q.pool, &props) != cudaSuccess) {
            cudaGetLastError();
            q.pool = nullptr;
            return;
        }
        unsigned long long keep = tot / 50;
        cudaMemPoolSetAttribute(q.pool, cudaMemPoolAttrReleaseThreshold, &keep);
    });
    return q.pool;
}
}  // namespace

cudaError_t dev_malloc_raw(void** p, size_t bytes, cudaStream_t s) {
    int dev = 0;
    cudaMemPool_t pool = cudaGetDevice(&dev) == cudaSuccess ? pool_of(dev) : nullptr;
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}
cudaError_t dev_malloc(void** p, size_t bytes, cudaStream_t s) {
    cudaError_t e = dev_malloc_raw(p, bytes, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        device_memory_reclaim();
        e = dev_malloc_raw(p, bytes, s);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();  // reported here, not by the next launch's check
    }
    return e;
}

void device_memory_trim(int device) {
    if (cudaMemPool_t p = pool_of(device)) cudaMemPoolTrimTo(p, 0);
}

bool device_memory_reclaim() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    struct Trim {  // what the pool keeps unused goes back too, after what is freed below
        int dev;
        ~Trim() { device_memory_trim(dev); }
    } trim{dev};
    std::lock_guard<std::mutex> lk(g_reclaim_mu);
    bool any = false;
    for (size_t i = 0; i < g_reclaim.size();) {
        Reclaimable* r = g_reclaim[i];
        const bool own = r == tl_own && pins_of(r) == 1;
        if (r->device != dev || (pins_of(r) > 0 && !own)) {
            ++i;
            continue;
        }
        // what is not pinned has no work in flight; this thread's own call waits for what it has
        // issued so far
        if (own && cudaStreamSynchronize(tl_own_stream) != cudaSuccess) return any;
        for (void*& p : r->mem) {
            if (p) cudaFree(p);
            p = nullptr;
        }
        g_reclaim.erase(g_reclaim.begin() + i);
        any = true;
    }
    return any;
}

}  // namespace adc
