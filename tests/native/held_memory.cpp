// The rule of memory.cu, that memory held for speed and not pinned has no work in flight, against a fake
// CUDA runtime: a stream is the set of buffers that its queued work uses, waiting for it empties the set,
// and freeing a buffer that some stream still uses is counted as a violation.
#include <cstdio>
#include <map>
#include <mutex>
#include <set>
#include <stdexcept>
#include <string>
#include <thread>

#include "memory.cuh"

namespace {
std::mutex mu;
std::map<void*, size_t> live;
std::map<cudaStream_t, std::set<void*>> queued;
size_t capacity = 100, used = 0;
int waits = 0, violations = 0, next_address = 1;
const cudaStream_t s1 = (cudaStream_t)1, s2 = (cudaStream_t)2;

void launch(cudaStream_t s, void* p) {
    std::lock_guard<std::mutex> lk(mu);
    if (p) queued[s].insert(p);
    if (p && !live.count(p)) ++violations;  // work on memory that is gone
}
cudaError_t allocate(void** p, size_t bytes) {
    std::lock_guard<std::mutex> lk(mu);
    if (used + bytes > capacity) return cudaErrorMemoryAllocation;
    *p = (void*)(size_t)(next_address++ * 256);
    live[*p] = bytes;
    used += bytes;
    return cudaSuccess;
}
void gone(void* p) {
    used -= live[p];
    live.erase(p);
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { return *f = capacity - used, *t = capacity, cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { return *p = (cudaMemPool_t)8, cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    std::lock_guard<std::mutex> lk(mu);
    ++waits;
    queued[s].clear();
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {  // (of memory from a pool: waits for nothing)
    std::lock_guard<std::mutex> lk(mu);
    for (auto& q : queued) violations += (int)q.second.count(p);
    gone(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {  // ordered after the work of its own stream
    std::lock_guard<std::mutex> lk(mu);
    for (auto& q : queued)
        if (q.first != s) violations += (int)q.second.count(p);
    queued[s].erase(p);
    gone(p);
    return cudaSuccess;
}
}

using namespace adc;

static int failures = 0;
#define CHECK(x)                                            \
    do {                                                    \
        if (!(x)) std::printf("line %d: %s\n", __LINE__, #x), ++failures; \
    } while (0)

struct Handle {
    cudaStream_t s;
    Reclaimable call, a, b;
    explicit Handle(cudaStream_t st) : s(st) { a.call = b.call = &call; }
    ~Handle() {
        a.drop(s);
        b.drop(s);
    }
    void form(Reclaimable& r, size_t n, const ReclaimPin& pin) {
        void* p = nullptr;
        CHECK(dev_malloc_raw(&p, n, s) == cudaSuccess);
        r.hold(p, nullptr, pin);
        launch(s, p);
    }
};

int main() {
    void* p = nullptr;
    {  // nothing is held without a pin that covers it
        Handle h(s1), g(s2);
        ReclaimPin other(g.call, s2);
        bool refused = false;
        void* q = nullptr;
        dev_malloc_raw(&q, 10, s1);
        try {
            h.a.hold(q, nullptr, other);
        } catch (const std::logic_error&) {
            refused = true;
        }
        CHECK(refused && !h.a.held());
        dev_free(q, s1);
    }
    {  // work queued when a call ends (also by an exception) has been waited for before another call's failing
       // allocation takes the memory; while the call is in progress it stays
        Handle h(s1);
        try {
            ReclaimPin call(h.call, s1);
            h.form(h.a, 60, call);
            CHECK(dev_malloc(&p, 80, s2) == cudaErrorMemoryAllocation && h.a.held());
            launch(s1, h.a.mem[0]);
            throw std::runtime_error("out of the call");
        } catch (const std::runtime_error&) {
        }
        CHECK(h.a.held());
        CHECK(dev_malloc(&p, 80, s2) == cudaSuccess && !h.a.held());
        dev_free(p, s2);
    }
    {  // pins inside a call wait for nothing and release nothing; one wait serves the call's end
        Handle h(s1);
        {
            ReclaimPin call(h.call, s1);
            h.form(h.a, 60, call);
            const int w = waits;
            {
                ReclaimPin inner(h.a, s1);
                launch(s1, h.a.mem[0]);
            }
            CHECK(waits == w);
            CHECK(dev_malloc(&p, 80, s2) == cudaErrorMemoryAllocation && h.a.held());
            CHECK(call.wait() == cudaSuccess && waits == w + 1);
        }
        CHECK(waits > 0 && h.a.held());
    }
    {  // a call's own allocation takes what it gave, after waiting; not what an inner pin keeps, nor the rest
        Handle h(s1);
        ReclaimPin call(h.call, s1);
        h.form(h.a, 40, call);
        h.form(h.b, 40, call);
        call.give(&h.a);
        launch(s1, h.a.mem[0]);
        launch(s1, h.b.mem[0]);
        {
            ReclaimPin inner(h.a, s1);
            CHECK(dev_malloc(&p, 50, s1) == cudaErrorMemoryAllocation && h.a.held() && h.b.held());
        }
        CHECK(dev_malloc(&p, 50, s1) == cudaSuccess && !h.a.held() && h.b.held());
        dev_free(p, s1);
    }
    {  // two host threads: one forms, uses and lets go, the other runs out of memory all the time
        Handle h(s1);
        std::thread user([&] {
            for (int i = 0; i < 20000; ++i) {
                ReclaimPin call(h.call, s1);
                if (!h.a.held()) {
                    void* q = nullptr;
                    if (dev_malloc_raw(&q, 60, s1) == cudaSuccess) h.a.hold(q, nullptr, call);
                }
                launch(s1, h.a.mem[0]);
                if (i % 2) call.wait();
            }
        });
        for (int i = 0; i < 20000; ++i)
            if (dev_malloc(&p, 80, s2) == cudaSuccess) dev_free(p, s2);
        user.join();
    }
    CHECK(violations == 0);
    CHECK(used == 0);
    if (failures || violations) std::printf("%d failures, %d violations\n", failures, violations);
    return failures || violations ? 1 : 0;
}
