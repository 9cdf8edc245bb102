// Device memory of the library (memory.cu): its pool, and what handles hold for speed only.  Host code
// over the CUDA runtime's C interface.
#pragma once

#include <cuda_runtime_api.h>

#include <cstddef>

namespace adc {

struct ReclaimPin;

// Device memory that a handle holds for speed only (the ladder's pair integrals, the coupling block).
// It goes back to the device when an allocation of any handle fails: that of handles with no call in
// progress (no pins), and that of the failing call itself where it has said so (ReclaimPin::give).
// Freeing memory of a stream-ordered pool waits for nothing, so the rule that makes this safe is that
// unpinned memory has no work in flight: hold() asks for a pin that covers the memory, and the last pin
// is let go only after the stream has been waited for.
struct Reclaimable {
    void* mem[2] = {};
    int device = 0, pins = 0;
    Reclaimable* call = nullptr;  // whose pins cover this memory too (a handle: its calls)
    void hold(void* a, void* b, const ReclaimPin& pin);  // takes over stream-ordered allocations of the current device
    void drop(cudaStream_t s);                           // releases them, ordered on s
    bool held() const;
    ~Reclaimable();
};

// Keeps r, and all memory whose `call` it is, while work that uses it may be issued on s or be in flight there.
struct ReclaimPin {
    Reclaimable& r;
    const cudaStream_t stream;
    ReclaimPin(Reclaimable& r, cudaStream_t s);
    ~ReclaimPin();  // waits for the stream first, unless other pins stay or wait() was the last thing done
    ReclaimPin(const ReclaimPin&) = delete;
    // A failing allocation of this host thread may release x (covered by this pin and by no other, or NULL)
    // after waiting for the stream, until this pin goes or another one is made inside it.
    void give(Reclaimable* x);
    cudaError_t wait();

   private:
    Reclaimable* before;
    cudaStream_t before_stream;
    bool waited = false;
};

// Releases what can be released on the current device (the pool's unused memory too); false if nothing was held.
bool device_memory_reclaim();
// Gives the device back what its pool keeps unused.
void device_memory_trim(int device);

// Stream-ordered allocation from the library's own pool of the current device: the pool keeps up to a
// fiftieth of the device's memory mapped between uses (mapping and unmapping costs about 60 us a buffer
// and 0.4 ms a GB each way: 14 of the 53 ms from a new molecule to its first sigma at 20/180/600).  It gives
// that back when an allocation fails (dev_malloc retries then), when it is asked to (adc_release_memory) and
// with the device's last handle: a program that has released its handles gets all of their memory, at 11.4
// and 4.4 ms for the 34 and 19 ms from the next handle to its first sigma (20/180/600 EA, 17/121/483 IP).
cudaError_t dev_malloc_raw(void** p, size_t bytes, cudaStream_t s);
cudaError_t dev_malloc(void** p, size_t bytes, cudaStream_t s);
// releases such memory, ordered on s
inline void dev_free(void* p, cudaStream_t s) {
    if (p && cudaFreeAsync(p, s) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(p);
    }
}

}  // namespace adc
