// pairs_wait.cuh -- what a host thread waits for a pair count with.
#pragma once

#include <cuda_runtime_api.h>

#include <cstdint>
#include <map>

namespace gi {

// A pinned word and an event, one of each per thread and device it has used,
// kept while the thread lives: a thread that alternates between devices makes
// nothing after its first call on each.
struct PairsWait {
    int64_t* k = nullptr;
    cudaEvent_t ev = nullptr;
    PairsWait() = default;
    PairsWait(const PairsWait&) = delete;
    PairsWait& operator=(const PairsWait&) = delete;
    ~PairsWait() {  // after the runtime has shut down both calls only return an error
        if (ev) cudaEventDestroy(ev);
        if (k) cudaFreeHost(k);
    }
};

// The current device's, or null when it cannot be made.
inline PairsWait* pairs_wait() {
    thread_local std::map<int, PairsWait> words;  // by device
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    PairsWait& w = words[dev];
    void* p = nullptr;
    if (!w.k && cudaHostAlloc(&p, sizeof(int64_t), cudaHostAllocDefault) == cudaSuccess) w.k = static_cast<int64_t*>(p);
    if (!w.ev && cudaEventCreateWithFlags(&w.ev, cudaEventDisableTiming) != cudaSuccess) w.ev = nullptr;
    return w.k && w.ev ? &w : nullptr;
}

}  // namespace gi
