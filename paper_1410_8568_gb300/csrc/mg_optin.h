// mg_optin.h -- kernel attributes (more shared memory, larger clusters), set
// once per device: cudaFuncSetAttribute acts on the current device alone, and
// one process may hold handles on several.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace gbmg {

// once(set): runs set() on the first call that finds its device current, and
// again after a failure; the error of set(), success where it has run.  Two
// threads that come first together may both run it (setting an attribute twice
// does no harm).
class DeviceOnce {
    std::atomic<unsigned long long> done{0};  // a bit per device; devices from 64 on: every time

public:
    template <class F>
    cudaError_t operator()(F &&set)
    {
        int device = 0;
        cudaError_t e = cudaGetDevice(&device);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = device < 64 ? 1ull << device : 0ull;
        if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = set();
        if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace gbmg
