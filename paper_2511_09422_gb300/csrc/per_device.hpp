// Set-up that a kernel needs once on every device: function attributes hold for
// the device they are set on only.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>

class PerDevice {
    std::atomic<unsigned long long> done{0};  // a bit per device

public:
    // Runs `setup` (returning a cudaError_t) unless it has succeeded on the current
    // device; threads that come at the same time may both run it.
    template <class Setup>
    cudaError_t once(Setup setup)
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess)
            return e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
        if (done.load() & bit)
            return cudaSuccess;
        e = setup();
        if (e == cudaSuccess)
            done.fetch_or(bit);
        return e;
    }
};
