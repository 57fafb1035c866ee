// Set-up that CUDA keeps per device, made once on each: a kernel's opt-in to more
// shared memory than 48 KB (cudaFuncSetAttribute) holds for the current device
// only, and contexts on several devices, the serving threads and the callers'
// share the process.
#pragma once

#include <cuda_runtime.h>

#include <mutex>
#include <vector>

namespace bfi {

class DeviceOnce {
  public:
    // calls set() unless it has succeeded on the current device
    template <typename F>
    cudaError_t run(F set)
    {
        int d = 0;
        cudaError_t e = cudaGetDevice(&d);
        if (e != cudaSuccess) return e;
        std::lock_guard<std::mutex> g(mu_);
        if ((size_t)d < done_.size() && done_[d]) return cudaSuccess;
        e = set();
        if (e != cudaSuccess) return e;
        if (done_.size() <= (size_t)d) done_.resize(d + 1, 0);
        done_[d] = 1;
        return cudaSuccess;
    }

  private:
    std::mutex mu_;
    std::vector<char> done_;
};

}  // namespace bfi
