// Work done once per device.
#pragma once
#include <algorithm>
#include <mutex>
#include <vector>

#include <cuda_runtime.h>

namespace hpt {

class OncePerDevice {
    std::mutex mu;
    std::vector<int> done;

  public:
    // f() the first time it is called for a device; again if it failed
    template <class F> cudaError_t operator()(int device, F f)
    {
        std::lock_guard<std::mutex> lk(mu);
        if (std::find(done.begin(), done.end(), device) != done.end()) return cudaSuccess;
        const cudaError_t e = f();
        if (e == cudaSuccess) done.push_back(device);
        return e;
    }
};

}  // namespace hpt
