// The once-per-device guard (csrc/hpt_once.h) compiled with the host compiler, for the tests.
#include "hpt_once.h"

#include <atomic>
#include <thread>

using namespace hpt;

// calls for the devices of 'dev' one after the other, failing the first time for device 'bad'; the status of each
// call, and how often the work ran
extern "C" int calls(int n, const int *dev, int bad, int *status)
{
    OncePerDevice once;
    int ran = 0;
    bool failed = false;
    for (int i = 0; i < n; ++i)
        status[i] = (int)once(dev[i], [&] {
            ++ran;
            if (dev[i] != bad || failed) return cudaSuccess;
            failed = true;
            return cudaErrorInvalidValue;
        });
    return ran;
}

// 'n' threads calling at once for one device: how often the work ran, and how many came back before it was done
extern "C" int together(int n, int *early)
{
    OncePerDevice once;
    std::atomic<int> ran{0}, done{0}, before{0};
    std::vector<std::thread> t;
    for (int i = 0; i < n; ++i)
        t.emplace_back([&] {
            (void)once(3, [&] {
                ++ran;
                std::this_thread::sleep_for(std::chrono::milliseconds(20));
                done = 1;
                return cudaSuccess;
            });
            before += !done;
        });
    for (auto &x : t) x.join();
    *early = before;
    return ran;
}
