// Host threads for conversions of large host arrays.
#pragma once

#include <algorithm>
#include <cstddef>
#include <exception>
#include <thread>

namespace klb {

// Runs fn(begin, end) over [0, n) on up to 8 host threads, in pieces that
// touch at least 4 MB of host memory (`bytes` in all); fn must not throw.
// The host arrays of the box calls are tens of megabytes to gigabytes, and
// one core reaches a tenth of the memory's bandwidth (128x64x64 checkpoint,
// 314 MB: 18.2 ms on one core, 8.4 on four, 7.6 on eight, 8.1 on sixteen).
template <typename F>
void host_parallel(size_t n, size_t bytes, F fn)
{
    constexpr size_t kThreads = 8;
    size_t k = std::min({n, kThreads, bytes >> 22});
    if (k > 1) {
        static const size_t cores = std::max(1u, std::thread::hardware_concurrency());
        k = std::min(k, cores);
    }
    std::thread pool[kThreads];
    size_t done = 0, started = 0;
    if (k > 1) {
        try {
            for (; started < k - 1; ++started) {
                const size_t end = n * (started + 1) / k;
                pool[started] = std::thread(fn, done, end);
                done = end;
            }
        } catch (const std::exception &) {  // no thread, or no memory for one: the rest runs here
        }
    }
    fn(done, n);
    for (size_t t = 0; t < started; ++t) pool[t].join();
}

}  // namespace klb
