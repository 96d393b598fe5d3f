// Host-side helpers: planning work on a few threads, and the guard of the C entry points.
#pragma once

#include <algorithm>
#include <new>
#include <stdexcept>
#include <thread>
#include <vector>

#include "csb_internal.hpp"

namespace csb {

// Runs `work` on at most `most` threads, the calling one among them, and waits for all; on fewer where no more are to be
// had.  `work` takes its share from a counter of its own and throws nothing.
template <typename F>
void run_on_threads(int most, F&& work) {
    const unsigned hw = std::thread::hardware_concurrency();
    const int n = std::min(most, (int)(hw ? hw : 1));
    std::vector<std::thread> pool;
    try {
        if (n > 1) pool.reserve((size_t)n - 1);
        while ((int)pool.size() + 1 < n) pool.emplace_back([&work]() { work(); });
    } catch (const std::exception&) {}                     // no memory or no thread: those that run do all of it
    work();
    for (std::thread& t : pool) t.join();
}

// No exception crosses a C entry point.
template <typename F>
int guarded(F&& f) {
    try { return f(); }
    catch (const std::exception&) { set_error("out of host memory"); return CSB_ERR_ALLOC; }   // allocations are all that throws here
}

}  // namespace csb
