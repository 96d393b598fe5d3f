// Host-side helpers: planning work on a few threads, the guard of the C entry points, and that of a product's handle.
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

// What a product leaves behind when a wait of its kernel ran out stays with the handle.
inline int product_gave_up(const csb_matrix* A) {
    const ProductPlan& PP = A->product;
    if (!PP.h_status || *PP.h_status == 0) return CSB_OK;
    set_error("an earlier product on this handle gave up waiting on the device (code %u)", *PP.h_status);
    return CSB_ERR_TIMEOUT;
}

}  // namespace csb
