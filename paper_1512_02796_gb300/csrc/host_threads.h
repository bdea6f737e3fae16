// Host threads of the mesh and multigrid plans (internal).
#pragma once

#include <algorithm>
#include <cstdint>
#include <exception>
#include <mutex>
#include <system_error>
#include <thread>
#include <vector>

namespace qpat {

inline int host_threads() {
    const unsigned h = std::thread::hardware_concurrency();
    return int(std::max(1u, std::min(h, 16u)));
}

// fn(t, begin, end) over nt contiguous ranges of [0, n), each on its own thread
// (or, where the system gives no more threads, on this one).  An exception of
// a range (memory) is thrown again here once all of them have ended.
template <typename F>
void parallel_ranges(int64_t n, int nt, const F& fn) {
    if (nt <= 1) {
        fn(0, int64_t(0), n);
        return;
    }
    std::mutex mu;
    std::exception_ptr error;
    auto range = [&](int t) {
        try {
            fn(t, n * t / nt, n * (t + 1) / nt);
        } catch (...) {
            std::lock_guard<std::mutex> lock(mu);
            if (!error) error = std::current_exception();
        }
    };
    std::vector<std::thread> threads;
    threads.reserve(size_t(nt));
    for (int t = 0; t < nt; ++t) {
        try {
            threads.emplace_back(range, t);
        } catch (const std::exception&) {  // no thread, or no memory for one
            range(t);
        }
    }
    for (auto& x : threads) x.join();
    if (error) std::rethrow_exception(error);
}

}  // namespace qpat
