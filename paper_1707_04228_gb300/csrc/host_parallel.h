// Loops over the host's threads for the set-up's symbolic work.
#pragma once

#include <algorithm>
#include <atomic>
#include <exception>
#include <future>
#include <mutex>
#include <system_error>
#include <thread>
#include <utility>
#include <vector>

namespace gl {

// fn(0) .. fn(n - 1) on up to 32 threads, this one among them (alone, if no
// other can be had).  The first exception of any is thrown again here once all
// threads have ended; items not begun by then are left out.
template <class F>
void parallel_for(int n, F fn) {
    const int nt = std::min<int>(n, std::max(1u, std::min(std::thread::hardware_concurrency(), 32u)));
    std::atomic<int> next(0);
    std::exception_ptr first;
    std::mutex mu;
    auto work = [&]() {
        for (int i = next++; i < n; i = next++) {
            try {
                fn(i);
            } catch (...) {
                std::lock_guard<std::mutex> g(mu);
                if (!first) first = std::current_exception();
                next = n;
            }
        }
    };
    std::vector<std::thread> th;
    if (nt > 1) th.reserve(nt - 1);
    try {
        for (int t = 1; t < nt; ++t) th.emplace_back(work);
    } catch (...) {   // no further thread to be had: those there are do it
    }
    work();
    for (auto &t : th) t.join();
    if (first) std::rethrow_exception(first);
}

// fn() on a thread of its own, or, if there is none to be had, when its result is asked for.
template <class F>
auto in_background(F fn) -> std::future<decltype(fn())> {
    try {
        return std::async(std::launch::async, fn);
    } catch (const std::system_error &) {
        return std::async(std::launch::deferred, std::move(fn));
    }
}

}  // namespace gl
