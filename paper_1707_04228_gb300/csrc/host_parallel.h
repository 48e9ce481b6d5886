// Loops over the host's threads for the set-up's symbolic work.
#pragma once

#include <algorithm>
#include <atomic>
#include <mutex>
#include <thread>
#include <vector>

#include "gl_internal.h"

namespace gl {

// fn(0) .. fn(n - 1) on up to 32 threads; the first Error of any is thrown again here.
template <class F>
void parallel_for(int n, F fn) {
    int nt = std::max(1u, std::min(std::thread::hardware_concurrency(), 32u));
    nt = std::min(nt, n);
    std::atomic<int> next(0);
    std::vector<std::thread> th;
    std::vector<Error> errs;
    std::mutex mu;
    for (int t = 0; t < nt; ++t)
        th.emplace_back([&]() {
            for (;;) {
                int i = next++;
                if (i >= n) break;
                try {
                    fn(i);
                } catch (const Error &e) {
                    std::lock_guard<std::mutex> g(mu);
                    errs.push_back(e);
                }
            }
        });
    for (auto &t : th) t.join();
    if (!errs.empty()) throw errs.front();
}

}  // namespace gl
