// threads.h -- a loop split over host threads.
#pragma once

#include <stdint.h>

#include <exception>
#include <mutex>
#include <thread>
#include <vector>

namespace titan {

// Calls part(0) .. part(n - 1), each on a thread of its own while threads can be had
// and on this one otherwise, waits for all of them and then rethrows the first
// exception any of them threw.
template <class F>
void run_parts(uint32_t n, F &&part) {
    std::exception_ptr first;
    std::mutex mu;
    auto guarded = [&](uint32_t t) {
        try {
            part(t);
        } catch (...) {
            std::lock_guard<std::mutex> lk(mu);
            if (!first) first = std::current_exception();
        }
    };
    std::vector<std::thread> pool;
    uint32_t t = 1;
    try {
        if (n > 1) pool.reserve(n - 1);
        for (; t < n; ++t) pool.emplace_back(guarded, t);
    } catch (...) {                          // no memory or no thread to be had: the rest on this one
    }
    for (; t < n; ++t) guarded(t);
    if (n) guarded(0);
    for (auto &th : pool) th.join();
    if (first) std::rethrow_exception(first);
}

}  // namespace titan
