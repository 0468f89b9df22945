// Host work on many games by a few threads.
#pragma once

#include <algorithm>
#include <atomic>
#include <new>
#include <thread>
#include <vector>

namespace kps {

// fn(i) for every i in [0, n), on up to 8 threads, one for every 32768 hands (a
// thread costs about as much as the records of 5000 hands, and its first
// allocations as much again); the calling thread is one of them.  fn throws nothing but bad_alloc, which is passed on when all have
// ended.  Every i is independent of the others, so results do not depend on the
// threads.
template <typename F>
void parallel_for(int n, long long hands, F fn) {
    int threads = (int)std::min<long long>({8, n, hands / 32768});
    // (asking for the number of cores takes 15 us: one game's plan does not)
    if (threads > 1) threads = std::min(threads, (int)std::thread::hardware_concurrency());
    std::atomic<int> next{0};
    std::atomic<bool> failed{false};
    auto work = [&]() {
        for (int i; !failed && (i = next.fetch_add(1)) < n;) {
            try {
                fn(i);
            } catch (...) {
                failed = true;
            }
        }
    };
    std::vector<std::thread> others;
    try {
        if (threads > 1) others.reserve(threads - 1);
        for (int k = 1; k < threads; ++k) others.emplace_back(work);
    } catch (...) {   // as many as there are
    }
    work();
    for (std::thread &t : others) t.join();
    if (failed) throw std::bad_alloc();
}

}  // namespace kps
