// Loops over the host's threads, for the setup code.
#pragma once

#include <algorithm>
#include <atomic>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

namespace gcmg {

// f(0) .. f(n - 1), independent of each other, over at most `most` of the host's
// threads (a thread's share should outweigh its start).  An exception of one reaches
// the caller after all threads have ended; a thread that cannot be had is done
// without.  (Neither may leave a thread's function or a joinable thread behind: both
// end the process.)
template <typename F>
void for_each_index(int n, size_t most, F &&f) {
    std::atomic<int> next{0};
    std::mutex lock;
    std::exception_ptr error;
    auto work = [&]() {
        try {
            for (int i = next++; i < n; i = next++) f(i);
        } catch (...) {
            next = n;
            std::lock_guard<std::mutex> g(lock);
            if (!error) error = std::current_exception();
        }
    };
    std::vector<std::thread> pool;
    try {
        const unsigned nt = std::min({(unsigned)std::min<size_t>(most, 16), (unsigned)n, std::thread::hardware_concurrency()});
        for (unsigned t = 1; t < nt; t++) pool.emplace_back(work);
    } catch (...) {   // fewer threads then
    }
    work();
    for (auto &t : pool) t.join();
    if (error) std::rethrow_exception(error);
}

}  // namespace gcmg
