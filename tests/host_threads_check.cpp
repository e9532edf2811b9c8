// Test program (built and run by tests/test_host_threads.py): for_each_index
// calls every index once, and an exception of any of them reaches the caller with
// every thread ended.  Exits 0 if so.
#include <atomic>
#include <cstdio>
#include <new>
#include <stdexcept>
#include <vector>

#include "host_threads.h"

int main() {
    long bad = 0;
    for (int n : {0, 1, 2, 7, 100, 5000})
        for (size_t most : {(size_t)0, (size_t)1, (size_t)3, (size_t)16, (size_t)400}) {
            std::vector<std::atomic<int>> seen(n + 1);
            gcmg::for_each_index(n, most, [&](int i) { seen[i]++; });
            for (int i = 0; i < n; i++) bad += seen[i] != 1;
            for (int at : {0, n / 2, n - 1}) {
                if (at < 0 || at >= n) continue;
                for (auto &x : seen) x = 0;
                int caught = 0;
                try {
                    gcmg::for_each_index(n, most, [&](int i) {
                        seen[i]++;
                        if (i == at) throw std::bad_alloc();
                        if (i == at + 1) throw std::runtime_error("second");
                    });
                } catch (const std::exception &) {
                    caught = 1;
                }
                bad += !caught;
                for (int i = 0; i < n; i++) bad += seen[i] > 1;
            }
        }
    std::printf("%ld\n", bad);
    return bad ? 1 : 0;
}
