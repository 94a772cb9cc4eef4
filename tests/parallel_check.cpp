// Test-only host program (compiled and run by tests/test_host_threads.py): the loop
// over host threads visits every index once, also where a thread cannot be started
// because its allocation fails.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include <vector>

#include "bst_parallel.h"

static std::atomic<int> left{1 << 30};   // allocations that succeed

void* operator new(std::size_t n) {
    if (left.fetch_sub(1) <= 0) throw std::bad_alloc();
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

int main() {
    for (int n : {0, 1, 2, 7, 8, 9, 1000})
        for (int ok = 0; ok <= 9; ++ok) {
            std::vector<std::atomic<int>> seen(n);
            left = ok;
            bsth::parallel(n, [&](int b, int e) {
                for (int i = b; i < e; ++i) ++seen[i];
            });
            left = 1 << 30;
            for (int i = 0; i < n; ++i)
                if (seen[i] != 1) {
                    std::printf("FAIL n=%d allocations=%d index %d visited %d times\n", n, ok, i, (int)seen[i]);
                    return 1;
                }
        }
    std::printf("OK\n");
    return 0;
}
