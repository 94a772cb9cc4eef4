// bst_parallel.h -- a loop divided over host threads (plan tables).
#pragma once
#include <algorithm>
#include <exception>
#include <thread>

namespace bsth {

// fn(begin, end) over [0, n) in up to 8 host threads; on the calling thread alone
// where a thread cannot be started, be it for want of threads (std::system_error) or
// of memory (std::bad_alloc): threads that run are joined either way.  fn must not
// throw (it allocates nothing).
template <class F>
void parallel(int n, F&& fn) {
    constexpr int MOST = 8;
    std::thread t[MOST];
    const int most = std::min({MOST, n, (int)std::max(1u, std::thread::hardware_concurrency())});
    int at = 0, running = 0;
    for (int i = 0; i + 1 < most; ++i) {
        const int end = (int)((long long)n * (i + 1) / most);
        try {
            t[running] = std::thread([&fn, at, end] { fn(at, end); });
        } catch (const std::exception&) {
            break;
        }
        ++running;
        at = end;
    }
    fn(at, n);
    for (int i = 0; i < running; ++i) t[i].join();
}

}  // namespace bsth
