// lbm_host.h -- host-side helpers of the CUDA library (not part of the ABI).
#pragma once

#include <algorithm>
#include <atomic>
#include <thread>
#include <vector>

namespace lbmk {

// f(t) for t in [0, n) on the host cores.  Returns false if an iteration threw
// (host allocation failure); f must not call set_error (its text is per thread).
template <class F>
bool host_parallel_for(int n, F&& f) {
    const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
    const int nt = std::max(1, std::min(n, (int)std::min(32u, hw)));
    std::atomic<int> next{0};
    std::atomic<bool> ok{true};
    auto work = [&]() {
        for (int t; (t = next.fetch_add(1)) < n;) {
            try {
                f(t);
            } catch (...) {
                ok = false;
            }
        }
    };
    std::vector<std::thread> pool;
    try {
        pool.reserve((size_t)nt - 1);
        for (int i = 0; i + 1 < nt; ++i) pool.emplace_back(work);
    } catch (...) {
        // no more threads to be had: those that started and this one do the work
    }
    work();
    for (std::thread& th : pool) th.join();
    return ok;
}

// Makes the pages of a large output array present, on the host cores, before a copy
// from the device overwrites it: fresh pages that the device meets first are mapped
// one small page at a time, which took up to 60 ms for 113 MB (a read before the
// write here would do the same).  For the two 13 MB outputs of the surrogate's
// prediction it costs more than it gives (3.6 against 2.8 ms a call of 1e5 inputs).
inline void touch_pages(void* p, size_t bytes) {
    constexpr size_t PIECE = size_t(2) << 20, PAGE = 4096;
    if (bytes < PIECE) return;
    volatile char* c = static_cast<volatile char*>(p);
    host_parallel_for((int)((bytes + PIECE - 1) / PIECE), [=](int i) {
        const size_t end = std::min(bytes, (size_t)(i + 1) * PIECE);
        for (size_t at = (size_t)i * PIECE; at < end; at += PAGE) c[at] = 0;
        c[end - 1] = 0;
    });
}

}  // namespace lbmk
