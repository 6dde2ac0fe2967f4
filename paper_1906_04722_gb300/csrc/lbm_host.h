// lbm_host.h -- host-side helpers of the CUDA library (not part of the ABI).
#pragma once

#include <sys/mman.h>
#include <unistd.h>

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

// Makes the pages of a large output array present, on the host cores, right before a
// copy from the device overwrites it (it writes to the array: only once nothing but that
// copy can fail): fresh pages that the device meets first are mapped one small page at a
// time, which took up to 60 ms for 113 MB (a read before the write here would do the
// same; madvise with MADV_POPULATE_WRITE, whose threads wait for each other: 5.7 against
// 3.1 ms for a whole read-out of 113 MB).  Pieces whose last page is present are left
// alone: starting threads for them costs more than it gives (a checkpoint of 48^3, 17 MB,
// into an array in use: 1.0 -> 0.5 ms).  For the two 13 MB outputs of the surrogate's
// prediction it costs more than it gives (3.6 against 2.8 ms a call of 1e5 inputs).
inline void touch_pages(void* p, size_t bytes) {
    constexpr size_t PIECE = size_t(2) << 20, STEP = 4096;
    if (bytes < PIECE) return;
    volatile char* c = static_cast<volatile char*>(p);
    const size_t page = (size_t)sysconf(_SC_PAGESIZE);
    std::vector<int> absent;
    const int pieces = (int)((bytes + PIECE - 1) / PIECE);
    try {
        for (int i = 0; i < pieces; ++i) {
            const size_t last = (size_t)p + std::min(bytes, (size_t)(i + 1) * PIECE) - 1;
            unsigned char present = 0;
            // (it fails where nothing is mapped, a device address for instance: the copy's to refuse)
            if (mincore(reinterpret_cast<void*>(last / page * page), page, &present) == 0 && !(present & 1))
                absent.push_back(i);
        }
    } catch (...) {
        return;  // a hint: the copy does without
    }
    host_parallel_for((int)absent.size(), [&](int k) {
        const size_t at = (size_t)absent[(size_t)k] * PIECE, end = std::min(bytes, at + PIECE);
        for (size_t b = at; b < end; b += STEP) c[b] = 0;
        c[end - 1] = 0;
    });
}

}  // namespace lbmk
