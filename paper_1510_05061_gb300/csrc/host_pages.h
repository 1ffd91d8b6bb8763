// host_pages.h -- backs a host destination with pages before the device
// writes it.
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstdint>
#include <thread>
#include <vector>

namespace hydro {

// A destination that was only reserved (a new array) takes a page fault per
// page from the device's copy: 35 MB read back into a new numpy array took 10
// to 16 ms on GB300, into one whose pages exist 0.36 ms.  Populating the pages
// from a few host threads first takes 0.8 ms with the copy.  The contents do
// not change, and a range that cannot be populated (not mapped, read only) is
// left to the copy and its error.  Sampled pages decide whether there is
// anything to do (an array in use, pinned memory: no threads, 16 short system
// calls); small buffers are left alone.
inline void touch_pages(void *dst, size_t bytes)
{
#ifdef MADV_POPULATE_WRITE
    constexpr size_t MIN_BYTES = 2u << 20;
    if (!dst || bytes < MIN_BYTES) return;
    const long ps = sysconf(_SC_PAGESIZE);
    if (ps <= 0) return;
    const uintptr_t page = static_cast<uintptr_t>(ps), p0 = reinterpret_cast<uintptr_t>(dst), p1 = p0 + bytes;
    constexpr int SAMPLES = 16;
    bool all = true;
    for (int i = 0; i < SAMPLES && all; ++i) {
        const uintptr_t a = (p0 + (bytes - 1) / SAMPLES * i) / page * page;
        unsigned char in = 0;
        if (mincore(reinterpret_cast<void *>(a), 1, &in) != 0) return;   // not mapped
        all = (in & 1) != 0;
    }
    if (all) return;
    const auto touch = [page](uintptr_t a, uintptr_t b) {
        a = a / page * page;
        if (a < b) madvise(reinterpret_cast<void *>(a), b - a, MADV_POPULATE_WRITE);
    };
    const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
    const unsigned n = static_cast<unsigned>(std::min<size_t>(std::min(8u, hw), bytes / (MIN_BYTES / 2)));
    const uintptr_t step = (bytes + n - 1) / n;
    try {
        std::vector<std::thread> pool;
        pool.reserve(n);
        struct Join {
            std::vector<std::thread> &t;
            ~Join() { for (auto &x : t) x.join(); }
        } join{pool};
        for (unsigned i = 1; i < n; ++i) pool.emplace_back(touch, std::min(p1, p0 + i * step), std::min(p1, p0 + (i + 1) * step));
        touch(p0, std::min(p1, p0 + step));
    } catch (...) {
        // no threads or memory to be had: the copy takes its own faults
    }
#else
    (void)dst;
    (void)bytes;
#endif
}

}  // namespace hydro
