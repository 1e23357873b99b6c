// A loop over a few host threads.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <new>
#include <thread>
#include <vector>

namespace softsim {

// f(i) for i in [0, n), the indices handed out in blocks to a few threads
// (every f writes its own outputs only).  What an f throws is thrown again here.
// work_size: vertices behind all of it (1-2 us of work each); a thread costs tens
// of microseconds to start, so it is given at least 512 of them.
template <typename F>
void parallel_for(int64_t work_size, int64_t n, int64_t block, F f)
{
    const int64_t n_blocks = (n + block - 1) / block;
    const int n_thr = (int)std::min<int64_t>(
        {n_blocks, work_size / 512 + 1, (int64_t)std::max(1u, std::thread::hardware_concurrency()), 16});
    std::atomic<int64_t> next(0);
    std::atomic<bool> failed(false);
    auto work = [&]() {
        try {
            for (int64_t b; !failed && (b = next.fetch_add(1)) < n_blocks;)
                for (int64_t i = b * block; i < std::min(n, (b + 1) * block); ++i) f(i);
        } catch (...) {
            failed = true;
        }
    };
    std::vector<std::thread> th;
    th.reserve(n_thr);
    try {
        for (int t = 1; t < n_thr; ++t) th.emplace_back(work);
    } catch (...) {  // no thread, or no memory to start one: fewer threads do
    }
    work();
    for (auto &t : th) t.join();
    if (failed) throw std::bad_alloc();
}

}  // namespace softsim
