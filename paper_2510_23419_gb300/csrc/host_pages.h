// host_pages.h -- pages of large host outputs made present before a device-to-host copy.
//
// Large outputs usually are fresh memory whose pages do not exist yet.  A copy that takes their first faults one by
// one ran at 14 GB/s, into present pages at 180 GB/s (33.5 MB: 2.4 against 0.19 ms), so the missing pages are
// populated on four host threads first (more did not help): 1.1 ms with the copy, 1.6 when the threads wrote a byte
// to every page instead.  Contents do not change, so a copy that fails leaves the
// buffer as it was, and memory that cannot be populated (not mapped here, read-only, a driver's own) is left to the
// copy.  From 32 MB on, where the C library's allocator maps fresh memory for every request; smaller
// buffers are mostly reused ones.  Reused and pinned buffers of that size cost one look at the page tables (copy and
// all 0.22 ms; 0.31 with a byte written to every page).
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <exception>
#include <thread>
#include <vector>

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif

namespace pb {

// Returns the number of host threads that populated pages (0: nothing to do).
inline int populate_pages(void* out, size_t bytes)
{
    constexpr size_t kMin = (size_t)32 << 20;
    if (bytes < kMin) return 0;
    const size_t page = (size_t)sysconf(_SC_PAGESIZE);
    const uintptr_t first = (uintptr_t)out / page * page;
    const size_t pages = ((uintptr_t)out + bytes - first + page - 1) / page;
    // the pages that are not there, at a sample of them: fresh memory has none, used memory all
    constexpr size_t kSamples = 64;
    size_t missing = 0;
    for (size_t k = 0; k < kSamples; ++k) {
        unsigned char here = 0;
        if (mincore((void*)(first + (pages - 1) * k / (kSamples - 1) * page), page, &here) != 0) return 0;
        missing += !(here & 1);
    }
    if (missing == 0) return 0;
    const int threads = (int)std::min(4u, std::max(1u, std::thread::hardware_concurrency()));
    auto populate = [&](size_t b, size_t e) {
        if (e > b) (void)madvise((void*)(first + b * page), (e - b) * page, MADV_POPULATE_WRITE);
    };
    std::vector<std::thread> ts;
    size_t done = 0;  // pages [0, done) have a thread of their own
    try {
        ts.reserve((size_t)threads);
        for (int k = 0; k + 1 < threads; ++k) {
            const size_t e = pages * (size_t)(k + 1) / (size_t)threads;
            ts.emplace_back(populate, done, e);
            done = e;
        }
    } catch (const std::exception&) {
        // no more threads to be had: the rest is populated here
    }
    populate(done, pages);
    for (std::thread& t : ts) t.join();
    return 1 + (int)ts.size();
}

}  // namespace pb
