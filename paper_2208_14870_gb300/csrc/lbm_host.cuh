// lbm_host.cuh -- host memory helpers of the batched and served paths.
//
// Callers' result arrays are often fresh (never written): the first write to
// each page then costs a fault, which a device-to-host copy or a single thread
// pays at about 20 GB/s, against 190 GB/s into pages that are there (GB300's
// host link; both measured).  The helpers spread copies, and the faults of a
// range about to be written, over a few threads.
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <cstring>
#include <thread>
#include <vector>

namespace lbm {

// f(begin, end) over [0, n) in pieces of `grain`, by up to eight threads where
// there is more than one piece (a thread that cannot be started is done without).
template <typename F>
inline void host_parallel(size_t n, size_t grain, F f) {
    const size_t pieces = (n + grain - 1) / grain;
    if (pieces <= 1) {
        if (n) f(size_t(0), n);
        return;
    }
    std::atomic<size_t> next{0};
    auto work = [&] {
        for (size_t p; (p = next.fetch_add(1)) < pieces;) f(p * grain, std::min(n, (p + 1) * grain));
    };
    std::vector<std::thread> team;
    const size_t want = std::min<size_t>({pieces, 8, std::max(1u, std::thread::hardware_concurrency())});
    try {
        for (size_t t = 1; t < want; ++t) team.emplace_back(work);
    } catch (...) {
    }
    work();
    for (auto& t : team) t.join();
}

inline void host_copy(void* dst, const void* src, size_t bytes) {
    host_parallel(bytes, size_t(1) << 20, [&](size_t b, size_t e) {
        std::memcpy(static_cast<char*>(dst) + b, static_cast<const char*>(src) + b, e - b);
    });
}

// Bring the pages of a range the caller is about to write into memory, without
// changing their contents (a kernel that does not know the request ignores it).
inline void host_populate(void* p, size_t bytes) {
#ifndef MADV_POPULATE_WRITE
    constexpr int MADV_POPULATE_WRITE = 23;
#endif
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE), b = ((uintptr_t)p + page - 1) / page * page,
                    e = ((uintptr_t)p + bytes) / page * page;
    if (e > b) madvise(reinterpret_cast<void*>(b), e - b, MADV_POPULATE_WRITE);
}

}  // namespace lbm
