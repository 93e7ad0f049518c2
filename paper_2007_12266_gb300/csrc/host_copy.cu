// Results' way to the caller's host memory.
//
// A caller usually hands over freshly allocated memory, whose pages do not exist
// yet. The copy engine then takes a fault per page: 18-28 GB/s on a GB300 with a
// Grace host (280 MB), against 190 GB/s into pages that exist. So for large
// copies a few threads have the kernel populate the pages (MADV_POPULATE_WRITE:
// contents are not touched) chunk by chunk, and each chunk is copied as soon as
// its pages are there. Measured for 280 MB: 10.4-16 ms plain; populating alone 9.8,
// 4.9, 3.8 and 7.5 ms with 1, 2, 4 and 8 threads (the kernel's lock), so four.
// Buffers that are mostly resident already, and small ones, are copied as they
// are.
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <memory>
#include <thread>
#include <vector>

#include "internal.h"

#ifndef MADV_POPULATE_WRITE
#define MADV_POPULATE_WRITE 23
#endif

namespace lbm {

namespace {

constexpr size_t kPopulateFrom = size_t{8} << 20;   // smaller copies: starting threads costs what it saves
constexpr size_t kChunk = size_t{8} << 20;
constexpr int kThreads = 4;

// Whether at least half of the whole pages in [p, p + bytes) exist (then nothing
// is gained); also true when the system cannot tell.
bool mostly_resident(char* p, size_t bytes, size_t page) {
    std::vector<unsigned char> in((bytes + page - 1) / page);
    if (mincore(p, bytes, in.data()) != 0) return true;
    size_t n = 0;
    for (unsigned char c : in) n += c & 1;
    return 2 * n >= in.size();
}

// The copy in chunks, each after its pages were populated by one of the threads.
cudaError_t populate_and_copy(char* dst, const char* src, size_t bytes, size_t page, cudaStream_t s) {
    const size_t n = (bytes + kChunk - 1) / kChunk;
    std::vector<std::atomic<int>> done(n);
    std::atomic<size_t> next{0};
    auto work = [&] {
        for (size_t i; (i = next.fetch_add(1)) < n;) {
            // the chunk's bounds rounded out to pages: neighbouring data keeps its contents
            const size_t a = reinterpret_cast<size_t>(dst + i * kChunk) / page * page;
            const size_t e = (reinterpret_cast<size_t>(dst + std::min(bytes, (i + 1) * kChunk)) + page - 1) / page * page;
            madvise(reinterpret_cast<void*>(a), e - a, MADV_POPULATE_WRITE);   // where it fails, the copy populates
            done[i].store(1, std::memory_order_release);
        }
    };
    std::vector<std::thread> threads;
    struct Join {
        std::vector<std::thread>& t;
        ~Join() {
            for (auto& x : t) x.join();
        }
    } join{threads};
    threads.reserve(kThreads);
    for (int t = 0; t < kThreads; ++t) threads.emplace_back(work);
    cudaError_t e = cudaSuccess;
    for (size_t i = 0; i < n; ++i) {
        while (!done[i].load(std::memory_order_acquire)) std::this_thread::yield();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(dst + i * kChunk, src + i * kChunk, std::min(kChunk, bytes - i * kChunk),
                                cudaMemcpyDeviceToHost, s);
    }
    return e;
}

}  // namespace

cudaError_t copy_to_host(void* dst, const void* src, size_t bytes, cudaStream_t s) {
    char* const d = static_cast<char*>(dst);
    if (bytes >= kPopulateFrom) {
        const size_t page = static_cast<size_t>(std::max(4096L, sysconf(_SC_PAGESIZE)));
        char* const first = reinterpret_cast<char*>((reinterpret_cast<size_t>(d) + page - 1) / page * page);
        try {
            if (!mostly_resident(first, bytes - static_cast<size_t>(first - d), page))
                return populate_and_copy(d, static_cast<const char*>(src), bytes, page, s);
        } catch (...) {   // no memory or no thread to be had: the plain copy
        }
    }
    return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s);
}

}  // namespace lbm
