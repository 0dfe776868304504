// A result array's pages made present by several threads.
//
// A read-out usually lands in memory that was just allocated: the copy then
// faults every page in, one at a time, at 25 GB/s where the copy itself runs at
// 180 (403 MB: 14.7 ms).  Four threads asking for the pages ahead of the copy take
// 4.6 ms for the same array, and the copy of a part starts once that part is
// there (256^3 velocity 16.5 -> 6.7 ms, populations 109 -> 33).
#pragma once

#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <memory>
#include <thread>
#include <vector>

namespace kin {

class HostPages {
public:
    // Arrays below kLeast are left to the copy.  A copy takes a part once its pages are
    // there: parts of 8 MB 128^3 velocity 1.21 ms, 160^3 1.99 (16 MB 1.39 and 2.15, 2 MB
    // 1.21 and 2.13).
    static constexpr size_t kLeast = size_t(32) << 20, kPart = size_t(8) << 20;
    // Threads, and bytes asked for at a time.  403 MB, pages alone: four threads 4.6 ms,
    // eight 14 (they wait for each other in the kernel); four with ranges of 64 KB
    // 5.7, of 16 MB 5.1.  With the copy: two threads 9.2, three 7.3, four 6.9.
    static constexpr size_t kThreads = 4;
    static constexpr size_t kRange = size_t(1) << 20;

    // [p, p + bytes) is about to be overwritten.  Below 32 MB, or where the pages
    // are there already, nothing is done (6 MB: 0.35 ms either way).
    HostPages(void* p, size_t bytes) : p_(static_cast<char*>(p)), bytes_(bytes) {
        if (bytes < kLeast || resident()) return;
        const size_t parts = (bytes + kPart - 1) / kPart;
        const unsigned cores = std::max(1u, std::thread::hardware_concurrency());
        const size_t threads = std::min<size_t>({kThreads, parts, std::max(1u, cores / 2)});
        try {
            done_.reset(new std::atomic<bool>[parts]);
            for (size_t k = 0; k < parts; ++k) done_[k].store(false, std::memory_order_relaxed);
            parts_ = parts;
            threads_.reserve(threads);
            for (size_t k = 0; k < threads; ++k) threads_.emplace_back([this] { work(); });
        } catch (...) {
            // fewer threads, or none: the copy faults the pages in itself
        }
    }
    HostPages(const HostPages&) = delete;
    HostPages& operator=(const HostPages&) = delete;
    ~HostPages() {
        next_.store(parts_);  // nothing new is started
        for (std::thread& t : threads_) t.join();
    }

    // Whether threads are at work on the pages.
    bool pending() const { return !threads_.empty(); }

    // Returns once [p, p + end) may be overwritten.
    void wait(size_t end) const {
        if (!pending()) return;
        const size_t parts = std::min(parts_, (end + kPart - 1) / kPart);
        for (size_t k = 0; k < parts; ++k)
            while (!done_[k].load(std::memory_order_acquire)) std::this_thread::yield();
    }

private:
    static size_t page() {
        static const long v = sysconf(_SC_PAGESIZE);
        return v > 0 ? (size_t)v : 4096;
    }
    // Eight pages spread over the array are in memory (or it cannot be told).
    bool resident() const {
        for (int k = 0; k < 8; ++k) {
            const uintptr_t a = (reinterpret_cast<uintptr_t>(p_) + bytes_ / 8 * k) / page() * page();
            unsigned char in = 0;
            if (mincore(reinterpret_cast<void*>(a), 1, &in) != 0) return true;
            if (!(in & 1)) return false;
        }
        return true;
    }
    // Make the pages of [a, end) present for writing, without a store of our own: what
    // they hold stays, should the read-out fail.  Memory that may not be written, or
    // is not there, ends the call with an error; the copy meets it and returns its own.
    static void populate(char* a, char* end) {
#ifdef MADV_POPULATE_WRITE
        const uintptr_t at = reinterpret_cast<uintptr_t>(a) / page() * page();
        (void)madvise(reinterpret_cast<void*>(at), reinterpret_cast<uintptr_t>(end) - at, MADV_POPULATE_WRITE);
#else
        (void)a;
        (void)end;
#endif
    }
    void work() {
        for (size_t k; (k = next_.fetch_add(1)) < parts_;) {
            char* const end = p_ + std::min(bytes_, (k + 1) * kPart);
            for (char* a = p_ + k * kPart; a < end; a += kRange) populate(a, std::min(end, a + kRange));
            done_[k].store(true, std::memory_order_release);
        }
    }

    char* p_;
    size_t bytes_, parts_ = 0;
    std::unique_ptr<std::atomic<bool>[]> done_;
    std::atomic<size_t> next_{0};
    std::vector<std::thread> threads_;
};

}  // namespace kin
