// Host side of the read-back: a parallel loop and the sort of the records that the device does
// not sort (few of them, or more than its 32-bit positions reach).
#pragma once

#include <stdint.h>

#include <algorithm>
#include <thread>
#include <vector>

namespace fstat {

// Runs f(t) for t in [0, nt) on nt threads (the calling thread takes t = 0, and what
// the system gives no thread for).
template <class Thread = std::thread, class Fn>
void parallel_for_threads(int nt, Fn f) {
    std::vector<Thread> th;
    th.reserve((size_t)nt);
    int own = nt;   // first slice without a thread
    for (int t = 1; t < nt; ++t) {
        try {
            th.emplace_back(f, t);
        } catch (...) {   // no thread, or no memory for its state: joinable threads must not be left behind
            own = t;
            break;
        }
    }
    f(0);
    for (int t = own; t < nt; ++t) f(t);
    for (auto &x : th) x.join();
}

// Sorts n records by (cell, bin), cells from cell0, bins from bin0, in `rec` with `tmp` as the other
// buffer: least-significant-digit counting passes of up to 11 bits over the key bits of
// the searched range, each thread counting and placing a run of the records.
template <class Rec>
void sort_records(Rec *rec, Rec *tmp, int64_t n, uint32_t cell0, uint32_t bin0, int bin_bits, int key_bits, int nt) {
    auto key = [&](const Rec &r) { return ((uint64_t)(r.cell - cell0) << bin_bits) | (r.bin - bin0); };
    if (n < 64) {
        std::sort(rec, rec + n, [&](const Rec &a, const Rec &b) { return key(a) < key(b); });
        return;
    }
    const int passes = std::max(1, (key_bits + 10) / 11), width = (key_bits + passes - 1) / passes;
    const uint64_t digits = uint64_t(1) << width, mask = digits - 1;
    std::vector<int64_t> at((size_t)nt * digits);   // [thread][digit]
    Rec *src = rec, *dst = tmp;
    for (int p = 0; p < passes; ++p) {
        const int shift = p * width;
        parallel_for_threads(nt, [&](int t) {
            int64_t *c = &at[(size_t)t * digits];
            std::fill(c, c + digits, 0);
            for (int64_t i = n * t / nt; i < n * (t + 1) / nt; ++i) ++c[(key(src[i]) >> shift) & mask];
        });
        int64_t sum = 0;
        for (uint64_t d = 0; d < digits; ++d)
            for (int t = 0; t < nt; ++t) {
                int64_t &c = at[(size_t)t * digits + d];
                const int64_t v = c;
                c = sum;
                sum += v;
            }
        parallel_for_threads(nt, [&](int t) {
            int64_t *c = &at[(size_t)t * digits];
            for (int64_t i = n * t / nt; i < n * (t + 1) / nt; ++i) dst[c[(key(src[i]) >> shift) & mask]++] = src[i];
        });
        std::swap(src, dst);
    }
    if (src != rec) std::copy(src, src + n, rec);
}

}  // namespace fstat
