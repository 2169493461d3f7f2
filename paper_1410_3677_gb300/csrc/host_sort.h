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

// One digit of the key (cell - cell0) << bin_bits | (bin - bin0).  The loops over a run of
// records take everything by value: through references captured for the threads every record
// reloaded them (4032 records 32 -> 58 us).
struct KeyDigit {
    uint32_t cell0, bin0;
    int bin_bits, shift;
    uint64_t mask;
    template <class Rec>
    uint64_t operator()(const Rec &r) const {
        return ((((uint64_t)(r.cell - cell0) << bin_bits) | (r.bin - bin0)) >> shift) & mask;
    }
};
template <class Rec>
void count_run(const Rec *src, int64_t n, KeyDigit d, int64_t *at) {
    for (int64_t i = 0; i < n; ++i) ++at[d(src[i])];
}
template <class Rec>
void place_run(const Rec *src, int64_t n, KeyDigit d, int64_t *at, Rec *dst) {
    for (int64_t i = 0; i < n; ++i) dst[at[d(src[i])]++] = src[i];
}

// Sorts n records by (cell, bin), cells from cell0, bins from bin0, in `rec` with `tmp` as the other
// buffer: least-significant-digit counting passes of up to 11 bits over the key bits of
// the searched range, each thread counting and placing a run of the records.
template <class Rec>
void sort_records(Rec *rec, Rec *tmp, int64_t n, uint32_t cell0, uint32_t bin0, int bin_bits, int key_bits, int nt) {
    if (n < 64) {
        const KeyDigit key{cell0, bin0, bin_bits, 0, ~uint64_t(0)};
        std::sort(rec, rec + n, [key](const Rec &a, const Rec &b) { return key(a) < key(b); });
        return;
    }
    const int passes = std::max(1, (key_bits + 10) / 11), width = (key_bits + passes - 1) / passes;
    const uint64_t digits = uint64_t(1) << width;
    std::vector<int64_t> at((size_t)nt * digits);   // [thread][digit]
    int64_t *const all = at.data();
    Rec *src = rec, *dst = tmp;
    for (int p = 0; p < passes; ++p) {
        const KeyDigit d{cell0, bin0, bin_bits, p * width, digits - 1};
        std::fill(at.begin(), at.end(), 0);
        parallel_for_threads(nt, [=](int t) {
            const int64_t a = n * t / nt, b = n * (t + 1) / nt;
            count_run(src + a, b - a, d, all + (size_t)t * digits);
        });
        int64_t sum = 0;
        for (uint64_t k = 0; k < digits; ++k)
            for (int t = 0; t < nt; ++t) {
                int64_t &c = all[(size_t)t * digits + k];
                const int64_t v = c;
                c = sum;
                sum += v;
            }
        parallel_for_threads(nt, [=](int t) {
            const int64_t a = n * t / nt, b = n * (t + 1) / nt;
            place_run(src + a, b - a, d, all + (size_t)t * digits, dst);
        });
        std::swap(src, dst);
    }
    if (src != rec) std::copy(src, src + n, rec);
}

}  // namespace fstat
