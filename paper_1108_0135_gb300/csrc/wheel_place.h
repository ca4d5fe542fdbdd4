// Places and dense cut-offs of a wheel plan's entries (wheel.h): the arithmetic that
// the planner and its kernels share, free of CUDA so that a host program can run it.
//
// 64 neighbouring places share one dense cut-off, which no entry's floor(k/jlo)
// (k = floor(n/x), jlo = floor(X/x) + 1) may be below.  That is small for a target
// that is small against the others: with n = 1 in the group of the last entries of
// n = 10^15 the cut-off was 0, every j up to k was gathered, and j passed 2^32.  So
// targets are split into classes, each with whole groups of its own.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <vector>

#ifdef __CUDACC__
#define MERT_RULE __host__ __device__ __forceinline__
#else
#define MERT_RULE inline
#endif

namespace mert {

constexpr uint32_t kWheelGroup = 64;  // consecutive places with one dense cut-off

// Cut-offs from k / kWheelMaxJ + 6 on (down to a multiple of 6) keep every gathered j
// below 2^32 - 6.
constexpr uint64_t kWheelMaxJ = 4000000000u;

// Dense cut-off of a group: dc sqrt(mean k of its one-word entries), at least what
// keeps j in range for kf, its largest k; at most cap (its least floor(k/jlo): beyond
// it no term is left) and `listed`, the end of the dense list; down to a multiple of 6.
MERT_RULE uint64_t wheel_cutoff(double dc, double mean, uint64_t kf, uint64_t cap,
                                uint64_t listed)
{
    const uint64_t want = (uint64_t)(dc * sqrt(mean)), least = kf / kWheelMaxJ + 6;
    uint64_t yc = want > least ? want : least;
    yc = yc < cap ? yc : cap;
    return (yc < listed ? yc : listed) / 6 * 6;
}

// A bound of all cut-offs of groups whose k are at most k (before cap), a multiple of
// 4096: the dense list has to reach it.  The mean of a group, summed in double
// precision, is above k by at most a relative 2^-46, and dc sqrt(k) stays below 2^42,
// so the cut-off's whole part is at most one above that of dc sqrt(k).
MERT_RULE uint64_t wheel_cutoff_bound(double dc, uint64_t k)
{
    const uint64_t want = (uint64_t)(dc * sqrt((double)k)), least = k / kWheelMaxJ + 6;
    return ((want > least ? want : least) + 4096) / 4096 * 4096;
}

// An entry's last gathered j at cut-off yc.
MERT_RULE uint64_t wheel_last_j(uint64_t k, uint64_t yc, uint64_t jlo)
{
    const uint64_t j = k / (yc + 1);
    return j >= jlo ? j : jlo - 1;
}

struct WheelTarget {
    unsigned __int128 n;
    uint64_t u, X;
    bool lookup;      // read from a table: no terms
    uint32_t cls;     // result: its class
};

// A class of targets: the places [first, first + entries), first a multiple of
// kWheelGroup.
struct WheelClass {
    uint64_t first, entries;
};

// Splits the targets into classes.  For every entry of target i floor(k/jlo) is at
// least n/(2X) (k/jlo = floor(floor(n/x) / (floor(X/x) + 1)), and x (floor(X/x) + 1)
// <= X + x <= 2X).  A class's head is the largest target left; a target joins it when
// its n/(2X) reaches the head's largest cut-off, dc sqrt(n), or -- limits near sqrt(n)
// and small targets bound every cut-off -- an eighth of the head's u, and in any case
// what keeps the head's j below 2^32.  So targets alike are one class, and a class's u
// (or, with one entry, n) are below a quarter of the last one's: 32 classes at most.
// With automatic limits targets below about 3 sqrt(n) are left out: 64 targets near
// 10^14 and requests from 10^10 to 10^15 are one class.  Targets with k up to
// `wide_from` have one-word entries.  Returns the classes with their places; *end is
// the first place after them all (lookups come there).
inline std::vector<WheelClass> wheel_classes(std::vector<WheelTarget> &t, double dc,
                                             unsigned __int128 wide_from, uint64_t *end)
{
    std::vector<WheelClass> out;
    std::vector<size_t> left, rest;
    for (size_t i = 0; i < t.size(); ++i)
        if (!t[i].lookup)
            left.push_back(i);
    uint64_t place = 0;
    while (!left.empty()) {
        size_t head = left[0];
        for (size_t i : left)
            if (t[i].n > t[head].n)
                head = i;
        const uint64_t k = (uint64_t)std::min(t[head].n, wide_from);
        const uint64_t least = k < kWheelMaxJ ? 0 : k / kWheelMaxJ + 12;
        const uint64_t want = std::max((uint64_t)(dc * std::sqrt((double)k)) + 12, least);
        const uint64_t thr = std::max(least, std::min(want, t[head].u / 8));
        place = (place + kWheelGroup - 1) / kWheelGroup * kWheelGroup;
        WheelClass c{place, 0};
        rest.clear();
        for (size_t i : left)
            if (i == head || t[i].n / (2 * (unsigned __int128)t[i].X) >= thr) {
                t[i].cls = (uint32_t)out.size();
                c.entries += t[i].X;
            } else {
                rest.push_back(i);
            }
        place += c.entries;
        out.push_back(c);
        left.swap(rest);
    }
    *end = place;
    return out;
}

}  // namespace mert
