// The wheel form of a whole run: the sums over integers coprime to 6 only.
//
// Let M6(v) = sum of mu(m) over m <= v coprime to 6.  Multiplying the
// zeta function by its Euler factors at 2 and 3 in the identity of Sec. 2
// (arXiv:1108.0135) gives, for every v >= 1,
//   sum over j >= 1 coprime to 6 of M6(floor(v/j)) = 1,
// and M(v) = M6(v) - M6(v/2) - M6(v/3) + M6(v/6) (floors; every m splits
// uniquely into a divisor of 6 times a part coprime to 6 when m is
// squarefree).  So the sieve, the gathered terms and the dense terms of the
// method run over a third of the integers, and a last pass turns M6 of the
// array entries into M.
//
// Integers coprime to 6 are numbered w = 0, 1, 2, ...: y(w) = 3w + 1 + (w & 1)
// (6i + 1 at w = 2i, 6i + 5 at w = 2i + 1).  phi6(v) counts those <= v.
#pragma once

#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

#include "common.cuh"
#include "internal.h"
#include "wheel_place.h"

namespace mert {

// y of one segment (2048 wheel numbers): every block starts at a multiple.
constexpr uint64_t kWheelSegY = 3ull * kSegY;
// y of a shared-memory gather tile (32768 wheel numbers, 64 KiB of int16).
constexpr uint64_t kWheelTileY = 3ull * kGatherTile;

// Number of integers in [1, v] coprime to 6: v = 6i + r has 2i + [r >= 1] +
// [r >= 5].
__host__ __device__ __forceinline__ uint64_t phi6(uint64_t v)
{
    const uint64_t i = v / 6, r = v - 6 * i;
    return 2 * i + (r >= 1 ? 1u : 0u) + (r >= 5 ? 1u : 0u);
}

// The same for v < 2^32 - 5: with the even part e of v + 5, e / 3 - 1.
__host__ __device__ __forceinline__ uint32_t phi6_u32(uint32_t v)
{
    return ((v + 5u) & ~1u) / 3u - 1u;
}

// Index of the last wheel number <= v relative to a multiple of 6 (1 <= v <
// 2^32): phi6(v) - 1 = floor(((v - 1) & ~1) / 3).
__host__ __device__ __forceinline__ uint32_t wheel_index(uint32_t v)
{
    return ((v - 1u) & ~1u) / 3u;
}

__host__ __device__ __forceinline__ uint64_t wheel_y(uint64_t w) { return 3 * w + 1 + (w & 1); }

// Wheel numbers per element of Mg.
constexpr uint32_t kMgShift = 4;

#ifdef __CUDACC__
// The part of M6 at wheel index i of a block that its Mg holds.
__device__ __forceinline__ int wheel_value(const uint2 *Mg, uint64_t i)
{
    const uint2 v = Mg[i >> kMgShift];
    const uint32_t upto = (2u << ((uint32_t)i & 15u)) - 1u;  // bits 0 .. i mod 16
    return (int)v.y + __popc(v.x & upto) - 2 * __popc((v.x >> 16) & upto);
}
#endif

// ---- sieve ------------------------------------------------------------------
// Sieving primes and scratch of a wheel sieve (device arrays, primes >= 5), all
// in one piece of memory of its owner.
struct WheelSieve {
    std::vector<uint32_t> host_p;  // primes 5 <= p <= P (2 and 3 are left out)
    uint32_t *p = nullptr;         // the same on the device
    uint4 *pat = nullptr;       // phase copies of the small primes' pattern
    uint4 *rec = nullptr;       // per block, see wheel_prep_kernel
    uint2 *rec2 = nullptr;
    uint32_t *sqcnt = nullptr, *sqlist = nullptr, *err = nullptr;
};

// One block: wheel numbers [w0, w0 + len), both multiples of kSegY.
//   M6(y(w)) = segoff[i >> kSegShift] + wheel_value(Mg, i), i = w - w0
// Mg holds 8 bytes per 16 numbers (0.5 bytes per number; int16 values took four
// times as much, and the sieve's decode was bound by writing them): x = the
// squarefree ones as 16 bits, those with mu = -1 in the high half; y = M6 before
// the 16 relative to the segment.
struct WheelLaunch {
    uint64_t w0 = 0, len = 0;
    uint2 *Mg = nullptr;
    int32_t *segsum = nullptr;
    int64_t *segoff = nullptr;
    const int64_t *carry_in = nullptr;  // device M6(y(w0) - 1)
    int64_t *carry_out = nullptr;       // device M6 of the block's end
    cudaEvent_t mid = nullptr, mid2 = nullptr;  // profiling: after a1, before a2
};

// Host part: the primes for blocks below y_max < 2^54 (up to its square root, at
// least 1024).
void wheel_sieve_primes(WheelSieve *t, uint64_t y_max);
// Device bytes for blocks of up to max_len wheel numbers; the same memory (256-
// byte aligned) split up, with the scratch cleared and the pattern made on `s`
// (the caller fills t->p from t->host_p).  The kernels set kErrTimeout and
// kErrList in *err.
size_t wheel_sieve_bytes(const WheelSieve *t, uint64_t max_len);
constexpr uint32_t kErrList = 4u;  // a square list overflowed its capacity
constexpr uint32_t kErrJ = 32u;    // a plan's gathered j beyond 32 bits
int wheel_sieve_bind(WheelSieve *t, void *base, uint64_t max_len, uint32_t *err, cudaStream_t s);
uint32_t wheel_primes_upto(const WheelSieve *t, uint64_t b);
int wheel_sieve_enqueue(const WheelSieve *t, const WheelLaunch &L, cudaStream_t s);
bool wheel_sieve_exact(uint64_t y_max);

// ---- plan -----------------------------------------------------------------------
constexpr uint32_t kWheelGroupBlock = 8;   // groups of a dense work item; the first
                                           // eight groups are items of their own (their
                                           // k is large: more terms take a slow form)
__host__ __device__ constexpr uint32_t wheel_group_blocks(uint32_t groups)
{
    return groups <= kWheelGroupBlock ? groups
                                      : kWheelGroupBlock + (groups - 1) / kWheelGroupBlock;
}
// First group of group block b (b = their number: at least `groups`).
__host__ __device__ constexpr uint32_t wheel_block_first(uint32_t b)
{
    return b < kWheelGroupBlock ? b : (b - kWheelGroupBlock + 1) * kWheelGroupBlock;
}
constexpr uint32_t kWheelItem = 256;       // wheel indices of a chunk of the global gather

// A target; n = 0: its value is read from a table (one entry, no terms).  Its
// entries x = 1 .. X are numbered off + x - 1 in the results; the update works on
// places: the same numbers for one target; for several, the entries of a class of
// targets (wheel_place.h) in decreasing order of k (so that 64 consecutive places
// have close k), class after class.
struct WheelQuery {
    uint64_t n, n_hi, X;
    uint64_t off, goff;     // first entry, first group of 64 entries
    uint64_t place;         // in order of k: the class's first place; else the target's
    uint64_t cls;           // its class
};

struct WheelGroup {
    uint32_t first, count;  // places
    uint64_t yc;            // dense cut-off (a multiple of 6)
    uint64_t kmax;          // largest k of the group
};

struct WheelGatherTile {
    uint64_t t0;            // y in [t0 + 1, t0 + len], t0 a multiple of 6
    uint64_t m1, m2;        // division magics of t0 + 1 and t0 + len + 1
    uint32_t len, l1, l2, pad;
};

// Totals of a target, made with the entries (WheelQuery order).
struct WheelTotals {
    unsigned long long direct, gathered;  // the method's terms (closed forms)
    unsigned long long gather_j;          // gathered terms at the dense cut-offs
    unsigned long long exec;              // those with j coprime to 6
    unsigned long long dense_y;           // y below the cut-offs, over the entries
};

struct WheelEntryArgs {
    const WheelQuery *qs;
    uint32_t nq;
    uint32_t nplaces;       // places: the entries, and unused ones (k = 0) after a class
    uint32_t qgroups;       // groups of 64 entries, target by target
    uint32_t ngroups;       // groups of 64 places
    double dc;              // dense cut-off factor
    uint64_t ydense;        // end of the dense list
    uint32_t *err;          // kErrJ when a gathered j did not fit 32 bits
    uint64_t wide_from;     // entries with k at or above: two-word ones (k = 0 here)
    uint32_t *P;            // place of every entry (null: the entry's number)
    uint32_t by_k;          // places in decreasing order of k
    uint64_t *K, *YC;
    uint32_t *JL, *JD;
    WheelGroup *groups;
    WheelTotals *totals;    // cleared
    uint32_t parts;         // parts of a dense chunk's list
    uint32_t *dpre;         // first dense item of every group block, then their number
    WheelGatherTile *tiles;
    const uint2 *tile_src;  // {first y / 6, len} of every tile
    uint32_t ntiles;
};
// Entries, groups, totals, the dense work items' prefix sums and the gather
// tiles' division constants of a plan.
int wheel_entries_enqueue(const WheelEntryArgs &a, cudaStream_t s);

// ---- update -------------------------------------------------------------------
constexpr int kWheelDenseThreads = 256;

struct WheelDenseArgs {
    uint32_t *counter;
    const WheelGroup *groups;
    uint32_t ngroups, parts;
    const uint32_t *pre;    // see WheelEntryArgs::dpre
    const uint64_t *K;
    const uint16_t *dl;     // kSegY offsets per chunk: mu = +1, then mu = -1
    const uint32_t *dl_cnt; // count(+1) | count(-1) << 16
    uint64_t *S;
};

struct WheelGatherArgs {
    uint64_t y0;            // block start: wheel index 0 of Mg is y0 + 1
    const WheelGatherTile *tiles;
    const uint4 *items;     // {tile, e0, e1, 0}
    uint32_t nitems;
    uint32_t *counter;
    const uint2 *Mg;
    const int64_t *segoff;
    const uint64_t *K, *YC;
    const uint32_t *JL, *JD;
    uint64_t *S;
    uint32_t long_lane;     // a lane sums fewer terms of an entry than this
    uint32_t all_long;      // 64-bit remainders for every term
};

// One block (y0, y0 + len] of the global-memory path.
struct WheelBlockArgs {
    uint64_t y0, len;
    uint64_t ylo;           // first y of the global path in the block
    uint64_t m_ylo, m_end;  // division magics of ylo and y0 + len + 1
    uint32_t l_ylo, l_end;
    uint64_t kmax;          // entries with k >= kmax take the block's tiles
    uint64_t nplaces;
    const uint64_t *K, *YC;
    const uint32_t *JL, *JD;
    uint64_t *S, *A;
    uint4 *queue;
    uint32_t *qlen;
    uint32_t qcap;
    uint32_t *err;
    const uint2 *Mg;
    const int64_t *segoff;
};

int wheel_dense_list_enqueue(const uint2 *Mg, uint64_t c0, uint64_t nchunks, uint16_t *dl,
                             uint32_t *dl_cnt, cudaStream_t s);
int wheel_dense_enqueue(const WheelDenseArgs &a, uint64_t max_items, cudaStream_t s);
int wheel_gather_enqueue(const WheelGatherArgs &a, cudaStream_t s);
int wheel_block_enqueue(const WheelBlockArgs &a, cudaStream_t s);

// Entries with k >= 2^63 (k = 0 in the arrays above), with 128-bit quotients: the
// direct terms M6(y) (phi6(floor(k/y)) - phi6(floor(k/(y+1)))) of the y <= s, which
// telescope over the y between two wheel numbers, and the gathered terms j in
// [jlo, jhi] coprime to 6 (update.h's WheelEntry fields); and the values of M
// with an argument floor(k/m) in the block, m = 2, 3, 6.
struct WideEntry;
struct WheelWideArgs {
    const WideEntry *W;
    uint64_t y0, len;
    const uint2 *Mg;
    const int64_t *segoff;
    uint64_t *S, *A;
};
// Terms of entry W in the block (y0, y0 + len]: `direct` wheel numbers, then the
// wheel indices [wj, wj + gathered).
void wheel_wide_units(const WideEntry &W, uint64_t y0, uint64_t len, uint64_t *direct,
                      uint64_t *wj, uint64_t *gathered);
int wheel_wide_enqueue(const WheelWideArgs &a, uint32_t nw, uint64_t units, cudaStream_t s);

// Reads of a resident table (Mg and segoff from y = 0 on): M(y) of (entry, y)
// pairs into R; M6(y0) into *out (y0 a multiple of a segment, > 0).
int wheel_lookup_enqueue(const uint64_t *pairs, uint32_t count, const uint2 *Mg,
                         const int64_t *segoff, uint64_t *R, cudaStream_t s);
int wheel_carry_at_enqueue(const uint2 *Mg, const int64_t *segoff, uint64_t y0, int64_t *out,
                           cudaStream_t s);

struct QueryDev;
// R6[x] = M6(floor(n/x)) from the sums S, then M in R (A: the parts of M whose
// M6 argument lies below the array; S and A by place).
int wheel_resolve_enqueue(const QueryDev *qs, uint32_t nq, uint64_t max_x, const uint32_t *P,
                          const uint64_t *S, const uint64_t *A, uint64_t *R6, uint64_t *R,
                          cudaStream_t s);

}  // namespace mert
