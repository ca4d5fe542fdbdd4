// Steps a3 (update) and a4 (resolve) of a whole run over the integers coprime
// to 6 (wheel.h).
//
// Entry x of a target n has k = floor(n/x); its M6(k) is 1 minus the sum of
// M6(floor(k/j)) over j >= 2 coprime to 6.  The terms with j <= floor(X/x) are
// other entries (resolve); those with floor(X/x) < j <= jd are gathered one by
// one; the rest, where floor(k/j) <= yc, are the dense part
//   sum over y <= yc coprime to 6 of mu(y) (phi6(floor(k/y)) - phi6(jd))
// (exchange the order of summation: phi6(floor(k/y)) - phi6(jd) counts the
// j > jd coprime to 6 with floor(k/j) >= y), whose second part is
// -M6(yc) phi6(jd).  jd = max(floor(k/(yc + 1)), floor(X/x)).
//
// phi6 of a quotient without the quotient: with Y(w) = 3w + 1 + (w & 1) =
// (3w + 1) | 1 the wheel numbers and T near k / (3y),
//   phi6(floor(k/y)) = T + [k >= y Y(T)]
// whenever Y(T - 1) <= k/y < Y(T + 1), which holds for -1/3 <= k/(3y) - T < 4/3
// (T even: 3T - 1 <= k/y < 3T + 5, T odd: 3T - 2 <= k/y < 3T + 4).  So the floor
// of an estimate of k/(3y) that errs by less than 1/3 is exact, and one 32-bit
// multiply-subtract and its sign bit give phi6.
#include <algorithm>
#include <cstdint>

#include "update.h"
#include "wheel.h"

namespace mert {

// A float estimate plus 1.5 2^23, rounded down, has the bits kMagicBits + its
// floor.
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr float kMagicF = 12582912.0f;

// Y(T) from the biased bits.
__device__ __forceinline__ uint32_t wheel_of_bits(uint32_t bits)
{
    return (3u * bits + (1u - 3u * kMagicBits)) | 1u;
}

// v as a float (relative error at most 2^-23) by two 32-bit conversions (a 64-bit
// one runs on the FP64 pipe here).
__device__ __forceinline__ float float_u64(uint64_t v)
{
    return __fmaf_rn(__uint2float_rn((uint32_t)(v >> 32)), 4294967296.0f,
                     __uint2float_rn((uint32_t)v));
}

// ---------------------------------------------------------------------------
// Plan: the entries of every target, a warp per group of 64 (two per lane).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t isqrt_dev(uint64_t v)
{
    uint64_t r = (uint64_t)sqrt((double)v);
    while (r * r > v)
        --r;
    while ((r + 1) * (r + 1) <= v)
        ++r;
    return r;
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Every entry's k = floor(n/x) and first gathered j, at its place, and the totals
// of the full sums (a warp per 64 entries of a target): gather_j counts the
// gathered terms of the full sums' dense cut-offs, dc sqrt(k of the first
// one-word entry), up to a multiple of 4096 less one, within [floor(sqrt(k)),
// floor(k/jlo) - 1].
__global__ void __launch_bounds__(128) wheel_entries_kernel(WheelEntryArgs a)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= a.qgroups)
        return;
    uint32_t lo_q = 0, hi_q = a.nq;  // the last target with goff <= g
    while (hi_q - lo_q > 1) {
        const uint32_t mid = (lo_q + hi_q) >> 1;
        if (a.qs[mid].goff <= g)
            lo_q = mid;
        else
            hi_q = mid;
    }
    const WheelQuery Q = a.qs[lo_q];
    const uint64_t x0 = (g - Q.goff) * kWheelGroup + 1;
    const uint32_t cnt = (uint32_t)min((uint64_t)kWheelGroup, Q.X - x0 + 1);
    uint64_t k[2], sq[2], vh[2], jlo[2];
    uint64_t lo = 0, nhi = 0, kf = 0;  // max of s, max of ~vh (= ~min), largest k
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t i = lane + 32u * (uint32_t)h;
        k[h] = 0;
        if (i < cnt) {
            const uint64_t x = x0 + i;
            if (Q.n_hi) {
                const unsigned __int128 kk = (((unsigned __int128)Q.n_hi << 64) | Q.n) / x;
                k[h] = kk < a.wide_from ? (uint64_t)kk : 0;
            } else {
                k[h] = Q.n / x;
                if (k[h] >= a.wide_from)
                    k[h] = 0;
            }
            jlo[h] = k[h] ? Q.X / x + 1 : 1;
            uint64_t place = Q.place + x - 1;
            if (a.by_k && Q.n)
                // entries of the class before this one in decreasing order of k
                // (ties: by target): floor(n'/x') >= k for the x' <= floor(n'/k)
                for (uint32_t q = 0; q < a.nq; ++q)
                    if (q != lo_q && a.qs[q].n && a.qs[q].cls == Q.cls)
                        place += min(a.qs[q].X, a.qs[q].n / (k[h] + (q < lo_q ? 0u : 1u)));
            if (a.P)
                a.P[Q.off + x - 1] = (uint32_t)place;
            a.K[place] = k[h];
            a.JL[place] = (uint32_t)jlo[h];
            if (k[h]) {
                kf = max(kf, k[h]);
                sq[h] = isqrt_dev(k[h]);
                vh[h] = jlo[h] <= k[h] / (sq[h] + 1) ? k[h] / jlo[h] - 1 : sq[h];
                lo = max(lo, sq[h]);
                nhi = max(nhi, ~vh[h]);
            }
        }
    }
    kf = warp_max_u64(kf);
    lo = warp_max_u64(lo);
    const uint64_t hi = ~warp_max_u64(nhi);
    uint64_t target = (uint64_t)(a.dc * sqrt((double)kf));
    target = (target + kChunk) / kChunk * kChunk - 1;
    uint64_t direct = 0, gathered = 0, gather_j = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if (k[h]) {
            const uint64_t yce =
                lo <= hi ? min(max(target, lo), hi) : min(max(target, sq[h]), vh[h]);
            direct += sq[h];
            const uint64_t jhi = k[h] / (sq[h] + 1), jc = k[h] / (yce + 1);
            gathered += jhi >= jlo[h] ? jhi - jlo[h] + 1 : 0;
            gather_j += jc >= jlo[h] ? jc - jlo[h] + 1 : 0;
        }
    direct = warp_sum_u64(direct);
    gathered = warp_sum_u64(gathered);
    gather_j = warp_sum_u64(gather_j);
    if (lane == 0) {
        WheelTotals *t = a.totals + lo_q;
        atomicAdd(&t->direct, direct);
        atomicAdd(&t->gathered, gathered);
        atomicAdd(&t->gather_j, gather_j);
    }
}

// A warp per group of 64 places: its dense cut-off dc sqrt(mean k of its one-word
// entries), at most floor(k/jlo) of every entry (beyond it no term is left), down
// to a multiple of 6, and every entry's last gathered j.  Any cut-off gives the
// same sums; a dense y costs the whole group one term per entry, a gathered j only
// its own, so the mean of k balances them (with the first entry's k, the first
// group had four times the dense terms: 14% of all at n = 10^13).  jd stays below
// 2^32: the classes of targets (wheel_place.h) keep an entry's floor(k/jlo) from
// taking the cut-off of a far larger k's group below kf / kWheelMaxJ.
__global__ void __launch_bounds__(128) wheel_groups_kernel(WheelEntryArgs a)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= a.ngroups)
        return;
    const uint32_t e0 = g * kWheelGroup, cnt = min(kWheelGroup, a.nplaces - e0);
    uint64_t k[2], jlo[2], kf = 0, ncap = 0;  // largest k, max of ~floor(k/jlo)
    // in double precision: the dense list and the tiles' ranges of places are laid out
    // for dc sqrt(k) as a double (in single precision the cut-offs of 64 close targets
    // near 10^17 could lie 40 above it)
    double ksum = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t i = lane + 32u * (uint32_t)h;
        k[h] = i < cnt ? a.K[e0 + i] : 0;
        if (k[h]) {
            jlo[h] = a.JL[e0 + i];
            kf = max(kf, k[h]);
            ksum += (double)k[h];
            ncap = max(ncap, ~(k[h] / jlo[h]));
        }
    }
    kf = warp_max_u64(kf);
    ncap = warp_max_u64(ncap);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        ksum += __shfl_xor_sync(0xffffffffu, ksum, o);
    const uint32_t one = __reduce_add_sync(0xffffffffu, (k[0] ? 1u : 0u) + (k[1] ? 1u : 0u));
    const uint64_t yc = kf ? wheel_cutoff(a.dc, ksum / one, kf, ~ncap, a.ydense) : 0;
    uint64_t exec = 0, jmax = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t i = lane + 32u * (uint32_t)h;
        if (i < cnt) {
            const uint64_t jd = k[h] ? wheel_last_j(k[h], yc, jlo[h]) : 0;
            a.YC[e0 + i] = k[h] ? yc : 0;
            a.JD[e0 + i] = (uint32_t)jd;
            jmax = max(jmax, jd);
            if (k[h])
                exec += phi6(jd) - phi6(jlo[h] - 1);
        }
    }
    if (jmax >= (1ull << 32) - 6)
        atomicOr(a.err, kErrJ);  // the plan is refused
    exec = warp_sum_u64(exec);
    if (lane == 0) {
        WheelGroup G;
        G.first = e0;
        G.count = cnt;
        G.yc = yc;
        G.kmax = kf;
        a.groups[g] = G;
        atomicAdd(&a.totals->exec, exec);
        atomicAdd(&a.totals->dense_y, yc * one);
    }
}

// Dense work items: (group block, chunk below its largest cut-off, part of the
// chunk's list); dpre[b] = items of the blocks before b.  One CTA.
__global__ void __launch_bounds__(1024) wheel_dense_items_kernel(WheelEntryArgs a)
{
    __shared__ uint32_t sh[33];
    const uint32_t nb = wheel_group_blocks(a.ngroups);
    uint32_t before = 0;
    for (uint32_t b0 = 0; b0 < nb; b0 += 1024u) {
        const uint32_t b = b0 + threadIdx.x;
        uint64_t yc = 0;
        if (b < nb)
            for (uint32_t g = wheel_block_first(b); g < min(wheel_block_first(b + 1), a.ngroups); ++g)
                yc = max(yc, a.groups[g].yc);
        const uint32_t c = (uint32_t)((yc + kWheelSegY - 1) / kWheelSegY) * a.parts;
        uint32_t tot;
        const uint32_t ex = block_scan_u32(c, sh, &tot);
        if (b < nb)
            a.dpre[b] = before + ex;
        before += tot;
    }
    if (threadIdx.x == 0)
        a.dpre[nb] = before;
}

__global__ void wheel_tiles_kernel(WheelEntryArgs a)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.ntiles)
        return;
    const uint2 v = a.tile_src[2 * i];
    WheelGatherTile T;
    T.t0 = (uint64_t)v.x | ((uint64_t)v.y << 32);
    T.len = a.tile_src[2 * i + 1].x;
    T.m1 = magic_of(T.t0 + 1);
    T.l1 = magic_shift(T.t0 + 1);
    T.m2 = magic_of(T.t0 + T.len + 1);
    T.l2 = magic_shift(T.t0 + T.len + 1);
    T.pad = 0;
    a.tiles[i] = T;
}

int wheel_entries_enqueue(const WheelEntryArgs &a, cudaStream_t s)
{
    wheel_entries_kernel<<<(a.qgroups + 3) / 4, 128, 0, s>>>(a);
    wheel_groups_kernel<<<(a.ngroups + 3) / 4, 128, 0, s>>>(a);
    wheel_dense_items_kernel<<<1, 1024, 0, s>>>(a);
    if (a.ntiles)
        wheel_tiles_kernel<<<(a.ntiles + 127) / 128, 128, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// ---------------------------------------------------------------------------
// Dense list: chunk c holds the wheel numbers [c kSegY, (c + 1) kSegY), one
// segment of the sieve; dl gets the offsets of its squarefree numbers, those
// with mu = +1 first.  A thread takes half an element of Mg.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) wheel_dense_list_kernel(const uint2 *__restrict__ Mg,
                                                               uint64_t c0,
                                                               uint16_t *__restrict__ dl,
                                                               uint32_t *__restrict__ dl_cnt)
{
    __shared__ uint32_t sh[33];
    const uint32_t v = Mg[((uint64_t)blockIdx.x * kSegY >> kMgShift) + (threadIdx.x >> 1)].x >>
                       (8u * (threadIdx.x & 1u));
    const uint32_t ng = (v >> 16) & 255u, ps = v & 255u & ~ng;
    const uint32_t cnt = (uint32_t)__popc(ps) + ((uint32_t)__popc(ng) << 16);
    uint32_t tot;
    const uint32_t ex = block_scan_u32(cnt, sh, &tot);
    uint32_t ip = ex & 0xffffu, im = (tot & 0xffffu) + (ex >> 16);
    uint16_t *d = dl + (c0 + blockIdx.x) * kSegY;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const uint16_t o = (uint16_t)(threadIdx.x * 8 + k);
        if ((ps >> k) & 1u)
            d[ip++] = o;
        else if ((ng >> k) & 1u)
            d[im++] = o;
    }
    if (threadIdx.x == 0)
        dl_cnt[c0 + blockIdx.x] = tot;
}

// ---------------------------------------------------------------------------
// Dense update: a warp takes the 64 entries of a group, two per lane, against
// the staged numbers of a chunk (shared-memory broadcasts; two entries per lane
// halve the broadcast per term, four measured 7.5 against 7.8 issue slots per
// term and leave half the groups of a small target).  Bound by issue: 6.4
// instructions, 7.8 slots per term in the float and linear modes (two of them
// multiplies).  n = 10^16, u = 4 10^10: 44.2 ms over every squarefree y by 64-bit
// multiply-high -> 15.3 ms (coprime to 6, remainder and two sign bits) -> 10.8
// (one comparison, two-step mode, cut-offs from the mean k) -> 9.4 (linear mode);
// n = 10^17: 90 -> 54 -> 46 ms by the last two.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t count_below(const uint16_t *a, uint32_t n, uint32_t v)
{
    uint32_t lo = 0, hi = n;  // number of a[i] < v
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < v)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Float mode: staged {1/(3y), -y}.  The estimate k (1/3y) has roundings of 2^-24
// in k, in the reciprocal and, from 3y = 2^24 on, in 3y: it errs by less than 1/3
// for k/(3y) < 2.06e6, or 1.8e6 there (the kernel's rule; n <= 2048 terms, so the
// sum of the T stays below 2^32).
__device__ __forceinline__ void dense_float(const uint4 *el, uint32_t n, const float kf[2],
                                            const uint32_t kl[2], uint64_t out[2])
{
    uint32_t st[2] = {0, 0}, ss[2] = {0, 0};
#pragma unroll 4
    for (uint32_t i = 0; i < n; ++i) {
        const uint4 v = el[i];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t T = __float_as_uint(__fmaf_rd(kf[e], __uint_as_float(v.x), kMagicF));
            ss[e] += (wheel_of_bits(T) * v.y + kl[e]) >> 31;
            st[e] += T;
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        out[e] = (uint64_t)(uint32_t)(st[e] - n * kMagicBits) + n - ss[e];
}

// Linear mode: as the float mode with the chunk's middle ym taken out: with
// q0 = floor(k/(3 ym)) and r0 = k - 3 ym q0, k/(3y) = q0 + (r0 - 3 q0 (y - ym))/(3y).
// For k <= 900 y0^2 (y0 the chunk's start, |y - ym| <= 3071) q0 is below 300 y0 and the
// second part below 300 3071 + 1 = 921 301 in size.  Six roundings of a relative 2^-24
// at most -- two in q0, then the product by 3, the multiply-add, 3y and its reciprocal
// -- make 0.3295 of it: less than the 1/3 needed, so that 900 is the most the rule may
// be.  The sum of 2048 of them fits 32 bits.  Staged {1/(3y), -y, y - ym}.
__device__ __forceinline__ void dense_linear(const uint4 *el, uint32_t n, const uint64_t q0[2],
                                             const float r0[2], const uint32_t kl[2],
                                             uint64_t out[2])
{
    uint32_t st[2] = {0, 0}, ss[2] = {0, 0};
    const float a[2] = {-3.0f * float_u64(q0[0]), -3.0f * float_u64(q0[1])};
    const uint32_t c[2] = {3u * (uint32_t)q0[0] + 1u - 3u * kMagicBits,
                           3u * (uint32_t)q0[1] + 1u - 3u * kMagicBits};
#pragma unroll 4
    for (uint32_t i = 0; i < n; ++i) {
        const uint4 v = el[i];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float R = __fmaf_rn(a[e], __uint_as_float(v.z), r0[e]);
            const uint32_t T = __float_as_uint(__fmaf_rd(R, __uint_as_float(v.x), kMagicF));
            ss[e] += (((3u * T + c[e]) | 1u) * v.y + kl[e]) >> 31;
            st[e] += T;
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        out[e] = (uint64_t)(int64_t)(int32_t)(st[e] - n * kMagicBits) + n * q0[e] + n - ss[e];
}

// High-word mode: staged {m, -y}, m = floor(2^(31 + ex)/(3y)) in [2^30, 2^31),
// ex = floor(log2 3y); kh the top 32 bits of k (b bits), T the floor of
// (kh m / 2^32) / 2^(ex + 31 - b).  Truncations of 2^-31 and 2^-30 and one of a
// unit before the shift (at least 4) with k/(3y) < 6e7: less than 0.15.
__device__ __forceinline__ void dense_high(const uint4 *el, uint32_t n, const uint32_t kh[2],
                                           const uint32_t sb[2], const uint32_t kl[2],
                                           uint64_t out[2])
{
    uint64_t st[2] = {0, 0};
    uint32_t ss[2] = {0, 0};
#pragma unroll 4
    for (uint32_t i = 0; i < n; ++i) {
        const uint4 v = el[i];
        const uint32_t ex = 31u - __clz(0u - 3u * v.y);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            // at most 31 (k far below 3y: T = 0)
            const uint32_t T = __umulhi(kh[e], v.x) >> min(ex + sb[e], 31u);
            ss[e] += (((3u * T + 1u) | 1u) * v.y + kl[e]) >> 31;
            st[e] += T;
        }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
        out[e] = st[e] + n - ss[e];
}

// Two steps, k/(3y) < 3e14, from the same staged values: q1 from the high words as
// above but in 64 bits (at most 3.3e-9 k/(3y) + 1 below k/(3y)), then the float
// mode's estimate for the rest k - 3y q1 < 2^35 (its quotient below 1e6).
__device__ __forceinline__ void dense_two(const uint4 *el, uint32_t n, const uint64_t k[2],
                                          const uint32_t kh[2], const uint32_t sb[2],
                                          uint64_t out[2])
{
    uint64_t st[2] = {0, 0};
    for (uint32_t i = 0; i < n; ++i) {
        const uint4 v = el[i];
        const uint32_t d = 0u - 3u * v.y, ex = 31u - __clz(d);
        const float rf = __uint2float_rn(v.x) * __uint_as_float((96u - ex) << 23);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t h = __umulhi(kh[e], v.x);
            const int sh = (int)(ex + sb[e]);
            const uint64_t q1 = sh >= 0 ? (uint64_t)(h >> min(sh, 31)) : (uint64_t)h << -sh;
            const uint64_t r1 = k[e] - q1 * d;
            const float rh = __uint_as_float(0x4B000000u | (uint32_t)(r1 >> 16)) - 8388608.0f;
            const float rl = __uint_as_float(0x4B000000u | ((uint32_t)r1 & 0xffffu)) - 8388608.0f;
            const uint32_t T2 =
                __float_as_uint(__fmaf_rd(__fmaf_rn(rh, 65536.0f, rl), rf, kMagicF)) - kMagicBits;
            const uint64_t T = q1 + T2;
            st[e] += T + 1u -
                     ((((3u * (uint32_t)T + 1u) | 1u) * v.y + (uint32_t)k[e]) >> 31);
        }
    }
    out[0] = st[0];
    out[1] = st[1];
}

// Any k < 2^63 and y < 2^60, by 64-bit division (few terms need it).
__device__ __forceinline__ void dense_wide(const uint16_t *off, uint32_t n, uint64_t y0,
                                           const uint64_t k[2], uint64_t out[2])
{
    out[0] = out[1] = 0;
    for (uint32_t i = 0; i < n; ++i) {
        const uint32_t o = off[i];
        const uint64_t y = y0 + 3u * o + 1u + (o & 1u), d = 6u * y;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint64_t t = k[e] / d, rem = k[e] - t * d;
            out[e] += 2u * t + (rem >= y ? 1u : 0u) + (rem >= 5u * y ? 1u : 0u);
        }
    }
}

// A work item is part of a chunk's list for kWheelGroupBlock groups.  Items whose
// k/(3y) all lie below the float mode's bound (and y < 3.5e8) take it, those with
// k <= 900 y0^2 the linear mode; in the others the y up to kmax/9e14 (all y from
// 3.5e8) take 64-bit division, those up to kmax/1.8e8 the two-step mode, the rest
// the high-word mode.  Each line is the bound to which the cheaper mode is exact.
// The high-word mode costs twice the float mode's time per term (without the
// linear mode it took 36% of the terms at n = 10^17: 54 against 46 ms); 64-bit
// divisions of the first group alone were a third of the kernel's instructions at
// n = 10^15 before the two-step mode.
__global__ void __launch_bounds__(kWheelDenseThreads) wheel_dense_kernel(WheelDenseArgs a)
{
    __shared__ uint4 s_el[kSegY];
    __shared__ uint16_t s_off[kSegY];
    __shared__ uint32_t s_item, s_block;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const uint32_t nb = wheel_group_blocks(a.ngroups);
    const uint32_t nitems = a.pre[nb];
    for (;;) {
        if (warp == 0) {
            uint32_t it = 0;
            if (lane == 0)
                it = atomicAdd(a.counter, 1u);
            it = __shfl_sync(0xffffffffu, it, 0);
            // the last group block with pre <= it, 32 candidates at a time
            uint32_t lo = 0, hi = nb;
            while (it < nitems && hi - lo > 1u) {
                const uint32_t step = (hi - lo + 31u) / 32u, p = lo + lane * step;
                const uint32_t le = __popc(__ballot_sync(0xffffffffu, p < hi && a.pre[p] <= it));
                hi = min(hi, lo + le * step);
                lo += (le - 1u) * step;
            }
            if (lane == 0) {
                s_item = it;
                s_block = lo;
            }
        }
        __syncthreads();
        if (s_item >= nitems)
            break;
        const uint32_t g0 = wheel_block_first(s_block);
        const uint32_t ng = min(wheel_block_first(s_block + 1), a.ngroups) - g0;
        const uint32_t rel = s_item - a.pre[s_block];
        const uint32_t c = rel / a.parts, part = rel % a.parts;
        uint64_t kmax = 0;
        for (uint32_t g = 0; g < ng; ++g)
            kmax = max(kmax, a.groups[g0 + g].kmax);
        const uint64_t y0 = (uint64_t)c * kWheelSegY;
        const bool small_y = y0 + kWheelSegY < 350000000u;
        const bool fl =
            small_y && kmax < (y0 + kWheelSegY < 5500000u ? 6200000ull : 5400000ull) * (y0 + 1);
        const bool lin = small_y && !fl && kmax / 900u <= y0 * y0;
        const uint32_t ym = (uint32_t)y0 + (uint32_t)kWheelSegY / 2u;
        const uint32_t cnt = a.dl_cnt[c];
        const uint32_t cp = cnt & 0xffffu, cm = cnt >> 16;
        const uint32_t p0 = cp * part / a.parts, m0 = cm * part / a.parts;
        const uint32_t np = cp * (part + 1u) / a.parts - p0, nm = cm * (part + 1u) / a.parts - m0;
        const uint16_t *src = a.dl + (uint64_t)c * kSegY;
        for (uint32_t i = threadIdx.x; i < np + nm; i += blockDim.x) {
            const uint32_t o = i < np ? src[p0 + i] : src[cp + m0 + (i - np)];
            s_off[i] = (uint16_t)o;
            if (!small_y)
                continue;
            const uint32_t y = (uint32_t)y0 + 3u * o + 1u + (o & 1u), d = 3u * y;
            const uint32_t ex = 31u - __clz(d);
            s_el[i] = make_uint4(fl || lin ? __float_as_uint(__frcp_rn(__uint2float_rn(d)))
                                           : (uint32_t)((1ull << (31u + ex)) / d),
                                 0u - y, __float_as_uint((float)(int32_t)(y - ym)), 0u);
        }
        __syncthreads();
        // one group per warp; fewer groups than warps: several warps share a
        // group, each with its part of the staged lists
        const uint32_t share = nwarp / ng;
        for (uint32_t t = warp; t < ng * share; t += nwarp) {
            const WheelGroup G = a.groups[g0 + t % ng];
            const uint32_t q = t / ng;
            if (G.yc <= y0)
                continue;
            uint64_t k[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t i = lane + 32u * (uint32_t)e;
                k[e] = i < G.count ? a.K[G.first + i] : 0ull;
            }
            uint32_t n0 = np, n1 = nm;
            if (G.yc < y0 + kWheelSegY) {
                const uint32_t lim = (uint32_t)(phi6(G.yc) - (uint64_t)c * kSegY);
                n0 = count_below(s_off, np, lim);
                n1 = count_below(s_off + np, nm, lim);
            }
            const uint32_t f0 = n0 * q / share, f1 = np + n1 * q / share;
            n0 = n0 * (q + 1u) / share - f0;
            n1 = n1 * (q + 1u) / share - (f1 - np);
            uint64_t sum[2], part2[2];
            if (fl) {
                const float kf[2] = {__ull2float_rn(k[0]), __ull2float_rn(k[1])};
                const uint32_t kl[2] = {(uint32_t)k[0], (uint32_t)k[1]};
                dense_float(s_el + f0, n0, kf, kl, sum);
                dense_float(s_el + f1, n1, kf, kl, part2);
                sum[0] -= part2[0];
                sum[1] -= part2[1];
            } else if (lin) {
                uint64_t q0[2];
                float r0[2];
                const uint32_t kl[2] = {(uint32_t)k[0], (uint32_t)k[1]};
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    q0[e] = k[e] / (3u * ym);
                    r0[e] = __uint2float_rn((uint32_t)(k[e] - q0[e] * (3u * ym)));
                }
                dense_linear(s_el + f0, n0, q0, r0, kl, sum);
                dense_linear(s_el + f1, n1, q0, r0, kl, part2);
                sum[0] -= part2[0];
                sum[1] -= part2[1];
            } else {
                // terms with y <= yl of a list
                const auto upto = [&](const uint16_t *off, uint32_t n, uint64_t yl) -> uint32_t {
                    if (yl <= y0)
                        return 0;
                    if (yl >= y0 + kWheelSegY)
                        return n;
                    return count_below(off, n, (uint32_t)(phi6(yl) - (uint64_t)c * kSegY));
                };
                const uint64_t yd = small_y ? G.kmax / 900000000000000ull : UINT64_MAX;
                const uint64_t yt = small_y ? G.kmax / 180000000ull : UINT64_MAX;
                uint32_t kh[2], sb[2], kl[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const uint32_t b = bitlen64(k[e]);
                    kl[e] = (uint32_t)k[e];
                    kh[e] = b >= 32u ? (uint32_t)(k[e] >> (b - 32u))
                                     : (uint32_t)k[e] << ((32u - b) & 31u);
                    sb[e] = 31u - b;
                }
                sum[0] = sum[1] = 0;
#pragma unroll 1
                for (uint32_t l = 0; l < 2u; ++l) {  // mu = +1, then -1
                    const uint32_t f = l ? f1 : f0, n = l ? n1 : n0;
                    const uint32_t nd = upto(s_off + f, n, yd), nt = upto(s_off + f, n, yt);
                    uint64_t t[2] = {0, 0};
                    if (nd) {
                        dense_wide(s_off + f, nd, y0, k, part2);
                        t[0] += part2[0];
                        t[1] += part2[1];
                    }
                    if (nt > nd) {
                        dense_two(s_el + f + nd, nt - nd, k, kh, sb, part2);
                        t[0] += part2[0];
                        t[1] += part2[1];
                    }
                    dense_high(s_el + f + nt, n - nt, kh, sb, kl, part2);
                    t[0] += part2[0];
                    t[1] += part2[1];
                    sum[0] += l ? 0u - t[0] : t[0];
                    sum[1] += l ? 0u - t[1] : t[1];
                }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (k[e])
                    atomicAdd(reinterpret_cast<unsigned long long *>(a.S + G.first + lane +
                                                                     32u * (uint32_t)e),
                              (unsigned long long)sum[e]);
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Gathered terms of a shared-memory tile: y in [t0 + 1, t0 + len], len <=
// 98304, staged as M6(y) - M6(t0) (int16: at most 24/25 of 32768 consecutive
// wheel numbers are squarefree) by wheel index.  A term's index is
// phi6(floor(R/j)) - 1 with R = k - t0 j < len j: T = floor of R / (3j) <= 2^15
// from single precision (relative error near 2^-21), then as above.
// Bound by issue (about 11 slots per term with all lanes on one j, 18 with a j
// per lane, and the ranges' divisions).  n = 10^16, u = 4 10^10, all gathered
// terms: 55.1 ms over every j -> 22.1 (j coprime to 6) -> 17.0 (one comparison,
// groups handed out one by one, the first entries shared by all warps, Mg).
// ---------------------------------------------------------------------------
constexpr uint32_t kGatherJ32 = 300000000u;  // 32-bit remainders below: 5j < 2^31
constexpr uint32_t kWheelLaneTerms = 16;     // few terms: always a lane per entry (8 and
                                             // 32 measure the same)

// Constants of a run of terms j = j0 + step i in a tile.
struct TileStep {
    float dRf, stepf;    // step t0 / 3, step
    uint32_t dR32, step; // step t0 (mod 2^32), step
    uint64_t dR;         // step t0
    __device__ __forceinline__ TileStep(uint64_t t0, uint32_t st)
        : dRf(float_u64(t0) * ((float)st / 3.0f)), stepf((float)st), dR32((uint32_t)t0 * st),
          step(st), dR(t0 * st)
    {
    }
};

// State of a run: R = k - t0 j and j of the current term.  Rf = R/3 and jf are
// stepped from the run's start with one multiply-add each; kLong (5j beyond 32
// bits) takes the remainder in 64 bits.
template <bool kLong>
struct TileRun {
    float Rf0, jf0;
    uint32_t nR, j;  // -R - 1 (mod 2^32), j
    uint64_t R;
    __device__ __forceinline__ TileRun(uint64_t k, uint64_t t0, uint32_t j0)
    {
        R = k - t0 * (uint64_t)j0;
        Rf0 = float_u64(R) * (1.0f / 3.0f);
        jf0 = __uint2float_rn(j0);
        j = j0;
        nR = ~(uint32_t)R;
    }
    // the staged value of term i (fi = i), then on to term i + 1
    __device__ __forceinline__ int take(const int16_t *Mt, uint32_t lim, float fi,
                                        const TileStep &d)
    {
        const float Rf = __fmaf_rn(fi, -d.dRf, Rf0), jf = __fmaf_rn(fi, d.stepf, jf0);
        float rj;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rj) : "f"(jf));
        const uint32_t T = __float_as_uint(__fmaf_rd(Rf, rj, kMagicF));
        const uint32_t W = wheel_of_bits(T);
        uint32_t i;  // T - 1 + [R >= j W]
        if (kLong) {
            i = T - kMagicBits - (uint32_t)((R - (uint64_t)(int64_t)(int32_t)W * j) >> 63);
            R -= d.dR;
        } else {
            i = T - (kMagicBits + 1u) + ((W * j + nR) >> 31);
            nR += d.dR32;
        }
        j += d.step;
        return Mt[i < lim ? i : lim];
    }
};

// Terms with wheel indices [wl, wh) of one entry on one lane: the two classes
// (even and odd indices, j in steps of 6) side by side.
template <bool kLong>
__device__ __forceinline__ int tile_lane(const int16_t *Mt, uint64_t k, uint64_t t0, uint32_t lim,
                                         uint32_t wl, uint32_t wh)
{
    const TileStep d(t0, 6u);
    const uint32_t we = (wl + 1u) & ~1u, wo = wl | 1u;  // first even, first odd index
    const uint32_t ne = we < wh ? (wh - we + 1u) >> 1 : 0u, no = wo < wh ? (wh - wo + 1u) >> 1 : 0u;
    TileRun<kLong> e(k, t0, 3u * we + 1u), o(k, t0, 3u * wo + 2u);
    const uint32_t n = ne < no ? ne : no;
    int acc = 0;
    float fi = 0.0f;
#pragma unroll 2
    for (uint32_t i = 0; i < n; ++i, fi += 1.0f)
        acc += e.take(Mt, lim, fi, d) + o.take(Mt, lim, fi, d);
    if (ne > n)
        acc += e.take(Mt, lim, fi, d);
    if (no > n)
        acc += o.take(Mt, lim, fi, d);
    return acc;
}

// The same on a whole warp, lanes over consecutive indices (returns the lane's part).
template <bool kLong>
__device__ __forceinline__ int tile_warp(const int16_t *Mt, uint64_t k, uint64_t t0, uint32_t lim,
                                         uint32_t wl, uint32_t wh, uint32_t lane)
{
    const TileStep d(t0, 96u);
    const uint32_t w = wl + lane;
    int acc = 0;
    if (w < wh) {
        TileRun<kLong> r(k, t0, 3u * w + 1u + (w & 1u));
        const uint32_t n = (wh - w + 31u) >> 5;
        float fi = 0.0f;
#pragma unroll 2
        for (uint32_t i = 0; i < n; ++i, fi += 1.0f)
            acc += r.take(Mt, lim, fi, d);
    }
    return acc;
}

// M6 at wheel index i of a block.
__device__ __forceinline__ int64_t wheel_M(const int64_t *segoff, const uint2 *Mg, uint64_t i)
{
    return segoff[i >> kSegShift] + (int64_t)wheel_value(Mg, i);
}

// Tiles at y <= kUniformY: 64 entries of a warp (two per lane) against the same
// j, whose constants {1/(3j), j} are made 32 at a time by the lanes and read back
// as broadcasts.  T estimates k/(3j) itself (3j < 2^24 here, so two roundings of
// 2^-24, and k/(3j) < 2.6e6 for 5% beyond the tile), and the sign bit of
// j Y(T) - k - 1 completes the index T - 1 + [k >= j Y(T)] less the tile's first
// one.  An index outside [lo, lim] -- a j whose y lies beyond the tile or at most
// yc (yc + 1 a wheel number) -- is sent to the zero after it.  jw: 32 uint2 of
// this warp; b2 = -C - 1 - (first index) - lo.
// That error bound sets the limit.  Up to it this form beats a j per lane: 39.4
// against 41.3 ms a run at n = 10^16, 27.4 against 29.5 for 64 targets near 10^14.
constexpr uint64_t kUniformY = 7400000;
constexpr uint32_t kUniformW = 1860000;  // 3j < 2^24

__device__ __forceinline__ void tile_uniform(const int16_t *Mt, uint2 *jw, const uint64_t k[2],
                                             const uint32_t b2[2], const uint32_t lo[2],
                                             uint32_t lim, uint32_t w0, uint32_t w1, uint32_t lane,
                                             int acc[2])
{
    const float kf[2] = {__ull2float_rn(k[0]), __ull2float_rn(k[1])};
    const uint32_t nk[2] = {~(uint32_t)k[0], ~(uint32_t)k[1]};
    const uint32_t hi[2] = {lim + 1u - lo[0], lim + 1u - lo[1]};
    const int16_t *Ml[2] = {Mt + lo[0], Mt + lo[1]};
    acc[0] = acc[1] = 0;
#pragma unroll 1
    for (uint32_t wb = w0; wb < w1; wb += 32u) {
        {
            const uint32_t w = wb + lane, j = 3u * w + 1u + (w & 1u);
            jw[lane] = make_uint2(__float_as_uint(__frcp_rn(__uint2float_rn(3u * j))), j);
        }
        __syncwarp();
        const uint32_t n = min(32u, w1 - wb);
#pragma unroll 4
        for (uint32_t i = 0; i < n; ++i) {
            const uint2 c = jw[i];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint32_t T =
                    __float_as_uint(__fmaf_rd(kf[e], __uint_as_float(c.x), kMagicF));
                const uint32_t x = T + b2[e] + ((wheel_of_bits(T) * c.y + nk[e]) >> 31);
                acc[e] += Ml[e][min(x, hi[e])];
            }
        }
        __syncwarp();
    }
}

// The ranges of wheel indices of the j of 64 entries eb .., two per lane, in a tile.
struct TileRanges {
    uint64_t k[2];
    uint32_t wl[2], wh[2];
    bool big, bound;  // some j beyond 32-bit remainders; some range starts at jlo
};

__device__ __forceinline__ TileRanges tile_ranges(const WheelGatherArgs &a,
                                                  const WheelGatherTile &T, uint32_t eb,
                                                  uint32_t e1, uint32_t lane)
{
    TileRanges r;
    r.big = a.all_long;
    r.bound = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t e = eb + 32u * (uint32_t)h + lane;
        r.k[h] = 0;
        r.wl[h] = r.wh[h] = 0;
        if (e < e1) {
            r.k[h] = a.K[e];
            const uint64_t jd = a.JD[e], jlo = a.JL[e];
            const uint64_t q1 = div_magic(r.k[h] << 1, T.m1, T.l1);  // floor(k/(t0+1))
            const uint64_t q2 = div_magic(r.k[h] << 1, T.m2, T.l2);  // floor(k/(t0+len+1))
            const uint64_t t = jd < q1 ? jd : q1, b = q2 + 1u > jlo ? q2 + 1u : jlo;
            r.bound |= b != q2 + 1u;
            if (r.k[h] && t >= b) {
                r.big |= t >= kGatherJ32;
                r.wl[h] = phi6_u32((uint32_t)b - 1u);
                r.wh[h] = phi6_u32((uint32_t)t);
            }
        }
    }
    return r;
}

// Sum of one entry's terms [wl, wh) by a warp, added to S[e].
__device__ __forceinline__ void tile_entry(const WheelGatherArgs &a, const int16_t *Mt,
                                           const WheelGatherTile &T, uint32_t lim, int64_t base,
                                           bool big, uint32_t e, uint64_t k, uint32_t wl,
                                           uint32_t wh, uint32_t lane)
{
    const int acc = big ? tile_warp<true>(Mt, k, T.t0, lim, wl, wh, lane)
                        : tile_warp<false>(Mt, k, T.t0, lim, wl, wh, lane);
    const int tot = __reduce_add_sync(0xffffffffu, acc);
    if (lane == 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(a.S + e),
                  (unsigned long long)((int64_t)tot + (int64_t)(wh - wl) * base));
}

// A work item is one tile and a range of places.  Warps take 64
// entries at a time, two per lane, and find the ranges of wheel indices of
// their j.  Low tiles where these ranges nearly coincide take tile_uniform.
// The others, 32 entries at a time: when the counts are close and no lane's sum
// would take long against the whole kernel (or all are small) every lane sums its
// own entry, else entries with many terms take the whole
// warp in turn; with many terms in all, at the end of the item, where all warps
// share them (the first 32 entries of a target hold a third of a tile's terms;
// on one warp, the other fifteen waited for it; all sets of 32 that way: 3.99
// against 3.32 ms at n = 10^15).  From 65536 terms a
// set: 0.154 against 0.131 ms at n = 10^10; from 4096: the same.
constexpr uint32_t kSharedMax = 128;         // sets of 32 left to the end of an item
constexpr uint32_t kSharedTerms = 16384;     // a set's terms from which it is
constexpr uint32_t kSharedSlice = 8192;      // an entry's terms from which warps split it

__global__ void __launch_bounds__(512, 3) wheel_gather_kernel(WheelGatherArgs a)
{
    extern __shared__ __align__(16) int16_t Mt[];  // kGatherTile, a zero, j constants
    __shared__ uint32_t s_item, s_nshared, s_next;
    __shared__ uint32_t s_shared[kSharedMax];
    __shared__ int64_t s_base;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    uint2 *jw = reinterpret_cast<uint2 *>(Mt + kGatherTile + 8) + warp * 32u;
    uint32_t staged = 0xffffffffu;
    for (;;) {
        if (threadIdx.x == 0) {
            s_item = atomicAdd(a.counter, 1u);
            s_nshared = 0;
            s_next = 0;
        }
        __syncthreads();
        if (s_item >= a.nitems)
            break;
        const uint4 I = a.items[s_item];
        const WheelGatherTile T = a.tiles[I.x];
        if (I.x != staged) {
            // 16 values per element of Mg, relative to M6(t0)
            const uint32_t o1 = (uint32_t)((T.t0 - a.y0) / 3u), n = T.len / 3u;
            const int64_t b0 = a.segoff[o1 >> kSegShift];
            if (threadIdx.x == 0) {
                s_base = b0;
                Mt[n] = 0;
            }
            const uint2 *src = a.Mg + (o1 >> kMgShift);
            uint4 *Mw = reinterpret_cast<uint4 *>(Mt);
            for (uint32_t i = threadIdx.x; i < n >> kMgShift; i += blockDim.x) {
                const uint2 v = src[i];
                int r = (int)v.y +
                        (int)(a.segoff[(o1 + (i << kMgShift)) >> kSegShift] - b0);
                uint32_t o[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    r += (int)((v.x >> (2 * k)) & 1u) - 2 * (int)((v.x >> (16 + 2 * k)) & 1u);
                    const uint32_t lo = (uint32_t)r & 0xffffu;
                    r += (int)((v.x >> (2 * k + 1)) & 1u) - 2 * (int)((v.x >> (17 + 2 * k)) & 1u);
                    o[k] = lo | ((uint32_t)r << 16);
                }
                Mw[2 * i] = make_uint4(o[0], o[1], o[2], o[3]);
                Mw[2 * i + 1] = make_uint4(o[4], o[5], o[6], o[7]);
            }
            staged = I.x;
        }
        __syncthreads();
        const int64_t base = s_base;
        const uint32_t lim = T.len / 3u - 1u;
        const bool low = T.t0 + T.len <= kUniformY;
        for (;;) {
            uint32_t eb = 0;  // the next 64 entries
            if (lane == 0)
                eb = I.y + 64u * atomicAdd(&s_next, 1u);
            eb = __shfl_sync(0xffffffffu, eb, 0);
            if (eb >= I.z)
                break;
            const TileRanges r = tile_ranges(a, T, eb, I.z, lane);
            const uint32_t c0 = r.wh[0] - r.wl[0], c1 = r.wh[1] - r.wl[1];
            const uint32_t sum = __reduce_add_sync(0xffffffffu, c0 + c1);
            if (sum == 0)
                continue;
            if (low && !__any_sync(0xffffffffu, r.bound || r.big)) {
                const uint32_t w0 = __reduce_min_sync(0xffffffffu, min(c0 ? r.wl[0] : 0xffffffffu,
                                                                       c1 ? r.wl[1] : 0xffffffffu));
                const uint32_t w1 = __reduce_max_sync(0xffffffffu, max(r.wh[0], r.wh[1]));
                // 64 (w1 - w0) terms at about 11 issue slots each against
                // `sum` at about 18
                if (40u * (w1 - w0) <= sum && w1 < kUniformW) {
                    uint32_t lo[2], b2[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t e = eb + 32u * (uint32_t)h + lane;
                        lo[h] = lim + 1u;  // no entry: nothing counts
                        if (r.k[h]) {
                            const uint64_t yc = a.YC[e];
                            lo[h] = yc <= T.t0 ? 0u
                                    : yc >= T.t0 + T.len ? lim + 1u
                                                         : phi6_u32((uint32_t)(yc - T.t0));
                        }
                        b2[h] = 0u - kMagicBits - 1u - (uint32_t)(T.t0 / 3u) - lo[h];
                    }
                    int acc[2];
                    tile_uniform(Mt, jw, r.k, b2, lo, lim, w0, w1, lane, acc);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t cnt = h ? c1 : c0;
                        if (cnt)
                            atomicAdd(reinterpret_cast<unsigned long long *>(a.S + eb +
                                                                             32u * (uint32_t)h + lane),
                                      (unsigned long long)((int64_t)acc[h] + (int64_t)cnt * base));
                    }
                    continue;
                }
            }
            const bool big = __any_sync(0xffffffffu, r.big);
#pragma unroll 1
            for (uint32_t h = 0; h < 2u; ++h) {
                const uint32_t cnt = h ? c1 : c0, wlh = h ? r.wl[1] : r.wl[0],
                               whh = h ? r.wh[1] : r.wh[0];
                const uint64_t kh = h ? r.k[1] : r.k[0];
                const uint32_t e0 = eb + 32u * h;
                const uint32_t mx = __reduce_max_sync(0xffffffffu, cnt);
                if (mx == 0)
                    continue;
                const uint32_t hsum = __reduce_add_sync(0xffffffffu, cnt);
                const bool lanes =
                    mx <= kWheelLaneTerms || (16u * mx <= hsum && mx < a.long_lane);
                if (!lanes && hsum >= kSharedTerms) {
                    uint32_t slot = 0;
                    if (lane == 0)
                        slot = atomicAdd(&s_nshared, 1u);
                    slot = __shfl_sync(0xffffffffu, slot, 0);
                    if (slot < kSharedMax) {
                        if (lane == 0)
                            s_shared[slot] = e0;
                        continue;
                    }
                }
                if (cnt && (lanes || cnt <= kWheelLaneTerms)) {
                    const int acc = big ? tile_lane<true>(Mt, kh, T.t0, lim, wlh, whh)
                                        : tile_lane<false>(Mt, kh, T.t0, lim, wlh, whh);
                    atomicAdd(reinterpret_cast<unsigned long long *>(a.S + e0 + lane),
                              (unsigned long long)((int64_t)acc + (int64_t)cnt * base));
                }
                uint32_t mask = lanes ? 0u : __ballot_sync(0xffffffffu, cnt > kWheelLaneTerms);
                while (mask) {
                    const int src = __ffs(mask) - 1;
                    mask &= mask - 1;
                    const uint32_t wls = __shfl_sync(0xffffffffu, wlh, src);
                    const uint32_t whs = __shfl_sync(0xffffffffu, whh, src);
                    const uint64_t ks = __shfl_sync(0xffffffffu, kh, src);
                    tile_entry(a, Mt, T, lim, base, big, e0 + src, ks, wls, whs, lane);
                }
            }
        }
        __syncthreads();
        // the groups left: every warp finds the ranges; entries in turn to the
        // warps, the largest split over all of them
        const uint32_t nsh = min(s_nshared, kSharedMax);
        uint32_t turn = 0;
        for (uint32_t q = 0; q < nsh; ++q) {
            const uint32_t eb = s_shared[q];
            const TileRanges r = tile_ranges(a, T, eb, min(I.z, eb + 32u), lane);
            const bool big = __any_sync(0xffffffffu, r.big);
#pragma unroll 1
            for (uint32_t i = 0; i < 32u; ++i) {
                uint32_t wl = __shfl_sync(0xffffffffu, r.wl[0], i);
                uint32_t wh = __shfl_sync(0xffffffffu, r.wh[0], i);
                const uint32_t cnt = wh - wl;
                if (cnt == 0)
                    continue;
                if (cnt >= kSharedSlice) {
                    const uint32_t part = ((cnt + nwarp - 1) / nwarp + 31u) & ~31u;
                    wl = min(wl + warp * part, wh);
                    wh = min(wl + part, wh);
                    if (wl >= wh)
                        continue;
                } else if (turn++ % nwarp != warp) {
                    continue;
                }
                const uint64_t k = __shfl_sync(0xffffffffu, r.k[0], i);
                tile_entry(a, Mt, T, lim, base, big, eb + i, k, wl, wh, lane);
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Global-memory part of a block (y0, y0 + len]: one lane per entry.  Gathered
// terms with floor(k/j) in [ylo, y0 + len] of entries with k < kmax (few: here;
// more: posted as chunks of kWheelItem wheel indices for wheel_chunk_kernel);
// the dense form's -M6(yc) phi6(jd) when yc is in the block; and the values
// M6(floor(k/m)), m = 2, 3, 6, of M(k) that lie in the block when m x is
// beyond the array (m >= floor(X/x) + 1).  Bound by the 64-bit divisions and
// random reads of entries with few terms, and by latency: at n = 10^16 0.64 ms per run
// of 25 blocks (with the entry's loads one after the other 17 us per block).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) wheel_range_kernel(WheelBlockArgs a)
{
    const uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t lane = threadIdx.x & 31u;
    // the entry's loads at once: one after the other they took most of the time
    uint64_t k = 0, jlo = 0, jd = 0, yc = 0;
    if (e < a.nplaces) {
        k = a.K[e];
        yc = a.YC[e];
        jlo = a.JL[e];
        jd = a.JD[e];
    }
    const uint64_t yend = a.y0 + a.len;
    uint32_t wl = 0, wh = 0;
    if (k) {
        if (k < a.kmax) {
            const uint64_t q1 = div_magic(k << 1, a.m_ylo, a.l_ylo);  // floor(k / ylo)
            const uint64_t q2 = div_magic(k << 1, a.m_end, a.l_end);  // floor(k / (yend + 1))
            const uint64_t t = jd < q1 ? jd : q1, b = q2 + 1u > jlo ? q2 + 1u : jlo;
            if (t >= b) {
                wl = phi6_u32((uint32_t)b - 1u);
                wh = phi6_u32((uint32_t)t);
            }
        }
        if (yc > a.y0 && yc <= yend)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.S + e),
                      (unsigned long long)(0ull - (uint64_t)wheel_M(a.segoff, a.Mg,
                                                                    wheel_index((uint32_t)(yc - a.y0))) *
                                                      phi6(jd)));
        int64_t tail = 0;
        if (jlo <= 6u && k / 6u <= yend) {
#pragma unroll
            for (uint32_t m = 2; m <= 6; m += (m == 2 ? 1u : 3u)) {
                const uint64_t y = k / m;
                if (m >= jlo && y > a.y0 && y <= yend) {
                    const int64_t v =
                        wheel_M(a.segoff, a.Mg, wheel_index((uint32_t)(y - a.y0)));
                    tail += m == 6 ? v : -v;
                }
            }
            if (tail)
                a.A[e] += (uint64_t)tail;
        }
    }
    const uint32_t cnt = wh - wl;
    if (cnt && cnt <= kWheelLaneTerms) {
        int64_t acc = 0;
#pragma unroll 4
        for (uint32_t w = wl; w < wh; ++w) {
            const uint64_t y = k / (3ull * w + 1u + (w & 1u));
            acc += wheel_M(a.segoff, a.Mg, wheel_index((uint32_t)(y - a.y0)));
        }
        atomicAdd(reinterpret_cast<unsigned long long *>(a.S + e), (unsigned long long)acc);
    }
    // heavy entries: chunk records, slots taken with one atomic per warp
    const uint32_t nch = cnt > kWheelLaneTerms ? (cnt + kWheelItem - 1) / kWheelItem : 0u;
    uint32_t incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t nb = __shfl_up_sync(0xffffffffu, incl, o);
        if ((int)lane >= o)
            incl += nb;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0)
        return;
    uint32_t base = 0;
    if (lane == 31)
        base = atomicAdd(a.qlen, total);
    base = __shfl_sync(0xffffffffu, base, 31);
    uint32_t slot = base + incl - nch;
    for (uint32_t c = 0; c < nch; ++c, ++slot) {
        const uint32_t w = wl + c * kWheelItem;
        if (slot < a.qcap)
            a.queue[slot] = make_uint4((uint32_t)e, w, min(wh - w, kWheelItem), 0u);
        else
            atomicOr(a.err, kErrQueue);
    }
}

// The posted chunks, a warp each (grid-stride), lanes over consecutive indices.
// Bound by 64-bit divisions and random reads; at n = 10^16 1.48 ms per run when
// the block held int16 values, 1.05 ms from Mg (a quarter of the memory, more of
// it in L2), 0.94 ms in blocks of 1.6e9 y.
__global__ void __launch_bounds__(256) wheel_chunk_kernel(WheelBlockArgs a)
{
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t total = min(*a.qlen, a.qcap);
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < total; q += nw) {
        const uint4 r = a.queue[q];
        const uint64_t k = a.K[r.x];
        int64_t acc = 0;
#pragma unroll 4
        for (uint32_t i = lane; i < r.z; i += 32u) {
            const uint32_t w = r.y + i;
            const uint64_t y = k / (3ull * w + 1u + (w & 1u));
            acc += wheel_M(a.segoff, a.Mg, wheel_index((uint32_t)(y - a.y0)));
        }
        acc = warp_sum_i64(acc);
        if (lane == 0)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.S + r.x), (unsigned long long)acc);
    }
}

// ---------------------------------------------------------------------------
// Two-word entries (grid.y of them), the block's terms numbered as one range,
// kWidePer consecutive ones per thread; sums mod 2^64.
// ---------------------------------------------------------------------------
typedef unsigned __int128 u128d;

// phi6(floor(k/y)) mod 2^64.
__device__ __forceinline__ uint64_t phi6_quot(u128d k, uint64_t y)
{
    const u128d d = (u128d)6u * y, t = k / d, rem = k - t * d;
    return 2u * (uint64_t)t + (rem >= y ? 1u : 0u) + (rem >= (u128d)5u * y ? 1u : 0u);
}

__host__ __device__ inline void wide_units(const WideEntry &W, uint64_t y0, uint64_t len,
                                           uint64_t *direct, uint64_t *wj, uint64_t *gathered)
{
    const unsigned __int128 k = ((unsigned __int128)W.k_hi << 64) | W.k_lo;
    const uint64_t yend = y0 + len, top = W.s < yend ? W.s : yend;
    *direct = top > y0 ? phi6(top) - phi6(y0) : 0;
    // j with floor(k/j) in (y0, yend]
    const unsigned __int128 q2 = k / ((unsigned __int128)yend + 1) + 1;
    const unsigned __int128 q1 = k / ((unsigned __int128)y0 + 1);
    const uint64_t b = q2 > W.jlo ? (q2 > W.jhi ? W.jhi + 1 : (uint64_t)q2) : W.jlo;
    const uint64_t t = q1 < W.jhi ? (uint64_t)q1 : W.jhi;
    *wj = b <= t ? phi6(b - 1) : 0;
    *gathered = b <= t ? phi6(t) - *wj : 0;
}

void wheel_wide_units(const WideEntry &W, uint64_t y0, uint64_t len, uint64_t *direct,
                      uint64_t *wj, uint64_t *gathered)
{
    wide_units(W, y0, len, direct, wj, gathered);
}

__global__ void __launch_bounds__(kWideThreads) wheel_wide_kernel(WheelWideArgs a)
{
    __shared__ uint64_t red[kWideThreads / 32];
    const WideEntry W = a.W[blockIdx.y];
    const u128d k = ((u128d)W.k_hi << 64) | W.k_lo;
    uint64_t nd, wj, ng;
    wide_units(W, a.y0, a.len, &nd, &wj, &ng);
    const uint64_t units = nd + ng;
    const uint64_t u0 = (uint64_t)blockIdx.x * kWideUnitsPerCta + (uint64_t)threadIdx.x * kWidePer;
    const uint64_t u1 = u0 + kWidePer < units ? u0 + kWidePer : units;
    uint64_t acc = 0, u = u0;
    if (u < u1 && u < nd) {
        // direct: wheel number w0 + u and the y up to the next one (or s)
        const uint64_t w0 = a.y0 / 3;
        uint64_t p = phi6_quot(k, wheel_y(w0 + u));
        for (const uint64_t ue = u1 < nd ? u1 : nd; u < ue; ++u) {
            const uint64_t yn = wheel_y(w0 + u + 1);
            const uint64_t pn = phi6_quot(k, yn <= W.s ? yn : W.s + 1);
            acc += (uint64_t)wheel_M(a.segoff, a.Mg, (uint32_t)u) * (p - pn);
            p = pn;
        }
    }
    for (; u < u1; ++u) {
        const uint64_t j = wheel_y(wj + (u - nd));
        acc += (uint64_t)wheel_M(a.segoff, a.Mg, wheel_index((uint32_t)((uint64_t)(k / j) - a.y0)));
    }
    acc = warp_sum_u64(acc);
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint64_t t = 0;
        for (int w = 0; w < kWideThreads / 32; ++w)
            t += red[w];
        if (t)
            atomicAdd(reinterpret_cast<unsigned long long *>(a.S + W.e), (unsigned long long)t);
        if (blockIdx.x == 0 && W.jlo <= 6u) {
            int64_t tail = 0;
            for (uint32_t m = 2; m <= 6; m += (m == 2 ? 1u : 3u)) {
                const u128d y = k / m;
                if (m >= W.jlo && y > a.y0 && y <= a.y0 + a.len) {
                    const int64_t v = wheel_M(a.segoff, a.Mg,
                                              wheel_index((uint32_t)((uint64_t)y - a.y0)));
                    tail += m == 6 ? v : -v;
                }
            }
            a.A[W.e] += (uint64_t)tail;
        }
    }
}

// ---------------------------------------------------------------------------
// Resident tables.
// ---------------------------------------------------------------------------
__global__ void wheel_lookup_kernel(const uint64_t *__restrict__ pairs, uint32_t count,
                                    const uint2 *__restrict__ Mg,
                                    const int64_t *__restrict__ segoff, uint64_t *__restrict__ R)
{
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count)
        return;
    const uint64_t y = pairs[2 * i + 1];
    const auto M6 = [&](uint64_t v) -> int64_t {
        const uint64_t w = phi6(v);
        return w ? wheel_M(segoff, Mg, w - 1) : 0;
    };
    R[pairs[2 * i]] = (uint64_t)(M6(y) - M6(y / 2) - M6(y / 3) + M6(y / 6));
}

__global__ void wheel_carry_at_kernel(const uint2 *__restrict__ Mg,
                                      const int64_t *__restrict__ segoff, uint64_t w,
                                      int64_t *__restrict__ out)
{
    *out = wheel_M(segoff, Mg, w);
}

// ---------------------------------------------------------------------------
// Resolve: R6[x] = 1 - S[x] - sum over j >= 2 coprime to 6, xj <= X, of R6[xj],
// then M[x] = R6[x] - V(2x) - V(3x) + V(6x), V(z) = R6[z] within the array (the
// values beyond it are in A).  The smallest such j is 5, so the entries of
// (X/5^(l+1), X/5^l] only read entries above X/5^l: level by level, every entry
// of a level in parallel: a thread per entry, a warp from X/x = 64 on, a CTA from
// 1024 on (a warp on the 83 000 terms of x = 1 took 243 of 370 us at X = 250 000).
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint64_t at_place(const uint64_t *v, const uint32_t *P, uint64_t e)
{
    return v[P ? P[e] : e];
}

__device__ __forceinline__ void resolve_level(const QueryDev &Q, const uint32_t *P,
                                              const uint64_t *S, uint64_t *R6,
                                              uint64_t xlo, uint64_t xhi, uint64_t tid,
                                              uint64_t nthreads, uint64_t *sh)
{
    const uint64_t X = Q.X, base = Q.off;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    if (X / xhi < 64) {
        for (uint64_t x = xlo + tid; x <= xhi; x += nthreads) {
            const uint32_t nw = (uint32_t)phi6(X / x);
            uint64_t acc = 0;
#pragma unroll 4
            for (uint32_t w = 1; w < nw; ++w)
                acc += R6[base + x * wheel_y(w) - 1];
            R6[base + x - 1] = 1ull - at_place(S, P, base + x - 1) - acc;
        }
    } else if (X / xhi < 1024) {
        for (uint64_t x = xlo + (tid >> 5); x <= xhi; x += nthreads >> 5) {
            const uint32_t nw = (uint32_t)phi6(X / x);
            uint64_t acc = 0;
#pragma unroll 4
            for (uint32_t w = 1 + lane; w < nw; w += 32)
                acc += R6[base + x * wheel_y(w) - 1];
            acc = warp_sum_u64(acc);
            if (lane == 0)
                R6[base + x - 1] = 1ull - at_place(S, P, base + x - 1) - acc;
        }
    } else {
        for (uint64_t x = xlo + tid / blockDim.x; x <= xhi; x += nthreads / blockDim.x) {
            const uint32_t nw = (uint32_t)phi6(X / x);
            uint64_t acc = 0;
#pragma unroll 4
            for (uint32_t w = 1 + threadIdx.x; w < nw; w += blockDim.x)
                acc += R6[base + x * wheel_y(w) - 1];
            acc = warp_sum_u64(acc);
            if (lane == 0)
                sh[warp] = acc;
            __syncthreads();
            if (warp == 0) {
                acc = warp_sum_u64(lane < nwarp ? sh[lane] : 0);
                if (lane == 0)
                    R6[base + x - 1] = 1ull - at_place(S, P, base + x - 1) - acc;
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ void resolve_final(const QueryDev &Q, const uint32_t *P, const uint64_t *A,
                                              const uint64_t *R6, uint64_t *R, uint64_t tid,
                                              uint64_t nthreads)
{
    const uint64_t X = Q.X, base = Q.off;
    for (uint64_t x = 1 + tid; x <= X; x += nthreads) {
        uint64_t v = R6[base + x - 1] + at_place(A, P, base + x - 1);
        if (2 * x <= X)
            v -= R6[base + 2 * x - 1];
        if (3 * x <= X)
            v -= R6[base + 3 * x - 1];
        if (6 * x <= X)
            v += R6[base + 6 * x - 1];
        R[base + x - 1] = v;
    }
}

// A CTA per target, all levels.  Bound by latency, level by level (n = 10^16: 0.4 ms
// with at most a warp per entry, 83 000 terms of x = 1 among them, 0.13 ms now).
__global__ void __launch_bounds__(1024) wheel_resolve_kernel(const QueryDev *__restrict__ qs,
                                                             const uint32_t *__restrict__ P,
                                                             const uint64_t *__restrict__ S,
                                                             const uint64_t *__restrict__ A,
                                                             uint64_t *R6, uint64_t *R)
{
    __shared__ uint64_t sh[32];
    const QueryDev Q = qs[blockIdx.x];
    for (uint64_t hi = Q.X; hi >= 1; hi /= 5) {
        resolve_level(Q, P, S, R6, hi / 5 + 1, hi, threadIdx.x, blockDim.x, sh);
        __syncthreads();
    }
    resolve_final(Q, P, A, R6, R, threadIdx.x, blockDim.x);
}

// One level (the last launch: the values of M) of every target, several CTAs each.
__global__ void __launch_bounds__(256) wheel_resolve_level_kernel(const QueryDev *__restrict__ qs,
                                                                  const uint32_t *__restrict__ P,
                                                                  const uint64_t *__restrict__ S,
                                                                  const uint64_t *__restrict__ A,
                                                                  uint64_t *R6, uint64_t *R,
                                                                  uint64_t div, uint32_t last)
{
    __shared__ uint64_t sh[32];
    const QueryDev Q = qs[blockIdx.y];
    const uint64_t tid = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t nt = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t hi = Q.X / div;
    if (last)
        resolve_final(Q, P, A, R6, R, tid, nt);
    else if (hi)
        resolve_level(Q, P, S, R6, hi / 5 + 1, hi, tid, nt, sh);
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
static int sm_count()
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return sms;
}

int wheel_dense_list_enqueue(const uint2 *Mg, uint64_t c0, uint64_t nchunks, uint16_t *dl,
                             uint32_t *dl_cnt, cudaStream_t s)
{
    wheel_dense_list_kernel<<<(unsigned)nchunks, 256, 0, s>>>(Mg, c0, dl, dl_cnt);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wheel_dense_enqueue(const WheelDenseArgs &a, uint64_t max_items, cudaStream_t s)
{
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, wheel_dense_kernel, kWheelDenseThreads, 0);
    const uint32_t grid = (uint32_t)std::min<uint64_t>((uint64_t)(sm_count() * std::max(per, 1)), max_items);
    cudaMemsetAsync(a.counter, 0, 4, s);
    wheel_dense_kernel<<<grid, kWheelDenseThreads, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wheel_gather_enqueue(const WheelGatherArgs &a, cudaStream_t s)
{
    if (a.nitems == 0)
        return 0;
    static std::atomic<uint64_t> attr_devs{0};
    const int smem = kGatherTile * 2 + 16 + 16 * 32 * 8;
    const uint64_t dbit = device_bit();
    if (attrs_needed(attr_devs, dbit)) {
        cudaFuncSetAttribute(wheel_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        attrs_done(attr_devs, dbit);
    }
    int per = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, wheel_gather_kernel, 512, smem);
    const uint32_t grid = std::min<uint32_t>((uint32_t)(sm_count() * std::max(per, 1)), a.nitems);
    cudaMemsetAsync(a.counter, 0, 4, s);
    wheel_gather_kernel<<<grid, 512, smem, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wheel_block_enqueue(const WheelBlockArgs &a, cudaStream_t s)
{
    cudaMemsetAsync(a.qlen, 0, 4, s);
    wheel_range_kernel<<<(unsigned)((a.nplaces + 255) / 256), 256, 0, s>>>(a);
    const uint32_t grid = std::min<uint32_t>((uint32_t)sm_count() * 8u, (a.qcap + 7u) / 8u);
    wheel_chunk_kernel<<<grid, 256, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

int wheel_wide_enqueue(const WheelWideArgs &a, uint32_t nw, uint64_t units, cudaStream_t s)
{
    if (nw == 0)
        return 0;
    const uint64_t gx = std::max<uint64_t>(1, (units + kWideUnitsPerCta - 1) / kWideUnitsPerCta);
    int n = 0;
    for (uint32_t w = 0; w < nw; w += 65535u, ++n) {  // grid.y is 16 bits
        WheelWideArgs b = a;
        b.W += w;
        wheel_wide_kernel<<<dim3((unsigned)gx, std::min(nw - w, 65535u)), kWideThreads, 0, s>>>(b);
    }
    return cudaGetLastError() == cudaSuccess ? n : -1;
}

int wheel_lookup_enqueue(const uint64_t *pairs, uint32_t count, const uint2 *Mg,
                         const int64_t *segoff, uint64_t *R, cudaStream_t s)
{
    if (count == 0)
        return 0;
    wheel_lookup_kernel<<<(count + 127) / 128, 128, 0, s>>>(pairs, count, Mg, segoff, R);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wheel_carry_at_enqueue(const uint2 *Mg, const int64_t *segoff, uint64_t y0, int64_t *out,
                           cudaStream_t s)
{
    wheel_carry_at_kernel<<<1, 1, 0, s>>>(Mg, segoff, y0 / 3 - 1, out);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int wheel_resolve_enqueue(const QueryDev *qs, uint32_t nq, uint64_t max_x, const uint32_t *P,
                          const uint64_t *S, const uint64_t *A, uint64_t *R6, uint64_t *R,
                          cudaStream_t s)
{
    if (max_x <= 16384 || nq >= 32) {
        wheel_resolve_kernel<<<nq, 1024, 0, s>>>(qs, P, S, A, R6, R);
        return cudaGetLastError() == cudaSuccess ? 1 : -1;
    }
    int n = 0;
    const dim3 grid((unsigned)std::min<uint64_t>((max_x + 255) / 256, 608), nq);
    for (uint64_t div = 1; div <= max_x; div *= 5, ++n)
        wheel_resolve_level_kernel<<<grid, 256, 0, s>>>(qs, P, S, A, R6, R, div, 0u);
    wheel_resolve_level_kernel<<<grid, 256, 0, s>>>(qs, P, S, A, R6, R, 1, 1u);
    return cudaGetLastError() == cudaSuccess ? n + 1 : -1;
}

}  // namespace mert
