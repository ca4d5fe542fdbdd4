// Steps a1 + a2 of a whole run over the integers coprime to 6 (wheel.h): the
// segmented log sieve with an exact decision rule and the fused prefix scan of
// the scale-2 byte kernel (sieve.cu), on a third of the integers.
//
// Byte w of a tile belongs to the wheel number y(w) and holds 1 + the sum of
// w2(p) over the distinct sieving primes p | y(w), w2(p) = 2 floor(log2 p) + 1
// (the odd integer nearest 2 log2 p), plus 128 when p^2 | y(w).  The sieving
// primes are 5 <= p <= P with P = max(1024, floor(sqrt(y2))).  With A the
// weight sum and E the largest number of distinct primes >= 5 dividing a
// y <= y2, A >= 2 log2 y - E when the sieved primes account for all of y and
// A <= 2 log2 y - 2 log2 P + E when one prime above P is left, so the
// threshold 2 log2 y - log2 P separates the two with log2 P - E either side:
// 10 - 5 at y2 = 2^20 and growing above (wheel_sieve_exact checks >= 2.5; an
// integer threshold anywhere in [T - 2, T] is then exact).
//
// A prime p hits two progressions of stride 2p in w: with i = w / 2, the
// class 6i + 1 at i = a0 (mod p) and the class 6i + 5 at i = a0 + d (mod p),
//   p = 1 (mod 6): a0 = (p - 1)/6,  d = 2 (p - 1)/3,
//   p = 5 (mod 6): a0 = (5p - 1)/6, d = (p - 2)/3.
//
// Measured (n = 10^16, u = 4 10^10, per run): every y 45.9 ms (the scale-2
// kernel of sieve.cu) -> 17.7 ms in this form -> 15.2 ms with squares below 1024
// by the descriptor jobs' lanes (one thread each stalled the rest at the barrier)
// -> 13.2 ms with 8 bytes written per 16 numbers: 265 us per block of 8.05e8 y.
// Bound by issue and by the shared atomics: of 330 us (decode still writing
// int16), lane primes took 106, descriptors 74, the decode 75, pattern copy and
// barriers 58.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "wheel.h"

namespace mert {

constexpr uint32_t kWPatPrimes = 3;           // table primes in the pattern: 5, 7, 11
constexpr uint32_t kWPatPeriod = 2u * 25u * 49u * 121u;  // in w
constexpr uint32_t kWPhases = 8;              // tile starts are even: phases 0, 2, .., 14
constexpr uint32_t kWTileBig = 98304;         // wheel numbers per tile
constexpr uint32_t kWTileSmall = 24576;
constexpr uint32_t kWPatLen = ((kWPatPeriod + kWTileBig + 31u) / 16u) * 16u;
constexpr uint32_t kWJobsMax = 192;           // descriptor jobs: primes 13 .. 1021
// Lane primes from 512 or 2048, and lists from 2048, measured slower at n = 10^16;
// so did tiles of 64 Ki (three CTAs per SM) and 48 Ki (four): 42.9 and 45.5 ms a
// run against 41.7.
constexpr uint32_t kWLaneMin = 1024;          // primes from here: a lane per prime
constexpr uint32_t kWListMin = 4096;          // squares from here: the block's lists
constexpr uint32_t kWSqCap = 64;
static_assert(kWLaneMin * kWLaneMin > kWTileBig / 2, "at most one square per class and tile");
static_assert((uint64_t)kWListMin * kWListMin < (1u << 26), "rec2 packs a residue mod p^2 in 26 bits");

// Pre-sieve pattern, kWPhases copies: copy k, byte j is wheel number j + 2k.
__global__ void wheel_pattern_kernel(uint8_t *__restrict__ pat)
{
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= kWPatLen)
        return;
    const uint32_t w = j + 2u * blockIdx.y;
    const uint32_t y = 3u * w + 1u + (w & 1u);
    uint32_t b = 1u;
    if (y % 5u == 0)
        b += 5u;  // 2 floor(log2 5) + 1
    if (y % 7u == 0)
        b += 5u;
    if (y % 11u == 0)
        b += 7u;
    if (y % 25u == 0 || y % 49u == 0 || y % 121u == 0)
        b |= 128u;
    pat[(size_t)blockIdx.y * kWPatLen + j] = (uint8_t)b;
}

// Per block (I0 = w0 / 2): for every sieving prime the record
//   rec  = {p, m32(p), (I0 - a0) mod p, s(p) | w2(p) << 8 | [p = 1 mod 6] << 16}
//   rec2 = {(I0 - a0(p^2)) mod p^2 | s(p^2) << 26, m32(p^2)}   (p < 4096)
// and, for p >= 4096, the multiples of p^2 as offsets into per-tile lists.
__global__ void wheel_prep_kernel(uint64_t I0, uint32_t np, const uint32_t *__restrict__ primes,
                                  uint4 *__restrict__ rec, uint2 *__restrict__ rec2, uint32_t ilen,
                                  uint32_t tile, uint32_t *__restrict__ cnt,
                                  uint32_t *__restrict__ list, uint32_t *__restrict__ err)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= np)
        return;
    const uint32_t p = primes[t];
    const bool one = p % 6u == 1u;
    const uint32_t a0 = one ? (p - 1u) / 6u : (uint32_t)((5ull * p - 1u) / 6u);
    unsigned s;
    const uint32_t m = magic32_of(p, &s);
    const uint32_t lg = 31u - __clz(p);
    const uint32_t r0 = (uint32_t)(I0 % p);
    const uint32_t r = r0 >= a0 ? r0 - a0 : r0 + p - a0;
    rec[t] = make_uint4(p, m, r, s | ((2u * lg + 1u) << 8) | (one ? 1u << 16 : 0u));
    const uint64_t q = (uint64_t)p * p;       // = 1 mod 6
    const uint64_t b0 = (q - 1u) / 6u, i0 = I0 % q;
    const uint64_t rr = i0 >= b0 ? i0 - b0 : i0 + q - b0;
    if (p < kWListMin) {
        unsigned s2;
        const uint32_t m2 = magic32_of((uint32_t)q, &s2);
        rec2[t] = make_uint2((uint32_t)rr | (s2 << 26), m2);
        return;
    }
    const uint64_t z0 = rr ? q - rr : 0;
    uint64_t z1 = z0 + 2u * (q / 3u);         // d(p^2) = 2 (p^2 - 1)/3
    if (z1 >= q)
        z1 -= q;
    for (uint32_t c = 0; c < 2; ++c)
        for (uint64_t i = c ? z1 : z0; i < ilen; i += q) {
            const uint32_t w = 2u * (uint32_t)i + c;
            const uint32_t ti = w / tile;
            const uint32_t slot = atomicAdd(&cnt[ti], 1u);
            if (slot < kWSqCap)
                list[(size_t)ti * kWSqCap + slot] = w - ti * tile;
            else
                atomicOr(err, kErrList);
        }
}

struct WSieveArgs {
    uint64_t w0;
    uint32_t tiles;
    uint32_t np, np_lane;   // primes used; [kWPatPrimes, np_lane) a warp per prime
    uint32_t np_list;       // [np_list, np): squares from the block's lists
    uint32_t len;           // wheel numbers in the block
    float log2P;
    const uint4 *rec;
    const uint2 *rec2;
    const uint4 *pat;
    uint32_t *sqcnt;
    const uint32_t *sqlist;
    uint2 *Mg;
    int32_t *segsum;
    uint32_t *err;
};

// First i >= the tile's of both classes of prime record q, as byte offsets
// 2 i and 2 i + 1 into the tile (T: the tile's first i within the block).
__device__ __forceinline__ void wheel_first(uint4 q, uint32_t T, uint32_t &b0, uint32_t &b1)
{
    const uint32_t p = q.x;
    const uint32_t v = q.z + T;  // < 2^31
    const uint32_t rem = v - div_magic32(v, q.y, q.w & 255u) * p;
    const uint32_t i0 = rem ? p - rem : 0u;
    uint32_t i1 = i0 + ((p / 3u) << ((q.w >> 16) & 1u));  // i0 + d
    if (i1 >= p)
        i1 -= p;
    b0 = 2u * i0;
    b1 = 2u * i1 + 1u;
}

// The same for the squares (record e), as byte offsets.
__device__ __forceinline__ void wheel_first_square(uint32_t p, uint2 e, uint32_t T, uint32_t &b0,
                                                   uint32_t &b1)
{
    const uint32_t q = p * p;    // < 2^24
    const uint32_t v = (e.x & 0x3ffffffu) + T;
    const uint32_t rem = v - div_magic32(v, e.y, e.x >> 26) * q;
    const uint32_t i0 = rem ? q - rem : 0u;
    uint32_t i1 = i0 + 2u * (q / 3u);
    if (i1 >= q)
        i1 -= q;
    b0 = 2u * i0;
    b1 = 2u * i1 + 1u;
}

__device__ __forceinline__ void wheel_flag(uint32_t *w, uint32_t b)
{
    atomicOr(&w[b >> 2], 0x80u << ((b & 3u) << 3));
}

// Descriptor job: the two progressions of one prime p < 1024, sixteen lanes
// each, and those of its square (first offsets sq).  32 p is a multiple of 4,
// so a lane's shifted weight is loop-invariant.
template <uint32_t TILE>
__device__ __forceinline__ void wheel_desc_job(uint4 d, uint2 sq, uint32_t *w, uint32_t lane)
{
    const uint32_t p = d.z & 0xffffu;
    for (uint32_t b = ((lane & 1u) ? sq.y : sq.x) + (lane >> 1) * 2u * p * p; b < TILE;
         b += 32u * p * p)
        wheel_flag(w, b);
    const uint32_t b = ((lane & 1u) ? d.y : d.x) + (lane >> 1) * 2u * p;
    if (b >= TILE)
        return;
    const uint32_t wsh = (d.z >> 16) << ((b & 3u) << 3);
    const uint32_t step = 8u * p;                       // words per 16 multiples
    const uint32_t end = (TILE + 3u - (b & 3u)) >> 2;   // b' < TILE <=> b' >> 2 < end
    uint32_t wi = b >> 2;
    for (; wi + 3u * step < end; wi += 4u * step) {
        atomicAdd(&w[wi], wsh);
        atomicAdd(&w[wi + step], wsh);
        atomicAdd(&w[wi + 2u * step], wsh);
        atomicAdd(&w[wi + 3u * step], wsh);
    }
    for (; wi < end; wi += step)
        atomicAdd(&w[wi], wsh);
}

// One prime p >= 1024 over the whole tile (one lane).  The two progressions
// interleave: lo, hi, lo + 2p, hi + 2p, ...; 2p = 2 (mod 4), so a
// progression's shifted weight alternates with its rotation by 16 bits.
template <uint32_t TILE>
__device__ __forceinline__ void wheel_lane_prime(uint4 q, uint32_t *w, uint32_t T)
{
    uint32_t b0, b1;
    wheel_first(q, T, b0, b1);
    const uint32_t p2 = 2u * q.x;
    uint32_t lo = min(b0, b1), hi = max(b0, b1);
    const uint32_t wt = (q.w >> 8) & 255u;
    if (p2 < TILE / 2u) {
        const uint32_t l0 = wt << ((lo & 3u) << 3), h0 = wt << ((hi & 3u) << 3);
        const uint32_t l1 = __funnelshift_l(l0, l0, 16), h1 = __funnelshift_l(h0, h0, 16);
        for (; hi + p2 < TILE; lo += 2u * p2, hi += 2u * p2) {
            atomicAdd(&w[lo >> 2], l0);
            atomicAdd(&w[hi >> 2], h0);
            atomicAdd(&w[(lo + p2) >> 2], l1);
            atomicAdd(&w[(hi + p2) >> 2], h1);
        }
        if (lo < TILE) {
            atomicAdd(&w[lo >> 2], l0);
            if (hi < TILE) {
                atomicAdd(&w[hi >> 2], h0);
                if (lo + p2 < TILE)
                    atomicAdd(&w[(lo + p2) >> 2], l1);
            }
        }
    } else if (p2 < TILE) {
        for (; lo < TILE; lo += p2)
            atomicAdd(&w[lo >> 2], __funnelshift_l(0u, wt, lo << 3));
        for (; hi < TILE; hi += p2)
            atomicAdd(&w[hi >> 2], __funnelshift_l(0u, wt, hi << 3));
    } else {
        if (lo < TILE)
            atomicAdd(&w[lo >> 2], __funnelshift_l(0u, wt, lo << 3));
        if (hi < TILE)
            atomicAdd(&w[hi >> 2], __funnelshift_l(0u, wt, hi << 3));
    }
}

// Decode + scan of one 2048-number segment (one warp): per byte the square flag
// and, from the sign of W = (byte & 127) + bias and the weight sum's parity, mu =
// -1; two words' flags become eight bits by dot products.  A round covers 1024
// numbers, each lane 16 at 16 lane and 16 at 512 + 16 lane; one warp scan carries
// both halves' lane sums packed in one int32.  kTileThr: one threshold for the
// tile (bias4); otherwise a threshold per number.  Returns the segment's sum.
template <bool kTileThr>
__device__ __forceinline__ int wheel_segment(const WSieveArgs &a, const uint4 *sb, uint64_t wt0,
                                             uint32_t so, uint32_t lane, uint32_t bias4,
                                             uint2 *dst0)
{
    int run = 0;
#pragma unroll 1
    for (uint32_t r = 0; r < (uint32_t)kSegY / 1024u; ++r) {
        uint32_t bits[2];
        int tot[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t o0 = so + r * 1024u + (uint32_t)h * 512u + lane * 16u;
            const uint4 q4 = sb[o0 >> 4];
            const uint32_t ws[4] = {q4.x, q4.y, q4.z, q4.w};
            uint32_t free8[2] = {0, 0}, neg8[2] = {0, 0};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t nsq = ~(ws[k] >> 7) & 0x01010101u;
                uint32_t m;
                if (kTileThr) {
                    const uint32_t W = (ws[k] & 0x7f7f7f7fu) + bias4;
                    m = (W ^ (W >> 7)) & nsq;
                } else {
                    m = 0;
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t y = wheel_y(wt0 + o0 + 4u * k + j);
                        const int A = (int)((ws[k] >> (8 * j)) & 127u) - 1;
                        const int th =
                            (int)floorf(2.0f * __log2f(__ull2float_rn(y)) - a.log2P);
                        const uint32_t bit = ((uint32_t)A & 1u) ^ (A > th ? 0u : 1u);
                        m |= bit << (8 * j);
                    }
                    m &= nsq;
                }
                const uint32_t weights = (k & 1) ? 0x80402010u : 0x08040201u;
                free8[k >> 1] = __dp4a(nsq, weights, free8[k >> 1]);
                neg8[k >> 1] = __dp4a(m, weights, neg8[k >> 1]);
            }
            const uint32_t sf = free8[0] | (free8[1] << 8), ng = neg8[0] | (neg8[1] << 8);
            bits[h] = sf | (ng << 16);
            tot[h] = __popc(sf) - 2 * __popc(ng);
        }
        int inc = tot[0] + tot[1] * 65536;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int nb = __shfl_up_sync(0xffffffffu, inc, o);
            if ((int)lane >= o)
                inc += nb;
        }
        const int all = __shfl_sync(0xffffffffu, inc, 31);
        const int incA = (int)(int16_t)(inc & 0xffff), incB = (inc - incA) >> 16;
        const int allA = (int)(int16_t)(all & 0xffff), allB = (all - allA) >> 16;
        uint2 *dst = dst0 + ((so + r * 1024u) >> kMgShift) + lane;
        dst[0] = make_uint2(bits[0], (uint32_t)(run + incA - tot[0]));
        dst[32] = make_uint2(bits[1], (uint32_t)(run + allA + incB - tot[1]));
        run += allA + allB;
    }
    return run;
}

// The low tiles (a threshold per number), in a function of their own so that
// they hold no registers of the common path.
__device__ __noinline__ int wheel_segment_low(const WSieveArgs &a, const uint4 *sb, uint64_t wt0,
                                              uint32_t so, uint32_t lane, uint2 *dst0)
{
    return wheel_segment<false>(a, sb, wt0, so, lane, 0u, dst0);
}

// One tile of TILE wheel numbers (3 TILE y): the pattern by one bulk
// asynchronous copy, overlapped with the descriptors of the primes below
// 1024; descriptor jobs (a warp per prime), then 128 primes >= 1024 at a time
// (four per lane) from a shared counter; decode and scan.
template <uint32_t TILE, int THREADS, int MINB>
__global__ void __launch_bounds__(THREADS, MINB) wheel_sieve_kernel(WSieveArgs a)
{
    static_assert(TILE == THREADS * 128, "each warp decodes two segments");
    static_assert(THREADS >= (int)kWJobsMax, "one descriptor per thread");
    extern __shared__ uint4 sb[];
    uint32_t *w = reinterpret_cast<uint32_t *>(sb);
    __shared__ uint32_t s_job;
    __shared__ uint4 s_jd[kWJobsMax];
    __shared__ uint2 s_sq[kWJobsMax];
    __shared__ uint64_t s_mbar;
    const uint32_t a0 = blockIdx.x * TILE;   // first number of the tile in the block
    const uint32_t T = a0 >> 1;              // its i
    const uint64_t wt0 = a.w0 + a0;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t jd = a.np_lane - kWPatPrimes;
    const uint32_t jobs = jd + (a.np - a.np_lane + 127u) / 128u;
    const uint32_t nsq = min(a.sqcnt[blockIdx.x], kWSqCap);

    if (threadIdx.x == 0) {
        const uint32_t ph = (uint32_t)(wt0 % kWPatPeriod);  // even
        mbar_init(&s_mbar);
        fence_proxy_async_smem();
        mbar_arrive_expect(&s_mbar, TILE);
        bulk_copy_g2s(sb, a.pat + (size_t)((ph & 15u) >> 1) * (kWPatLen / 16) + (ph >> 4), TILE,
                      &s_mbar);
        s_job = 0;
    }
    if (threadIdx.x < jd) {
        const uint32_t t = kWPatPrimes + threadIdx.x;
        const uint4 q = a.rec[t];
        uint32_t b0, b1;
        wheel_first(q, T, b0, b1);
        s_jd[threadIdx.x] = make_uint4(b0, b1, q.x | (((q.w >> 8) & 255u) << 16), 0u);
        wheel_first_square(q.x, a.rec2[t], T, b0, b1);
        s_sq[threadIdx.x] = make_uint2(b0, b1);
    }
    __syncthreads();  // the mbarrier is initialised; every thread has read sqcnt
    if (__syncthreads_or(!mbar_wait(&s_mbar, 0u))) {
        if (threadIdx.x == 0) {
            a.sqcnt[blockIdx.x] = 0;
            atomicOr(a.err, kErrTimeout);
        }
        mbar_wait(&s_mbar, 0u);
        return;
    }
    if (threadIdx.x == 0)
        a.sqcnt[blockIdx.x] = 0;  // read above; cleared for the next block
    // squares: p < 1024 in the descriptor jobs, 1024 <= p < 4096 a thread per
    // prime (at most one per class), the rest from the list
    for (uint32_t t = a.np_lane + threadIdx.x; t < a.np_list; t += THREADS) {
        uint32_t b0, b1;
        wheel_first_square(a.rec[t].x, a.rec2[t], T, b0, b1);
        if (b0 < TILE)
            wheel_flag(w, b0);
        if (b1 < TILE)
            wheel_flag(w, b1);
    }
    {
        const uint32_t *ls = a.sqlist + (size_t)blockIdx.x * kWSqCap;
        for (uint32_t i = threadIdx.x; i < nsq; i += THREADS)
            wheel_flag(w, ls[i]);
    }
    for (;;) {
        uint32_t job = 0;
        if (lane == 0)
            job = atomicAdd(&s_job, 1u);
        job = __shfl_sync(0xffffffffu, job, 0);
        if (job >= jobs)
            break;
        if (job < jd) {
            wheel_desc_job<TILE>(s_jd[job], s_sq[job], w, lane);
        } else {
            // a lane takes primes i and 63 - i of each half of the job, so
            // the lanes' hit counts even out
#pragma unroll 1
            for (uint32_t hb = 0; hb < 128u; hb += 64u) {
                const uint32_t b0 = a.np_lane + (job - jd) * 128u + hb;
                const uint32_t t0 = b0 + lane, t1 = b0 + 63u - lane;
                uint4 q0 = make_uint4(0, 0, 0, 0), q1 = q0;
                if (t0 < a.np)
                    q0 = a.rec[t0];
                if (t1 < a.np)
                    q1 = a.rec[t1];
                if (t0 < a.np)
                    wheel_lane_prime<TILE>(q0, w, T);
                if (t1 < a.np)
                    wheel_lane_prime<TILE>(q1, w, T);
            }
        }
    }
    __syncthreads();

    const uint64_t y1 = wheel_y(wt0);
    const bool tile_thr = y1 >= kByteTileThrMin;
    uint32_t bias4 = 0;
    if (tile_thr) {
        const int thr = (int)floorf(2.0f * log2f(__ull2float_rn(y1)) - a.log2P) & ~1;
        bias4 = (uint32_t)(126 - thr) * 0x01010101u;
    }
    uint2 *dst0 = a.Mg + (a0 >> kMgShift);
    for (uint32_t sgi = 0; sgi < 2; ++sgi) {
        const uint32_t so = warp * (2u * kSegY) + sgi * kSegY;
        if (a0 + so >= a.len)
            break;
        const int run = tile_thr ? wheel_segment<true>(a, sb, wt0, so, lane, bias4, dst0)
                                 : wheel_segment_low(a, sb, wt0, so, lane, dst0);
        if (lane == 0)
            a.segsum[(a0 + so) >> kSegShift] = run;
    }
}

// a2 finish: segoff[s] = carry_in + sum of segsum[0..s), carry_out = carry_in
// + all of them.  Each CTA scans 4096 segments, four per thread, and adds the sum
// of all segments before its range (16-byte loads).  Bound by latency: 10 us for
// 131 072 segments (12 us with one segment per thread).
__global__ void __launch_bounds__(1024) seg_carry_kernel(const int32_t *__restrict__ segsum,
                                                           uint32_t nseg,
                                                           const int64_t *__restrict__ carry_in,
                                                           int64_t *__restrict__ segoff,
                                                           int64_t *__restrict__ carry_out)
{
    __shared__ int64_t sh[33];
    const uint32_t base = blockIdx.x * 4096u;
    int64_t before = 0;
    const int4 *s4 = reinterpret_cast<const int4 *>(segsum);
    for (uint32_t i = threadIdx.x; i < base / 4u; i += 1024u) {
        const int4 v = s4[i];
        before += (int64_t)v.x + v.y + v.z + v.w;
    }
    int64_t tb;
    block_excl_scan<int64_t>(before, sh, &tb);
    const uint32_t i = base + 4u * threadIdx.x;
    int32_t v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        v[k] = i + k < nseg ? segsum[i + k] : 0;
    int64_t tot;
    const int64_t ex =
        block_excl_scan<int64_t>((int64_t)v[0] + v[1] + v[2] + v[3], sh, &tot);
    const int64_t c0 = *carry_in;
    int64_t o = c0 + tb + ex;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (i + k < nseg)
            segoff[i + k] = o;
        o += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0)
        *carry_out = c0 + tb + tot;
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
static uint64_t isqrt_floor(uint64_t v)
{
    uint64_t r = (uint64_t)std::sqrt((double)v);
    while (r > 0 && r > v / r)
        --r;
    while ((r + 1) <= v / (r + 1))
        ++r;
    return r;
}

// Sieving bound of a block ending at y2.
static uint64_t sieve_bound(uint64_t y2) { return std::max<uint64_t>(kWLaneMin, isqrt_floor(y2)); }

// Most distinct primes >= 5 dividing any y' <= y.
static int omega_wheel(uint64_t y)
{
    static const uint32_t pr[12] = {5, 7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43};
    uint64_t v = 1;
    int w = 0;
    while (w < 12 && v <= y / pr[w])
        v *= pr[w++];
    return w;
}

// The decision rule is exact for every block below y_max: log2 P - E >= 2.5,
// sums below 2^7, thresholds and biased bytes within their fields.  E steps
// up only at the products of the first primes >= 5, where P = max(1024, sqrt y)
// is smallest for it, so the products and y_max itself are checked.
bool wheel_sieve_exact(uint64_t y_max)
{
    if (y_max >= (1ull << 54))
        return false;
    static const uint32_t pr[12] = {5, 7, 11, 13, 17, 19, 23, 29, 31, 37, 41, 43};
    uint64_t v = 1;
    for (int i = -1; i < 13; ++i) {
        if (i >= 0 && i < 12 && v <= y_max / pr[i])
            v *= pr[i];
        else if (i >= 0)
            v = y_max;
        const double P = std::log2((double)sieve_bound(v));
        const double E = omega_wheel(v), top = 2.0 * std::log2((double)v) + E;
        const double thr = 2.0 * std::log2((double)v) - P;
        if (P < E + 2.5 || thr >= 124.0 || 1.0 + top >= 127.0 || top - (thr - 2.0) + 127.0 >= 255.0)
            return false;
        if (v == y_max)
            break;
    }
    return true;
}

void wheel_sieve_primes(WheelSieve *t, uint64_t y_max)
{
    // the last block is rounded up to a whole segment
    const uint64_t B = sieve_bound(y_max + kWheelSegY);
    std::vector<uint8_t> comp(B / 2 + 1, 0);  // odd numbers 2i + 1
    t->host_p.clear();
    for (uint64_t q = 3; q <= B; q += 2) {
        if (comp[q >> 1])
            continue;
        if (q >= 5)
            t->host_p.push_back((uint32_t)q);
        for (uint64_t j = q * q; j <= B; j += 2 * q)
            comp[j >> 1] = 1;
    }
}

// Lays the arrays out from `base` (null: only counts); returns the bytes.
static size_t wheel_layout(WheelSieve *t, size_t np, uint64_t max_len, char *base, size_t *clear)
{
    const uint64_t nt = (max_len + kWTileSmall - 1) / kWTileSmall;
    size_t off = 0;
    const auto take = [&](size_t bytes) {
        char *q = base + off;
        off += (bytes + 255) & ~(size_t)255;
        return q;
    };
    char *c0 = take(nt * 4), *pat = take((size_t)kWPhases * kWPatLen), *p = take(np * 4),
         *rec = take(np * sizeof(uint4)), *rec2 = take(np * sizeof(uint2)),
         *list = take(nt * kWSqCap * 4);
    if (t) {
        t->sqcnt = (uint32_t *)c0;
        t->pat = (uint4 *)pat;
        t->p = (uint32_t *)p;
        t->rec = (uint4 *)rec;
        t->rec2 = (uint2 *)rec2;
        t->sqlist = (uint32_t *)list;
        *clear = nt * 4;
    }
    return off;
}

size_t wheel_sieve_bytes(const WheelSieve *t, uint64_t max_len)
{
    return wheel_layout(nullptr, t->host_p.size(), max_len, nullptr, nullptr);
}

int wheel_sieve_bind(WheelSieve *t, void *base, uint64_t max_len, uint32_t *err, cudaStream_t s)
{
    size_t clear = 0;
    wheel_layout(t, t->host_p.size(), max_len, (char *)base, &clear);
    t->err = err;
    cudaMemsetAsync(t->sqcnt, 0, clear, s);
    wheel_pattern_kernel<<<dim3((kWPatLen + 255) / 256, kWPhases), 256, 0, s>>>((uint8_t *)t->pat);
    return cudaGetLastError() == cudaSuccess ? 0 : 3;
}

uint32_t wheel_primes_upto(const WheelSieve *t, uint64_t b)
{
    return (uint32_t)(std::upper_bound(t->host_p.begin(), t->host_p.end(),
                                       (uint32_t)std::min<uint64_t>(b, 0xffffffffu)) -
                      t->host_p.begin());
}

void seg_carry_enqueue(const int32_t *segsum, uint32_t nseg, const int64_t *carry_in,
                       int64_t *segoff, int64_t *carry_out, cudaStream_t s)
{
    seg_carry_kernel<<<(nseg + 4095) / 4096, 1024, 0, s>>>(segsum, nseg, carry_in, segoff,
                                                           carry_out);
}

template <uint32_t TILE, int THREADS, int MINB>
static int wheel_launch(const WheelSieve *t, const WheelLaunch &L, cudaStream_t s)
{
    static std::atomic<uint64_t> attr_devs{0};
    const uint64_t dbit = device_bit();
    if (attrs_needed(attr_devs, dbit)) {
        cudaFuncSetAttribute(wheel_sieve_kernel<TILE, THREADS, MINB>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, TILE);
        attrs_done(attr_devs, dbit);
    }
    const uint64_t y2 = wheel_y(L.w0 + L.len - 1);
    const uint64_t P = sieve_bound(y2);
    WSieveArgs a{};
    a.w0 = L.w0;
    a.len = (uint32_t)L.len;
    a.tiles = (uint32_t)((L.len + TILE - 1) / TILE);
    a.np = wheel_primes_upto(t, P);
    a.np_lane = std::min(wheel_primes_upto(t, kWLaneMin - 1), a.np);
    a.np_list = std::min(wheel_primes_upto(t, kWListMin - 1), a.np);
    a.log2P = (float)std::log2((double)P);
    a.rec = t->rec;
    a.rec2 = t->rec2;
    a.pat = t->pat;
    a.sqcnt = t->sqcnt;
    a.sqlist = t->sqlist;
    a.Mg = L.Mg;
    a.segsum = L.segsum;
    a.err = t->err;
    wheel_prep_kernel<<<(a.np + 127) / 128, 128, 0, s>>>(L.w0 / 2, a.np, t->p, t->rec, t->rec2,
                                                         (uint32_t)(L.len / 2), TILE, t->sqcnt,
                                                         t->sqlist, t->err);
    wheel_sieve_kernel<TILE, THREADS, MINB><<<a.tiles, THREADS, TILE, s>>>(a);
    return 2;
}

int wheel_sieve_enqueue(const WheelSieve *t, const WheelLaunch &L, cudaStream_t s)
{
    // small tiles while the large ones would leave SMs without a CTA (two per
    // SM): n = 10^10 0.131 against 0.147 ms a run, 10^12 in blocks of 5 10^7 y 0.36
    // against 0.39; small ones always: 10^16 54 against 39.4
    int launches = L.len < 304ull * kWTileBig ? wheel_launch<kWTileSmall, 192, 8>(t, L, s)
                                              : wheel_launch<kWTileBig, 768, 2>(t, L, s);
    if (L.mid)
        cudaEventRecord(L.mid, s);
    if (L.mid2)
        cudaEventRecord(L.mid2, s);
    const uint32_t nseg = (uint32_t)(L.len >> kSegShift);
    seg_carry_enqueue(L.segsum, nseg, L.carry_in, L.segoff, L.carry_out, s);
    return cudaGetLastError() == cudaSuccess ? launches + 1 : -1;
}

}  // namespace mert
