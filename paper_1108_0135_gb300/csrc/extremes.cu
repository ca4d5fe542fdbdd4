// Interval scan: M(y) for every y of [y_first, y_last] from a known
// M(y_first - 1), by the sieve and prefix scan (steps a1 + a2, Sec. 3), and
// the extremes of M(y) and of M(y)/sqrt(y) over the interval -- the search
// that Sec. 6 of the paper runs around its candidate to find the new extreme
// value of M(n)/sqrt(n).  Ratios are compared exactly: for M1, M2 >= 0,
// M1/sqrt(y1) > M2/sqrt(y2) iff M1^2 y2 > M2^2 y1 (128-bit products).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/libmertens.h"
#include "common.cuh"
#include "internal.h"

using namespace mert;

namespace {

typedef unsigned __int128 u128;

// Running extremes; ties go to the smaller y.
struct Ext {
    int64_t mx, mn;    // largest and smallest M(y)
    uint64_t ymx, ymn;
    int64_t rpM, rnM;  // M at the largest and smallest M(y)/sqrt(y)
    uint64_t rpy, rny;
};

// a/sqrt(ya) > b/sqrt(yb) exactly
__host__ __device__ inline bool ratio_gt(int64_t a, uint64_t ya, int64_t b, uint64_t yb)
{
    if ((a >= 0) != (b >= 0))
        return a >= 0;
    const u128 aa = (u128)(uint64_t)(a >= 0 ? a : -a), bb = (u128)(uint64_t)(b >= 0 ? b : -b);
    const u128 l = aa * aa * yb, r = bb * bb * ya;
    return a >= 0 ? l > r : l < r;
}

__host__ __device__ inline void ext_init(Ext &e)
{
    e.mx = INT64_MIN;
    e.mn = INT64_MAX;
    e.ymx = e.ymn = e.rpy = e.rny = UINT64_MAX;
    e.rpM = e.rnM = 0;
}

__host__ __device__ inline void ext_point(Ext &e, int64_t M, uint64_t y)
{
    if (M > e.mx || (M == e.mx && y < e.ymx)) {
        e.mx = M;
        e.ymx = y;
    }
    if (M < e.mn || (M == e.mn && y < e.ymn)) {
        e.mn = M;
        e.ymn = y;
    }
    if (e.rpy == UINT64_MAX || ratio_gt(M, y, e.rpM, e.rpy) ||
        (!ratio_gt(e.rpM, e.rpy, M, y) && y < e.rpy)) {
        e.rpM = M;
        e.rpy = y;
    }
    if (e.rny == UINT64_MAX || ratio_gt(e.rnM, e.rny, M, y) ||
        (!ratio_gt(M, y, e.rnM, e.rny) && y < e.rny)) {
        e.rnM = M;
        e.rny = y;
    }
}

__host__ __device__ inline void ext_merge(Ext &e, const Ext &o)
{
    if (o.ymx != UINT64_MAX && (o.mx > e.mx || (o.mx == e.mx && o.ymx < e.ymx))) {
        e.mx = o.mx;
        e.ymx = o.ymx;
    }
    if (o.ymn != UINT64_MAX && (o.mn < e.mn || (o.mn == e.mn && o.ymn < e.ymn))) {
        e.mn = o.mn;
        e.ymn = o.ymn;
    }
    if (o.rpy != UINT64_MAX &&
        (e.rpy == UINT64_MAX || ratio_gt(o.rpM, o.rpy, e.rpM, e.rpy) ||
         (!ratio_gt(e.rpM, e.rpy, o.rpM, o.rpy) && o.rpy < e.rpy))) {
        e.rpM = o.rpM;
        e.rpy = o.rpy;
    }
    if (o.rny != UINT64_MAX &&
        (e.rny == UINT64_MAX || ratio_gt(e.rnM, e.rny, o.rnM, o.rny) ||
         (!ratio_gt(o.rnM, o.rny, e.rnM, e.rny) && o.rny < e.rny))) {
        e.rnM = o.rnM;
        e.rny = o.rny;
    }
}

constexpr int kExtThreads = 256;
constexpr uint32_t kExtWarps = kExtThreads / 32;
constexpr uint32_t kExtSegs = 4;      // segments per warp of the first pass
constexpr uint32_t kExtScan = 304;    // CTAs of the exact pass

// The scan of a block is bound by reading its int16 M(y) once (2 GB per 2^30
// y); the exact comparison of every M(y)/sqrt(y) in 128 bits took 18.1 ms per
// 2^30 y (instruction-bound).  So: (1) the largest and smallest M of every
// 2048-y segment, by packed 16-bit maxima; (2) of every segment [a, b] the
// bounds of M/sqrt(y) that these give -- a positive largest M is reached at some
// y <= b, and no ratio of the segment is above it at y = a (a negative one:
// the other way round) -- and the best lower bound of the block; (3) only the
// segments whose upper bound reaches it, or that hold the block's extreme M,
// are compared point by point.
__device__ __forceinline__ Ext ext_shfl(const Ext &e, int src)
{
    Ext o;
    o.mx = __shfl_down_sync(0xffffffffu, e.mx, src);
    o.mn = __shfl_down_sync(0xffffffffu, e.mn, src);
    o.ymx = __shfl_down_sync(0xffffffffu, e.ymx, src);
    o.ymn = __shfl_down_sync(0xffffffffu, e.ymn, src);
    o.rpM = __shfl_down_sync(0xffffffffu, e.rpM, src);
    o.rnM = __shfl_down_sync(0xffffffffu, e.rnM, src);
    o.rpy = __shfl_down_sync(0xffffffffu, e.rpy, src);
    o.rny = __shfl_down_sync(0xffffffffu, e.rny, src);
    return o;
}

// The CTA's records into one (thread 0's return value).
__device__ __forceinline__ Ext ext_reduce(Ext e, Ext *sh)
{
    for (int o = 16; o > 0; o >>= 1) {
        const Ext q = ext_shfl(e, o);
        ext_merge(e, q);
    }
    if ((threadIdx.x & 31) == 0)
        sh[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x == 0)
        for (uint32_t w = 1; w < kExtWarps; ++w)
            ext_merge(e, sh[w]);
    return e;
}

// Bounds of a segment [a, b] with largest value M (smallest: of -M):
// `reached` is at most a ratio that occurs, `limit` at least every ratio.
__device__ __forceinline__ uint64_t ext_reached(int64_t M, uint64_t a, uint64_t b)
{
    return M >= 0 ? b : a;
}
__device__ __forceinline__ uint64_t ext_limit(int64_t M, uint64_t a, uint64_t b)
{
    return M >= 0 ? a : b;
}

// Pass 1: {max, min} of every segment into mm (16-bit halves), and per CTA the
// extreme M (its segment's first y in ymx, ymn) and the best reached ratios.
__global__ void __launch_bounds__(kExtThreads) segment_extremes_kernel(
    uint64_t y1, uint64_t len, uint32_t nseg, const int16_t *__restrict__ Mloc,
    const int64_t *__restrict__ segoff, uint32_t *__restrict__ mm, Ext *__restrict__ part)
{
    __shared__ Ext sh[kExtWarps];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    Ext e;
    ext_init(e);
    for (uint32_t q = 0; q < kExtSegs; ++q) {
        const uint32_t sg = (blockIdx.x * kExtWarps + warp) * kExtSegs + q;
        if (sg >= nseg)
            break;
        const uint64_t i0 = (uint64_t)sg << kSegShift;
        uint32_t hi = 0x80008000u, lo = 0x7fff7fffu;
        if (i0 + kSegY <= len) {
            const uint4 *v = reinterpret_cast<const uint4 *>(Mloc + i0);
#pragma unroll
            for (uint32_t r = 0; r < (uint32_t)kSegY / 256u; ++r) {
                const uint4 x = v[r * 32u + lane];
                hi = __vmaxs2(__vmaxs2(__vmaxs2(hi, x.x), __vmaxs2(x.y, x.z)), x.w);
                lo = __vmins2(__vmins2(__vmins2(lo, x.x), __vmins2(x.y, x.z)), x.w);
            }
        } else {
            for (uint64_t i = i0 + lane; i < len; i += 32u) {
                const uint32_t x = (uint16_t)Mloc[i] * 0x00010001u;
                hi = __vmaxs2(hi, x);
                lo = __vmins2(lo, x);
            }
        }
        const int mx = __reduce_max_sync(0xffffffffu, max((int)(int16_t)(hi & 0xffffu),
                                                          (int)(int16_t)(hi >> 16)));
        const int mn = __reduce_min_sync(0xffffffffu, min((int)(int16_t)(lo & 0xffffu),
                                                          (int)(int16_t)(lo >> 16)));
        if (lane == q) {
            mm[sg] = (uint32_t)(uint16_t)mx | ((uint32_t)(uint16_t)mn << 16);
            Ext o;
            const uint64_t a = y1 + i0, b = y1 + min(i0 + kSegY, len) - 1;
            o.mx = segoff[sg] + mx;
            o.mn = segoff[sg] + mn;
            o.ymx = o.ymn = a;
            o.rpM = o.mx;
            o.rpy = ext_reached(o.mx, a, b);
            o.rnM = o.mn;
            o.rny = ext_reached(-o.mn, a, b);
            ext_merge(e, o);
        }
    }
    e = ext_reduce(e, sh);
    if (threadIdx.x == 0)
        part[blockIdx.x] = e;
}

// The records i = b, b + grid, ... into part[b] (which no other CTA reads).
__global__ void __launch_bounds__(kExtThreads) merge_extremes_kernel(Ext *part, uint32_t n)
{
    __shared__ Ext sh[kExtWarps];
    Ext e;
    ext_init(e);
    for (uint64_t i = blockIdx.x + (uint64_t)threadIdx.x * gridDim.x; i < n;
         i += (uint64_t)kExtThreads * gridDim.x)
        ext_merge(e, part[i]);
    __syncthreads();
    e = ext_reduce(e, sh);
    if (threadIdx.x == 0)
        part[blockIdx.x] = e;
}

// All records into part[0]: a record per thread, then one CTA (one CTA alone took
// 86 us for the 16 384 records of 2^30 y).
void merge_extremes(Ext *part, uint32_t n, cudaStream_t s)
{
    const uint32_t ctas = std::min((n + kExtThreads - 1) / kExtThreads, (uint32_t)kExtThreads);
    if (ctas > 1)
        merge_extremes_kernel<<<ctas, kExtThreads, 0, s>>>(part, n);
    merge_extremes_kernel<<<1, kExtThreads, 0, s>>>(part, ctas > 1 ? ctas : n);
}

// Pass 3: the exact extremes over the segments that can hold one, given the
// block's best record in best[0]; a record per CTA.
__global__ void __launch_bounds__(kExtThreads) exact_extremes_kernel(
    uint64_t y1, uint64_t len, uint32_t nseg, const int16_t *__restrict__ Mloc,
    const int64_t *__restrict__ segoff, const uint32_t *__restrict__ mm,
    const Ext *__restrict__ best, Ext *__restrict__ part)
{
    __shared__ Ext sh[kExtWarps];
    __shared__ uint32_t s_list[kExtThreads], s_n;
    const Ext B = best[0];
    Ext e;
    ext_init(e);
    for (uint32_t s0 = blockIdx.x * kExtThreads; s0 < nseg; s0 += gridDim.x * kExtThreads) {
        const uint32_t sg = s0 + threadIdx.x;
        if (threadIdx.x == 0)
            s_n = 0;
        __syncthreads();
        if (sg < nseg) {
            const int64_t so = segoff[sg];
            const int64_t mx = so + (int16_t)(mm[sg] & 0xffffu), mn = so + (int16_t)(mm[sg] >> 16);
            const uint64_t i0 = (uint64_t)sg << kSegShift;
            const uint64_t a = y1 + i0, b = y1 + min(i0 + kSegY, len) - 1;
            if ((mx == B.mx && a == B.ymx) || (mn == B.mn && a == B.ymn) ||
                !ratio_gt(B.rpM, B.rpy, mx, ext_limit(mx, a, b)) ||
                !ratio_gt(mn, ext_limit(-mn, a, b), B.rnM, B.rny))
                s_list[atomicAdd(&s_n, 1u)] = sg;
        }
        __syncthreads();
        // the segments left, one after the other by the whole CTA (a warp each took
        // 72 us for the seven of a last block)
        const uint32_t n = s_n;
        for (uint32_t q = 0; q < n; ++q) {
            const uint64_t i0 = (uint64_t)s_list[q] << kSegShift;
            const uint64_t i1 = min(i0 + kSegY, len);
            const int64_t so = segoff[i0 >> kSegShift];
            for (uint64_t i = i0 + threadIdx.x; i < i1; i += kExtThreads)
                ext_point(e, so + (int64_t)Mloc[i], y1 + i);
        }
        __syncthreads();
    }
    e = ext_reduce(e, sh);
    if (threadIdx.x == 0)
        part[blockIdx.x] = e;
}

}  // namespace

extern "C" {

int mertens_scan_extremes(uint64_t y_first, uint64_t y_last, int64_t carry,
                          mertens_extremes *out, void *stream)
{
    if (!out || y_first == 0 || y_last < y_first || y_last >= (1ull << 62)) {
        set_last_error("mertens_scan_extremes: need 1 <= y_first <= y_last < 2^62 and an output");
        return MERTENS_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const Allocator al = current_allocator();
    const uint64_t span = y_last - y_first + 1;
    const uint64_t L = std::min<uint64_t>(1ull << 30, ((span + kSegY - 1) / kSegY) * kSegY);
    const uint64_t nblocks = (span + L - 1) / L;
    const uint64_t nseg = sieve_segments(L);
    const uint64_t ctas = (nseg + kExtWarps * kExtSegs - 1) / (kExtWarps * kExtSegs);
    const uint64_t nparts = nblocks * kExtScan;  // records of the exact passes
    if (nblocks * ((L + 16383) / 16384) >= (1ull << 32)) {
        set_last_error("mertens_scan_extremes: interval too long");
        return MERTENS_ENOTSUP;
    }
    PrimeTable pt;
    int rc = MERTENS_OK;
    int prc = prime_table_create(&pt, al, y_last, s);
    if (prc == 0)
        prc = sieve_scratch_create(&pt, L, s);
    if (prc != 0)
        rc = prc == 6 ? MERTENS_ENOTSUP : (prc == 2 ? MERTENS_ENOMEM : MERTENS_ECUDA);
    int16_t *ml = (int16_t *)dev_alloc(al, (L + 2) * 2);
    int32_t *ss = (int32_t *)dev_alloc(al, nseg * 4);
    int64_t *so = (int64_t *)dev_alloc(al, nseg * 8);
    int64_t *cy = (int64_t *)dev_alloc(al, (nblocks + 1) * 8);
    Ext *part = (Ext *)dev_alloc(al, nparts * sizeof(Ext));
    Ext *first = (Ext *)dev_alloc(al, ctas * sizeof(Ext));  // records of a first pass
    if (rc == MERTENS_OK && (!ml || !ss || !so || !cy || !part || !first))
        rc = MERTENS_ENOMEM;
    if (rc == MERTENS_OK) {
        cudaMemcpyAsync(cy, &carry, 8, cudaMemcpyHostToDevice, s);
        for (uint64_t b = 0; b < nblocks && rc == MERTENS_OK; ++b) {
            SieveLaunch Lc;
            Lc.y1 = y_first + b * L;
            Lc.len = std::min(L, y_last - Lc.y1 + 1);
            Lc.Mloc = ml;
            Lc.segsum = ss;
            Lc.segoff = so;
            Lc.carry_in = cy + b;
            Lc.carry_out = cy + b + 1;
            if (sieve_block_enqueue(&pt, Lc, s) < 0)
                rc = MERTENS_ECUDA;
            // the segment sums are no longer needed: they become the segments'
            // {max, min}
            const uint32_t ns = (uint32_t)sieve_segments(Lc.len);
            const uint32_t nc = (ns + kExtWarps * kExtSegs - 1) / (kExtWarps * kExtSegs);
            uint32_t *mm = reinterpret_cast<uint32_t *>(ss);
            segment_extremes_kernel<<<nc, kExtThreads, 0, s>>>(Lc.y1, Lc.len, ns, ml, so, mm, first);
            merge_extremes(first, nc, s);
            exact_extremes_kernel<<<kExtScan, kExtThreads, 0, s>>>(Lc.y1, Lc.len, ns, ml, so, mm,
                                                                  first, part + b * kExtScan);
            if (cudaGetLastError() != cudaSuccess)
                rc = MERTENS_ECUDA;
        }
        if (rc == MERTENS_OK)
            merge_extremes(part, (uint32_t)nparts, s);
        Ext e;
        int64_t last = 0;
        if (rc == MERTENS_OK &&
            (cudaMemcpyAsync(&e, part, sizeof(Ext), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
             cudaMemcpyAsync(&last, cy + nblocks, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
             cudaStreamSynchronize(s) != cudaSuccess))
            rc = MERTENS_ECUDA;
        if (rc == MERTENS_OK) {
            const uint32_t st = sieve_scratch_status(&pt);
            if (st) {
                set_last_error("mertens_scan_extremes: %s", sieve_status_text(st));
                rc = sieve_status_code(st);
            }
        }
        if (rc == MERTENS_OK) {
            out->M_last = last;
            out->M_max = e.mx;
            out->y_M_max = e.ymx;
            out->M_min = e.mn;
            out->y_M_min = e.ymn;
            out->R_max_M = e.rpM;
            out->y_R_max = e.rpy;
            out->R_min_M = e.rnM;
            out->y_R_min = e.rny;
            out->R_max = (double)e.rpM / std::sqrt((double)e.rpy);
            out->R_min = (double)e.rnM / std::sqrt((double)e.rny);
        }
    }
    if (rc == MERTENS_ECUDA)
        set_last_error("mertens_scan_extremes: %s", cudaGetErrorString(cudaGetLastError()));
    dev_free(al, ml, (L + 2) * 2);
    dev_free(al, ss, nseg * 4);
    dev_free(al, so, nseg * 8);
    dev_free(al, cy, (nblocks + 1) * 8);
    dev_free(al, part, nparts * sizeof(Ext));
    dev_free(al, first, ctas * sizeof(Ext));
    if (pt.np)
        prime_table_destroy(&pt);
    return rc;
}

}  // extern "C"
