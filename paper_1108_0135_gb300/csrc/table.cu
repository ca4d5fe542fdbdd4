// Resident M(y) table: the sieve (steps a1 + a2, in the form of wheel.h) run
// once up to y_max and kept in device memory (0.17 bytes per y), together with
// the part of the update that does not depend on the target (the dense list of
// squarefree numbers).  Plans made on a table (mertens_plan_on_table) read M6(y)
// from it and run only the update and resolve.  The paper sieves per target
// (Sec. 3); keeping the sieve's output resident lets many queries share it.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/libmertens.h"
#include "common.cuh"
#include "internal.h"
#include "update.h"
#include "wheel.h"

namespace mert {
double plan_dense_factor();
}  // namespace mert

using namespace mert;

namespace {

typedef unsigned __int128 u128;

uint64_t isqrt_u128(u128 v)
{
    u128 r = (u128)std::sqrt((double)v);
    if (r > 0)
        r = (r + v / r) / 2;
    while (r * r > v)
        --r;
    while ((r + 1) * (r + 1) <= v)
        ++r;
    return (uint64_t)r;
}

template <typename T>
T *table_alloc(mertens_table_s *t, size_t count)
{
    const size_t bytes = count * sizeof(T);
    void *p = dev_alloc(t->al, bytes);
    if (p) {
        t->allocs.push_back({p, bytes});
        t->bytes += bytes;
    }
    return (T *)p;
}

}  // namespace

extern "C" {

int mertens_table_create(mertens_table_t *out, uint64_t y_max, mertens_u128 n_max, void *stream)
{
    if (!out)
        return MERTENS_EINVAL;
    *out = nullptr;
    if (y_max == 0 || y_max >= (1ull << 40) || (n_max.lo == 0 && n_max.hi == 0) ||
        n_max.hi >= (1ull << 63)) {
        set_last_error("mertens_table_create: need 1 <= y_max < 2^40 and 1 <= n_max < 2^127");
        return MERTENS_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    mertens_table_s *t = new (std::nothrow) mertens_table_s();
    if (!t)
        return MERTENS_ENOMEM;
    t->al = current_allocator();
    cudaGetDevice(&t->device);
    t->y_max = y_max;
    t->n_max_lo = n_max.lo;
    t->n_max_hi = n_max.hi;
    const u128 nm = ((u128)n_max.hi << 64) | n_max.lo;
    const uint64_t r = isqrt_u128(nm);
    // the planner's dense cut-offs stay below the chunk-aligned dc sqrt(n)
    // (or sqrt(n) itself)
    const double dc = plan_dense_factor();
    uint64_t yd = (uint64_t)(std::max(dc, 1.0) * std::sqrt((double)nm)) + 2 * kChunk;
    yd = ((yd + kChunk - 1) / kChunk) * kChunk - 1;
    t->ydense = std::min(yd, y_max);
    // M6 of the integers coprime to 6 up to whole segments of 6144 y, and the
    // dense list of the first nchunks of them
    t->y_cov = (y_max + kWheelSegY - 1) / kWheelSegY * kWheelSegY;
    const uint64_t nseg = t->y_cov / kWheelSegY;
    const uint64_t nchunks = (t->ydense + kWheelSegY - 1) / kWheelSegY;
    t->Mg = table_alloc<uint2>(t, nseg * kSegY >> kMgShift);
    t->segoff = table_alloc<int64_t>(t, nseg);
    t->dl = table_alloc<uint16_t>(t, nchunks * kSegY);
    t->dl_cnt = table_alloc<uint32_t>(t, nchunks);
    // scratch of the build: sieve tables, segment sums, carries, status word
    const uint64_t L = std::min<uint64_t>((1ull << 30) / kWheelSegY * kWheelSegY, t->y_cov);
    const uint64_t nblocks = (t->y_cov + L - 1) / L;
    WheelSieve ws;
    wheel_sieve_primes(&ws, y_max);
    const auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t b_ws = up(wheel_sieve_bytes(&ws, L / 3)), b_sum = up(L / kWheelSegY * 4),
                 b_cy = up((nblocks + 1) * 8), bytes = b_ws + b_sum + b_cy + 256;
    char *buf = (char *)dev_alloc(t->al, bytes);
    int rc = t->Mg && t->segoff && t->dl && t->dl_cnt && buf ? MERTENS_OK : MERTENS_ENOMEM;
    if (rc == MERTENS_OK) {
        int32_t *segsum = (int32_t *)(buf + b_ws);
        int64_t *carry = (int64_t *)(buf + b_ws + b_sum);
        uint32_t *err = (uint32_t *)(buf + b_ws + b_sum + b_cy);
        cudaMemsetAsync(carry, 0, 8, s);
        cudaMemsetAsync(err, 0, 4, s);
        if (wheel_sieve_bind(&ws, buf, L / 3, err, s) != 0)
            rc = MERTENS_ECUDA;
        cudaMemcpyAsync(ws.p, ws.host_p.data(), ws.host_p.size() * 4, cudaMemcpyHostToDevice, s);
        for (uint64_t b = 0; b < nblocks && rc == MERTENS_OK; ++b) {
            const uint64_t y0 = b * L;
            WheelLaunch Lc;
            Lc.w0 = y0 / 3;
            Lc.len = std::min(L, t->y_cov - y0) / 3;
            Lc.Mg = t->Mg + (y0 / 3 >> kMgShift);
            Lc.segsum = segsum;
            Lc.segoff = t->segoff + y0 / kWheelSegY;
            Lc.carry_in = carry + b;
            Lc.carry_out = carry + b + 1;
            if (wheel_sieve_enqueue(&ws, Lc, s) < 0)
                rc = MERTENS_ECUDA;
        }
        if (rc == MERTENS_OK &&
            wheel_dense_list_enqueue(t->Mg, 0, nchunks, t->dl, t->dl_cnt, s) < 0)
            rc = MERTENS_ECUDA;
        uint32_t st = 0;
        if (cudaMemcpyAsync(&st, err, 4, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            rc = MERTENS_ECUDA;
        if (rc == MERTENS_OK && st) {
            set_last_error("mertens_table_create: %s", sieve_status_text(st));
            rc = sieve_status_code(st);
        }
    }
    if (rc == MERTENS_ECUDA)
        set_last_error("mertens_table_create: %s", cudaGetErrorString(cudaGetLastError()));
    else if (rc == MERTENS_ENOMEM)
        set_last_error("mertens_table_create: device allocation failed");
    dev_free(t->al, buf, bytes);
    if (rc != MERTENS_OK) {
        mertens_table_destroy(t);
        return rc;
    }
    *out = t;
    return MERTENS_OK;
}

int mertens_table_info(mertens_table_t t, uint64_t *y_max, mertens_u128 *n_max, size_t *bytes)
{
    if (!t)
        return MERTENS_EINVAL;
    if (y_max)
        *y_max = t->y_max;
    if (n_max) {
        n_max->lo = t->n_max_lo;
        n_max->hi = t->n_max_hi;
    }
    if (bytes)
        *bytes = t->bytes;
    return MERTENS_OK;
}

void mertens_table_destroy(mertens_table_t t)
{
    if (!t)
        return;
    cudaDeviceSynchronize();
    for (auto &a : t->allocs)
        dev_free(t->al, a.first, a.second);
    delete t;
}

}  // extern "C"
