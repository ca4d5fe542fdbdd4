"""Places and dense cut-offs of plans over the integers coprime to 6: the rules of
csrc/wheel_place.h, run by a host program over batches of unlike targets, and on the
GPU such batches against their targets planned alone."""
import ctypes
import math
import os
import random
import subprocess
import threading

import numpy as np
import pytest

import paper_1108_0135_gb300 as pm

CSRC = os.path.join(os.path.dirname(os.path.abspath(pm.__file__)), "csrc")


def compiled(d, name, text):
    src, exe = d / (name + ".cpp"), d / name
    src.write_text(text)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


# reads: dc wide_from count by_k, then n u per target (n as high and low word);
# prints per batch: classes, places, largest j, largest yc, gathered j, bad entries
PROGRAM = r"""
#include <cstdio>
#include "wheel_place.h"
using namespace mert;
typedef unsigned __int128 u128;
int main()
{
    double dc;
    unsigned long long wide, hi, lo, u;
    int count, by_k;
    while (scanf("%lf %llu %d %d", &dc, &wide, &count, &by_k) == 4) {
        std::vector<WheelTarget> t(count);
        for (auto &v : t) {
            if (scanf("%llu %llu %llu", &hi, &lo, &u) != 3)
                return 1;
            v.n = ((u128)hi << 64) | lo;
            v.u = u;
            v.X = (uint64_t)(v.n / u);
            v.lookup = false;
        }
        uint64_t end = 0;
        const std::vector<WheelClass> cls = wheel_classes(t, dc, wide, &end);
        struct E { uint64_t k, jlo; };
        std::vector<E> place(end, E{0, 0});
        uint64_t bad = 0;
        for (size_t c = 0; c < cls.size(); ++c) {
            std::vector<E> e;
            for (auto &v : t)
                for (uint64_t x = 1; v.cls == c && x <= v.X; ++x) {
                    const u128 k = v.n / x;
                    e.push_back({k < wide ? (uint64_t)k : 0, v.X / x + 1});
                }
            if (by_k)
                std::stable_sort(e.begin(), e.end(),
                                 [](const E &a, const E &b) { return a.k > b.k; });
            bad += e.size() != cls[c].entries || cls[c].first % kWheelGroup != 0;
            for (size_t i = 0; i < e.size(); ++i) {
                bad += place[cls[c].first + i].jlo != 0;  // places do not overlap
                place[cls[c].first + i] = e[i];
            }
        }
        uint64_t jmax = 0, ymax = 0;
        double gathered = 0;
        for (uint64_t g = 0; g < end; g += kWheelGroup) {
            uint64_t kf = 0, cap = UINT64_MAX;
            double sum = 0;
            int one = 0;
            const uint64_t to = std::min(end, g + kWheelGroup);
            for (uint64_t i = g; i < to; ++i)
                if (place[i].k) {
                    kf = std::max(kf, place[i].k);
                    cap = std::min(cap, place[i].k / place[i].jlo);
                    sum += (double)place[i].k;
                    ++one;
                }
            const uint64_t yc = kf ? wheel_cutoff(dc, sum / one, kf, cap, UINT64_MAX) : 0;
            bad += kf && yc > wheel_cutoff_bound(dc, kf);
            ymax = std::max(ymax, yc);
            for (uint64_t i = g; i < to; ++i)
                if (place[i].k) {
                    const uint64_t j = wheel_last_j(place[i].k, yc, place[i].jlo);
                    jmax = std::max(jmax, j);
                    gathered += (double)(j - (place[i].jlo - 1));
                    bad += yc > place[i].k / place[i].jlo;
                }
        }
        printf("%zu %llu %llu %llu %.0f %llu\n", cls.size(), (unsigned long long)end,
               (unsigned long long)jmax, (unsigned long long)ymax, gathered,
               (unsigned long long)bad);
    }
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    exe = compiled(tmp_path_factory.mktemp("places"), "places", PROGRAM)

    def run(batches, dc=1.4, wide=1 << 63, by_k=1):
        text = ""
        for targets in batches:
            text += f"{dc} {wide} {len(targets)} {by_k}\n"
            for n, u in targets:
                text += f"{n >> 64} {n & (2**64 - 1)} {u}\n"
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True)
        names = ("classes", "places", "jmax", "ymax", "gathered", "bad")
        return [dict(zip(names, map(int, line.split()))) for line in out.stdout.splitlines()]

    return run


def auto_u(ns):
    """The documented automatic limits of a batch."""
    g = min(1.78, max(1.0, (max(ns) / 1e18) ** -0.25))
    ub = 0.45 * g * float(sum(ns)) ** (2 / 3)
    return [(n, min(n, max(int(ub), math.isqrt(n) + 1)) if n > 3 else n) for n in ns]


BATCHES = [
    [10**15, 1], [10**17, 5], [10**17, 50], [10**14, 10], [10**14, 100],
    [10**i for i in range(17)],                       # the paper's table in one call
    [1000, 10**19], [7, 10**19, 12, 3 * 10**18],      # two-word entries
    [10**14 + i * 10**9 for i in range(64)],
    [10**12, 10**12 + 10**6, 5 * 10**9 + 9, 12345, 6, 1],
    [1], [2, 1], [3, 3, 3, 1, 1],
]


@pytest.mark.parametrize("by_k", [1, 0])
def test_groups_of_unlike_targets(rules, by_k):
    """No j reaches 2^32, no cut-off is above an entry's floor(k/jlo), and a batch
    gathers at most twice what its targets gather one by one at the same limits (a
    group of a batch takes the mean of its own k)."""
    rng = random.Random(3)
    batches = list(BATCHES)
    for _ in range(40):
        top = rng.uniform(2, 17)
        batches.append([int(10 ** rng.uniform(0, top)) for _ in range(rng.randrange(2, 12))])
    batches = [auto_u(ns) for ns in batches]
    got = rules(batches, by_k=by_k)
    for targets, r in zip(batches, got):
        assert r["bad"] == 0 and r["jmax"] < 2**32 - 6, (targets, r)
        alone = sum(v["gathered"] for v in rules([[t] for t in targets]))
        assert r["gathered"] <= 2 * alone + 64 * 6, (targets, r, alone)
        assert r["places"] < sum(n // u for n, u in targets) + 64 * r["classes"]


def test_like_targets_share_a_class(rules):
    """Close targets, and requests over the serving range, stay one class."""
    rng = random.Random(4)
    batches = [[10**14 + i * 10**9 for i in range(64)],
               [int(10 ** rng.uniform(10, 15)) for _ in range(32)]]
    for r in rules([auto_u(ns) for ns in batches]):
        assert r["classes"] == 1


def test_many_small_targets(rules):
    """A hundred thousand tiny targets make a few classes, not one each."""
    rng = random.Random(6)
    for ns in ([3] * 100_000 + [1], [rng.randrange(1, 30) for _ in range(100_000)],
               [int(10 ** rng.uniform(0, 9)) for _ in range(100_000)]):
        r, = rules([auto_u(ns)])
        assert r["bad"] == 0 and r["classes"] <= 6


@pytest.mark.parametrize("dc", [0.7, 1.4, 7.5, 900.0])
def test_limits_near_the_square_root(rules, dc):
    """Explicit limits: every cut-off is bound by floor(k/jlo); the classes stay few."""
    rng = random.Random(5)
    batches = []
    for _ in range(30):
        u = int(10 ** rng.uniform(1, 5))
        ns = [int(10 ** rng.uniform(math.log10(u), 2 * math.log10(u))) for _ in range(6)]
        batches.append([(n, u) for n in ns if math.isqrt(n) < u <= n] or [(u, u)])
        batches.append([(n, min(n, math.isqrt(n) + 1)) for n in ns])
    for targets, r in zip(batches, rules(batches, dc=dc)):
        assert r["bad"] == 0 and r["jmax"] < 2**32 - 6 and r["classes"] <= 8, (targets, r)


# reads: dc, largest k, then 64 k of a group; prints the cut-off, its bound, the
# largest j (all without floor(k/jlo) and the list's end)
CUTOFF = r"""
#include <cstdio>
#include "wheel_place.h"
using namespace mert;
int main()
{
    double dc;
    unsigned long long kf, k[64];
    while (scanf("%lf %llu", &dc, &kf) == 2) {
        double sum = 0;
        for (auto &v : k) {
            if (scanf("%llu", &v) != 1)
                return 1;
            sum += (double)v;
        }
        const uint64_t yc = wheel_cutoff(dc, sum / 64, kf, UINT64_MAX, UINT64_MAX);
        uint64_t j = 0;
        for (auto v : k)
            j = std::max(j, wheel_last_j(v, yc, 1));
        printf("%llu %llu %llu\n", (unsigned long long)yc,
               (unsigned long long)wheel_cutoff_bound(dc, kf), (unsigned long long)j);
    }
}
"""


def test_dense_list_reaches_every_cutoff(tmp_path):
    """The bound that sizes the dense list is at least the cut-off of every group, for
    factors over the accepted range, k up to 2^63 and groups of close or equal k (where
    the rounding of the mean counts), and j stays in range."""
    rng = random.Random(9)
    text, n = "", 0
    for _ in range(4000):
        dc = 10 ** rng.uniform(-7, 2.999)
        kf = min(2**63 - 1, int(10 ** rng.uniform(0, 18.97)))
        if rng.random() < 0.3:  # dc sqrt(k) just below a multiple of 4096
            v = 4096 * rng.randrange(1, 10**6)
            kf = max(1, min(2**63 - 1, int((v / dc) ** 2) - rng.randrange(3)))
        spread = rng.choice([0, 0, 1e-15, 1e-9, 1e-3, 1])
        ks = [kf - int(kf * spread * rng.random()) for _ in range(63)] + [kf]
        text += f"{dc!r} {kf} " + " ".join(str(max(1, k)) for k in ks) + "\n"
        n += 1
    out = subprocess.run([compiled(tmp_path, "cutoff", CUTOFF)], input=text,
                         capture_output=True, text=True, check=True).stdout.split("\n")
    assert len(out) == n + 1
    for line, given in zip(out, text.split("\n")):
        if line:
            yc, bound, j = map(int, line.split())
            assert yc <= bound and j < 2**32 - 6, (given[:60], yc, bound, j)


@pytest.mark.gpu
def test_small_dense_factor_does_not_change_results(monkeypatch):
    """A factor far below 1 (the accepted range starts above 0): the same array as the
    full sums."""
    n, u = 10**12 + 39, 10**11
    tuning = pm.mertens_get_tuning()
    try:
        pm.mertens_set_tuning(dense_c=2e-4)
        got = _array(n, u)
    finally:
        pm.mertens_set_tuning(**tuning)
    monkeypatch.setenv("MERTENS_SHARE", "0")
    assert np.array_equal(got, _array(n, u))


def _array(n, u):
    plan = pm.mertens_plan([n], u)
    try:
        pm.mertens_run(plan)
        return pm.mertens_result(plan, 0, entries=True)[1]
    finally:
        pm.mertens_destroy(plan)


@pytest.mark.gpu
@pytest.mark.parametrize("ns,wide_from", [
    ([10**15, 1], None),
    ([10**i for i in range(17)], None),
    ([50, 10**15, 10**14 + 3, 2, 10**15 + 1, 777], None),
    ([1000, 10**14, 3], 10**13),          # target by target: two-word entries
    ([5, 10**15 + 7, 10**6], 10**14),
])
def test_unlike_targets_equal_the_same_planned_alone(ns, wide_from, monkeypatch):
    if wide_from:
        monkeypatch.setenv("MERTENS_WIDE_FROM", str(wide_from))
    plan = pm.mertens_plan(ns)
    try:
        pm.mertens_run(plan)
        got = [(pm.mertens_plan_info(plan, i)["u"], pm.mertens_result(plan, i, entries=True)[1])
               for i in range(len(ns))]
    finally:
        pm.mertens_destroy(plan)
    monkeypatch.delenv("MERTENS_WIDE_FROM", raising=False)
    for n, (u, arr) in zip(ns, got):
        assert np.array_equal(arr, _array(n, u)), n


@pytest.mark.gpu
def test_unlike_targets_on_a_table():
    """Lookups, tiny targets with terms and large ones in one plan on a table."""
    table = pm.mertens_table_create(1 << 26, 10**15)
    ns = [10**i for i in range(15)] + [(1 << 26) + 1, 3]
    try:
        plan = pm.mertens_plan_on_table(table, ns)
        pm.mertens_run(plan)
        got = [(pm.mertens_plan_info(plan, i)["u"], pm.mertens_result(plan, i, entries=True)[1])
               for i in range(len(ns))]
        pm.mertens_destroy(plan)
    finally:
        pm.mertens_table_destroy(table)
    for n, (u, arr) in zip(ns, got):
        assert np.array_equal(arr, _array(n, u)), n


@pytest.mark.gpu
@pytest.mark.parametrize("ns", [[7 * 10**11 + 3], [7 * 10**11 + 3, 7 * 10**11 + 10**6, 10**6]])
def test_table_whose_list_ends_below_the_factor_times_sqrt_n(ns):
    """1.4 sqrt(n) lies above the table, floor(k/jlo) of every entry below its end."""
    table = pm.mertens_table_create(1 << 20, 10**12)
    try:
        plan = pm.mertens_plan_on_table(table, ns, 10**6)
        pm.mertens_run(plan)
        got = [pm.mertens_result(plan, i, entries=True)[1] for i in range(len(ns))]
        pm.mertens_destroy(plan)
    finally:
        pm.mertens_table_destroy(table)
    for n, arr in zip(ns, got):
        assert np.array_equal(arr, _array(n, 10**6)), n


@pytest.mark.gpu
def test_plan_info_needs_no_device():
    """Term counts of a plan from many threads at once, and inside a stream capture
    (which a copy on the default stream would break)."""
    ns = [10**12 + i for i in range(5)] + [7]
    plan = pm.mertens_plan(ns)
    try:
        # a capture of a stream that waits for the default stream: a copy on that would
        # break it
        with open("/proc/self/maps") as f:
            rt = ctypes.CDLL(next(line.split()[-1] for line in f if "libcudart" in line))
        side, graph = ctypes.c_void_p(), ctypes.c_void_p()
        assert rt.cudaStreamCreate(ctypes.byref(side)) == 0
        assert rt.cudaStreamBeginCapture(side, 0) == 0
        try:
            inside = [pm.mertens_plan_info(plan, i) for i in range(len(ns))]
        finally:
            ended = rt.cudaStreamEndCapture(side, ctypes.byref(graph))
            rt.cudaStreamDestroy(side)
        assert ended == 0
        rt.cudaGraphDestroy(graph)
        got = [None] * 16
        start = threading.Barrier(16)

        def read(t):
            start.wait()
            got[t] = [pm.mertens_plan_info(plan, i) for i in range(len(ns))]

        threads = [threading.Thread(target=read, args=(t,)) for t in range(16)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        want = [pm.mertens_describe(n, v["u"]) for n, v in zip(ns, inside)]
        for v in got + [inside]:
            assert [(x["direct_terms"], x["gathered_terms"]) for x in v] == \
                [(x["direct_terms"], x["gathered_terms"]) for x in want]
    finally:
        pm.mertens_destroy(plan)


def test_windows_are_planned_again_only_for_shorter_blocks():
    """A window plan that gets no memory is tried again with block_len only when its
    blocks were longer than that (each attempt asks for the same number of buffers)."""
    asked = []

    def alloc(nbytes, stream, ctx):
        asked[-1] += 1
        return 0

    pm.mertens_set_allocator(alloc, lambda *a: None)
    try:
        for span in (10**6, 10**6 + 1):
            asked.append(0)
            with pytest.raises(pm.MertensError) as e:
                pm.mertens_plan_window([10**14 + 7], 10**9, 10**9 + span - 1, 3 * 10**9, 10**6)
            assert e.value.code == pm.MERTENS_ENOMEM
    finally:
        pm.mertens_set_allocator()
    assert asked[0] > 0 and asked[1] == 2 * asked[0]


@pytest.mark.gpu
@pytest.mark.parametrize("y1,blocks", [(1, 10), (10**9 + 1, 3)])
def test_short_windows_over_the_tile_range_keep_their_blocks(y1, blocks):
    """Ten blocks from y = 1, where the tiles of all entries end inside, and above."""
    bl = 1 << 22
    plan = pm.mertens_plan_window([10**14 + 7], y1, y1 + 10 * bl - 1, 3 * 10**9, bl)
    try:
        pm.mertens_run(plan)
        assert pm.mertens_run_stats_get(plan)["blocks"] == blocks
    finally:
        pm.mertens_destroy(plan)
