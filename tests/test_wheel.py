"""The sums over integers coprime to 6 (csrc/wheel.h): CPU models of the
identities and of the remainder rule the kernels use, and, on the GPU, whole
runs of that form against runs of the full sums (MERTENS_SHARE=0)."""
import math
import random

import numpy as np
import pytest

import oracle
import paper_1108_0135_gb300 as pm


def phi6(v):
    i, r = divmod(v, 6)
    return 2 * i + (r >= 1) + (r >= 5)


def test_identities_over_integers_coprime_to_6():
    """Sum over j coprime to 6 of M6(floor(v/j)) = 1, and M from M6."""
    top = 3000
    M = oracle.mertens_table(top)
    mu = np.diff(M, prepend=0)
    M6 = np.cumsum([int(mu[m]) if m % 2 and m % 3 else 0 for m in range(top + 1)])
    for v in list(range(1, 200)) + [997, 1000, 2310, 3000]:
        assert sum(M6[v // j] for j in range(1, v + 1) if math.gcd(j, 6) == 1) == 1
        assert M[v] == M6[v] - M6[v // 2] - M6[v // 3] + M6[v // 6]


def test_phi6_from_the_floor_of_an_estimate():
    """phi6(floor(k/y)) = T + [k >= y Y(T)], Y(T) = (3T + 1) | 1, for the floor T
    of any estimate of k/(3y) that errs by less than 1/3."""
    rng = random.Random(6)
    for _ in range(20000):
        y = rng.choice([1, 5, 7, rng.randrange(1, 50), rng.randrange(1, 10**8)])
        k = rng.choice([rng.randrange(1, 200) * y + rng.randrange(-1, 2),
                        rng.randrange(1, 10**15)])
        if k < 1:
            continue
        # floors of k/(3y) - 1/3 < v < k/(3y) + 1/3
        for T in {(k - y) // (3 * y), k // (3 * y), -(-(k + y) // (3 * y)) - 1}:
            if T >= 0:
                assert T + (k >= y * ((3 * T + 1) | 1)) == phi6(k // y), (k, y, T)


def test_float_estimate_of_the_dense_terms():
    """The float modes' estimate, k (1/3y) with every operation in single
    precision (the sum with 1.5 2^23 is exact before it is rounded down), errs by
    less than 1/3 up to the bounds the kernels use."""
    rng = random.Random(7)
    f = np.float32
    for bound, ylo, yhi in ((2_600_000 / 1.05, 5, 5_590_000), (1_800_000, 5_590_000, 350_000_000)):
        for _ in range(20000):
            y = rng.randrange(ylo, yhi)
            k = rng.randrange(1, int(3 * y * bound) + 1)
            kf, rf = float(f(k)), float(f(1.0) / f(3 * y))
            assert abs(kf * rf - k / (3 * y)) < 1 / 3


def test_index_forms():
    """The 32-bit forms of phi6 and of the index of the last wheel number."""
    for v in list(range(0, 200)) + [2**31 - 1, 2**31, 2**32 - 6]:
        assert ((v + 5) & ~1) // 3 - 1 == phi6(v)
        if v:
            assert ((v - 1) & ~1) // 3 == phi6(v) - 1
    for w in range(100):
        y = 3 * w + 1 + (w & 1)
        assert math.gcd(y, 6) == 1 and phi6(y) == w + 1


def _arrays(ns, u, bl):
    plan = pm.mertens_plan(ns, u, bl)
    try:
        pm.mertens_run(plan)
        return [pm.mertens_result(plan, i, entries=True)[1] for i in range(len(ns))]
    finally:
        pm.mertens_destroy(plan)


@pytest.mark.gpu
@pytest.mark.parametrize("ns,u,bl", [
    ([7 * 10**9 + 1], 3 * 10**5, 0),             # u near sqrt(n): bounds of floor(X/x) in low tiles
    ([10**13 + 7], 0, 6144 * 1000),              # every dense mode; blocks of whole segments
    ([10**13 + 7], 5 * 10**8 + 3, 10**7 + 1),    # ragged blocks, tiles cut at block ends
    ([3 * 10**14 + 11], 0, 0),                   # blocks above the tile range
    ([10**12, 10**12 + 10**6, 5 * 10**9 + 9, 12345, 6, 1], 0, 0),  # several targets
])
@pytest.mark.parametrize("quot", [None, "2"])
def test_wheel_runs_equal_full_sums(ns, u, bl, quot, monkeypatch):
    monkeypatch.setenv("MERTENS_SHARE", "0")
    full = _arrays(ns, u, bl)
    monkeypatch.delenv("MERTENS_SHARE")
    if quot:
        monkeypatch.setenv("MERTENS_GATHER_QUOT", quot)  # 64-bit remainders
    for a, b in zip(full, _arrays(ns, u, bl)):
        assert np.array_equal(a, b)


def test_linear_estimate_of_the_dense_terms():
    """The linear mode's estimate of k/(3y) - q0 in single precision (float_u64 of
    q0, one multiply-add, the reciprocal) errs by less than 1/3 for k <= 900 y0^2."""
    rng = random.Random(8)
    f = np.float32
    for _ in range(20000):
        y0 = 6144 * rng.randrange(1, 56_000)
        k = min(rng.randrange(900 * y0 * y0 // 8, 900 * y0 * y0 + 1), 2**63 - 1)
        ym = y0 + 3072
        y = y0 + rng.randrange(1, 6144)
        q0, r0 = divmod(k, 3 * ym)
        qf = f(float(f(q0 >> 32)) * 2.0**32 + float(f(q0 & 0xffffffff)))
        R = f(float(f(-3.0) * qf) * float(y - ym) + float(f(r0)))
        est = float(R) * float(f(1.0) / f(3 * y))
        exact = (k - 3 * y * q0) / (3 * y)
        assert abs(est - exact) < 1 / 3 and abs(exact) < 1.0e6


@pytest.mark.gpu
@pytest.mark.parametrize("env", [None, "MERTENS_SIEVE_BUCKETS"])
@pytest.mark.parametrize("y1,ln", [(1, 40_003), (10**9 + 4, 131_073), (10**9 + 5, 98_305),
                                   (10**12 + 2, 400_001), (10**12 + 3, 262_147)])
def test_bucketed_sieve_leaves_out_the_multiples_of_4(env, y1, ln, monkeypatch):
    """mu from every start mod 4 (the bucketed kernel's primes give the multiples of
    4 no weight), over several tiles and with primes below, in and above a tile."""
    import torch

    if env:
        monkeypatch.setenv(env, "1")
    out = torch.empty(ln, dtype=torch.int8, device="cuda")
    pm.mertens_sieve_mu(y1, ln, out)
    assert np.array_equal(out.cpu().numpy(), oracle.mu_window(y1, ln))


@pytest.mark.gpu
@pytest.mark.parametrize("n,u,y1,ny", [(10**14 + 7, 3 * 10**9, 10**8 + 3, 5 * 10**6 + 11),
                                       (10**20, 21544346900318, 10**12 + 2, 3 * 10**7 + 1)])
def test_window_does_not_depend_on_the_block_length(n, u, y1, ny):
    """A window in one block and in blocks of four times block_len, the last one
    ragged: the same sums, carry coefficients and mu sum."""
    got = []
    for bl in (ny, ny // 5, ny // 13 + 1):
        plan = pm.mertens_plan_window([n], y1, y1 + ny - 1, u, bl)
        pm.mertens_run(plan)
        got.append(pm.mertens_window_result(plan, 0))
        pm.mertens_destroy(plan)
    for S, coef, mu in got[1:]:
        assert mu == got[0][2]
        assert np.array_equal(S, got[0][0]) and np.array_equal(coef, got[0][1])


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3 * 10**12 + 1, 10**13 + 37, 4 * 10**13 + 5])
def test_long_lanes_equal_the_full_sums(n, monkeypatch):
    """Targets whose sets of 32 entries have thousands of terms per entry in a tile
    (all warps share them) give the same array as the full sums."""
    got = []
    for share in (None, "0"):
        if share:
            monkeypatch.setenv("MERTENS_SHARE", share)
        plan = pm.mertens_plan([n])
        pm.mertens_run(plan)
        got.append(pm.mertens_result(plan, 0, entries=True)[1])
        pm.mertens_destroy(plan)
    assert np.array_equal(got[0], got[1])


@pytest.mark.gpu
def test_window_without_the_memory_for_long_blocks():
    """A window plan whose blocks of four times block_len do not get their memory is
    made with block_len, with the same results."""
    import torch

    n, u, y1, bl = 10**14 + 7, 3 * 10**9, 10**9 + 3, 1 << 22
    sizes, limit, refused = [], [1 << 62], []

    def alloc(nbytes, stream, ctx):
        if nbytes > limit[0]:
            refused.append(nbytes)
            return 0
        sizes.append(nbytes)
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream or 0))

    def release(ptr, nbytes, stream, ctx):
        torch.cuda.caching_allocator_delete(ptr)

    got = []
    pm.mertens_set_allocator(alloc, release)
    try:
        for _ in range(2):
            plan = pm.mertens_plan_window([n], y1, y1 + 9 * bl + 4, u, bl)
            pm.mertens_run(plan)
            got.append(pm.mertens_window_result(plan, 0))
            pm.mertens_destroy(plan)
            limit[0] = 2 * 4 * bl - 1  # the int16 M of a long block is larger
    finally:
        pm.mertens_set_allocator()
    assert max(sizes) > limit[0] and refused
    assert got[0][2] == got[1][2]
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
