"""Timed cases: the calls that users of libmertens make, over their range.

Kinds (the "kind" of a case):
  query     M(n) and its array M(floor(n/x)) in one call: plan, run, read, free
  resident  a plan that is kept and run again, its whole array read back
  batch     close targets in one plan, sharing one sieve pass
  serve     a burst of queries through the continuous-batching server
  window    one y-window of a two-word target (the unit of a sharded run)
  sieve     mu(y) or M(y) of a window into a device buffer
  scan      the extremes of M(y) and M(y)/sqrt(y) over an interval
  table     a query planned on a resident M(y) table

All outputs are whole numbers (but the two rounded ratios of a scan).
"""
import math
import random

import numpy as np
import torch

import paper_1108_0135_gb300 as pm
from paper_1108_0135_gb300 import _lib as L


def listed():
    return [
        # the bottom of the serving range: planning, allocation and launches count
        {"name": "query 1e10", "kind": "query", "n": 10**10},
        # the middle of the serving range
        {"name": "query 1e13", "kind": "query", "n": 10**13},
        # near the top of the serving range, no round size
        {"name": "query 3e15", "kind": "query", "n": 3141592653589793},
        # one isolated value near the targets of the close batch
        {"name": "query 1e17", "kind": "query", "n": 10**17},
        # the small fixed configuration: n = 10^12, u = 10^8, 2^24-y blocks
        {"name": "resident 1e12", "kind": "resident", "n": 10**12, "u": 10**8, "block_len": 1 << 24},
        # the headline configuration: n = 10^16, u = 4 10^10, 2^28-y blocks
        {"name": "resident 1e16", "kind": "resident", "n": 10**16, "u": 4 * 10**10,
         "block_len": 1 << 28},
        # 64 close targets 10^9 apart in one plan
        {"name": "batch 64 x 1e14", "kind": "batch", "n": 10**14, "count": 64, "gap": 10**9},
        # a burst of the seeded request stream (log-uniform n), closed loop
        {"name": "serve 96", "kind": "serve", "count": 96, "lo": 10.0, "hi": 15.0},
        # n = 10^20: 64 blocks of 2^28 y from y = 10^13, where large primes dominate the sieve
        {"name": "window 1e20", "kind": "window", "n": "100000000000000000000",
         "u": 21544346900318, "block_len": 1 << 28, "y_first": 10**13, "blocks": 64},
        # the step-level sieve on a short ragged window, as a caller with its own buffers uses it
        {"name": "sieve M 1e9", "kind": "sieve", "out": "M", "y1": 10**9, "len": 1_000_003},
        # an interval around a candidate extreme
        {"name": "scan 1e11", "kind": "scan", "y1": 10**11, "len": (1 << 30) + 12345},
        # a query on a table of 2^30 y that stays on the device
        {"name": "table 1e13", "kind": "table", "n": 10**13, "y_max": 1 << 30, "n_max": 10**15},
    ]


def _log(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "resident", "resident", "batch", "serve",
                       "window", "sieve", "scan", "table"])
    if kind == "query":
        return {"kind": kind, "n": _log(rng, 10**10, 10**17)}
    if kind == "resident":
        n = _log(rng, 10**11, 10**16)
        # around the usual limit ~ n^(2/3), and 4 to 160 blocks with ragged ends
        u = int(n ** (2 / 3) * rng.uniform(0.4, 1.2))
        blocks = _log(rng, 4, 160)
        return {"kind": kind, "n": n, "u": u, "block_len": u // blocks + rng.randrange(1, 99)}
    if kind == "batch":
        count = _log(rng, 2, 64)
        return {"kind": kind, "n": _log(rng, 10**12, 10**14), "count": count,
                "gap": _log(rng, 10**6, 10**9)}
    if kind == "serve":
        return {"kind": kind, "count": _log(rng, 8, 96), "lo": 10.0, "hi": rng.uniform(12.0, 15.0)}
    if kind == "window":
        return {"kind": kind, "n": "100000000000000000000", "u": 21544346900318,
                "block_len": 1 << 28, "y_first": _log(rng, 10**12, 10**13),
                "blocks": rng.randrange(4, 64)}
    if kind == "sieve":
        return {"kind": kind, "out": rng.choice(["M", "mu"]), "y1": _log(rng, 10**6, 10**13),
                "len": _log(rng, 10**5, 10**9) | 1}
    if kind == "scan":
        return {"kind": kind, "y1": _log(rng, 10**6, 10**12), "len": _log(rng, 10**6, 2 * 10**9) | 1}
    return {"kind": kind, "n": _log(rng, 10**11, 10**14), "y_max": 1 << rng.randrange(26, 32),
            "n_max": 10**15}


def _targets(case, seed):
    """The targets of a case: its n moved a little, from the seed (so little that
    the array keeps its length)."""
    rng = random.Random(seed)
    n = int(case["n"]) + rng.randrange(int(case["n"]) // 10**8 + 4096)
    if case["kind"] == "batch":
        return [n + i * case["gap"] for i in range(case["count"])]
    return [n]


class _Held:
    """A plan, server or table that a program keeps; freed with it."""

    def __init__(self, handle, free):
        self.handle, self._free = handle, free

    def __del__(self):
        self._free(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    rng = random.Random(seed)
    st = {"case": case, "kind": kind}
    if kind in ("query", "batch", "table", "resident"):
        st["n"] = _targets(case, seed)
    if kind == "resident":
        plan = pm.mertens_plan(st["n"], case["u"], case["block_len"])
        st["plan"] = _Held(plan, pm.mertens_destroy)
        st["out"] = np.empty(pm.mertens_plan_info(plan, 0)["X"], dtype=np.int64)
    elif kind == "table":
        st["table"] = _Held(L.mertens_table_create(case["y_max"], case["n_max"]),
                            L.mertens_table_destroy)
    elif kind == "serve":
        st["server"] = _Held(L.mertens_server_create(), L.mertens_server_destroy)
        g = np.random.default_rng(seed)
        st["n"] = [int(v) for v in 10.0 ** g.uniform(case["lo"], case["hi"], size=case["count"])]
    elif kind == "window":
        y = case["y_first"] + rng.randrange(10**6)
        plan = L.mertens_plan_window([int(case["n"])], y, y + case["blocks"] * case["block_len"] - 1,
                                     case["u"], case["block_len"])
        st["plan"] = _Held(plan, pm.mertens_destroy)
    elif kind == "sieve":
        st["y1"] = case["y1"] + rng.randrange(10**5)
        st["carry"] = rng.randrange(-5000, 5000)
        st["out"] = torch.empty(case["len"], device="cuda",
                                dtype=torch.int8 if case["out"] == "mu" else torch.int32)
    elif kind == "scan":
        st["y1"] = case["y1"] + rng.randrange(10**5)
        st["carry"] = rng.randrange(-5000, 5000)
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    stream = torch.cuda.current_stream()
    if kind == "query":
        return pm.mertens(st["n"][0], entries=True, stream=stream)
    if kind == "batch":
        got = pm.mertens(st["n"], entries=True, stream=stream)
        return [np.array([m for m, _ in got]), np.concatenate([a for _, a in got])]
    if kind == "resident":
        pm.mertens_run(st["plan"].handle, stream)
        return [pm.mertens_result_into(st["plan"].handle, 0, st["out"]), st["out"]]
    if kind == "serve":
        srv = st["server"].handle
        tickets = [L.mertens_server_submit(srv, n) for n in st["n"]]
        return np.array([L.mertens_server_wait(srv, t) for t in tickets], dtype=np.int64)
    if kind == "window":
        pm.mertens_run(st["plan"].handle, stream)
        S, coef, mu_sum = L.mertens_window_result(st["plan"].handle, 0)
        return [S.view(np.int64), coef.view(np.int64), mu_sum]
    if kind == "sieve":
        if case["out"] == "mu":
            pm.mertens_sieve_mu(st["y1"], case["len"], st["out"], stream)
        else:
            pm.mertens_sieve_M(st["y1"], case["len"], st["carry"], st["out"], stream)
        return st["out"]
    if kind == "scan":
        return L.mertens_scan_extremes(st["y1"], st["y1"] + case["len"] - 1, st["carry"], stream)
    plan = L.mertens_plan_on_table(st["table"].handle, st["n"])
    try:
        pm.mertens_run(plan, stream)
        return list(pm.mertens_result(plan, 0, entries=True))
    finally:
        pm.mertens_destroy(plan)


def _limit(ns):
    """The documented automatic sieve limit of targets ns."""
    g = min(1.78, max(1.0, (max(ns) / 1e18) ** -0.25))
    return 0.45 * g * float(sum(ns)) ** (2 / 3)


def _terms(n, u):
    # direct and gathered terms: about 2 sqrt(n/x) for each entry x <= n/u
    return 4.0 * math.sqrt(float(n) * max(1.0, n / u))


def work(case):
    """Bytes: the results that the caller gets (the inputs are a few integers).
    flops: one operation per update term of the method and one per y sieved."""
    kind = case["kind"]
    if kind in ("sieve", "scan"):
        size = {"M": 4, "mu": 1}.get(case.get("out"), 0)
        return {"bytes": size * case["len"], "flops": 1.0 * case["len"]}
    if kind == "window":
        y, n = case["blocks"] * case["block_len"], int(case["n"])
        return {"bytes": 16.0 * (n // case["u"]), "flops": float(y)}
    if kind == "serve":
        e = (case["hi"] - case["lo"]) / case["count"]
        ns = [10.0 ** (case["lo"] + (i + 0.5) * e) for i in range(case["count"])]
        u = _limit(ns)
        return {"bytes": 8.0 * len(ns), "flops": u + sum(_terms(n, min(n, u)) for n in ns)}
    count = case.get("count", 1)
    ns = [case["n"]] * count
    u = case.get("u") or min(_limit(ns), case["n"])
    if kind == "table":
        u = max(u, case["y_max"])
        return {"bytes": 8.0 * (case["n"] // u), "flops": _terms(case["n"], u)}
    return {"bytes": 8.0 * count * (case["n"] // u), "flops": u + count * _terms(case["n"], u)}


def _mu_window(y1, length):
    """mu(y1 .. y1 + length - 1) by trial division over a window, in numpy."""
    y = np.arange(y1, y1 + length, dtype=np.int64)
    left, mu = y.copy(), np.ones(length, dtype=np.int8)
    top = math.isqrt(y1 + length - 1)
    comp = np.zeros(top + 1, dtype=bool)
    for p in range(2, top + 1):
        if comp[p]:
            continue
        comp[p * p::p] = True
        a = -y1 % p
        left[a::p] //= p
        mu[a::p] *= -1
        mu[-y1 % (p * p)::p * p] = 0
    mu[left > 1] *= -1
    return mu


def exact(case, seed):
    if case["kind"] == "sieve" and case["len"] <= 2 * 10**6 and case["y1"] <= 2 * 10**9:
        st = random.Random(seed)
        y1, carry = case["y1"] + st.randrange(10**5), st.randrange(-5000, 5000)
        mu = _mu_window(y1, case["len"])
        if case["out"] == "mu":
            return torch.from_numpy(mu)
        return torch.from_numpy((carry + np.cumsum(mu, dtype=np.int64)).astype(np.int32))
    if case["kind"] not in ("query", "resident") or case["n"] > 10**11:
        return None
    n = _targets(case, seed)[0]
    u = case.get("u") or max(math.isqrt(n) + 1, min(n, int(_limit([n]))))
    X = n // u
    table = np.concatenate(([0], np.cumsum(_mu_window(1, n // (X + 1) + 1), dtype=np.int64)))
    m = np.zeros(X + 1, dtype=np.int64)
    for x in range(X, 0, -1):
        k = n // x
        s = math.isqrt(k)
        j = np.arange(X // x + 1, k // (s + 1) + 1, dtype=np.int64)
        q = k // np.arange(1, s + 2, dtype=np.int64)
        m[x] = (1 - m[2 * x::x].sum() - table[k // j].sum() -
                (table[1:s + 1] * (q[:-1] - q[1:])).sum())
    return [int(m[1]), m[1:]]
