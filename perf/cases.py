"""Performance cases of the Combined Sieve: what a user's program runs, in the
sizes it runs them in.

Each case is one call sequence through the package's public entry points on
plans (or a batch, or a server) that the program keeps:

  sieve   Plan.sieve and the per-row survivor counts, F and checksum a search
          reads back to rank its rows; the bitset stays on the device.
  batch   Batch.run over the plans of several searches that share residue
          caches, then every plan's counts.
  serve   requests submitted to a Server as its slots free up, each result
          fetched to the host (bitset and counts) and released.

`seed` moves the searches by a multiple of d, so another seed sieves other numbers
with as many rows; the sizes come from the case alone.  Words and counts are
returned in signed types of their width, the checksum as a signed 64-bit number.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2012_03771_gb300 as cs


def _sieve_case(name, P, d, M_start, M_inc, SL, L, **tuning):
    return {"name": name, "kind": "sieve", "P": P, "d": d, "M_start": M_start, "M_inc": M_inc, "SL": SL,
            "L": L, **tuning}


def listed():
    return [
        # the smallest call: a quick look at 1000 multipliers, primes to 1e6
        # (the shape of the smoke test)
        _sieve_case("quick_503", 503, 210, 1, 1000, 2000, 10**6),
        # the small plain search: K = 503#/210, primes to 1e7
        _sieve_case("plain_503", 503, 210, 1, 1000, 7000, 10**7),
        # the paper-shaped search around the 35,308 record gap, with the
        # threshold and tile height the autotuner keeps for it
        _sieve_case("search_953", 953, 210, 100_000_000, 100_000, 20_000, 10**9, threshold=120_003, tile_rows=16),
        # the same search kept in the compact layout (rows of the columns the wheel leaves)
        _sieve_case("compact_953", 953, 210, 100_000_000, 100_000, 20_000, 10**9, layout=1),
        # one search of the uneven mix: d = 2310, a ragged range, primes on both
        # sides of 2^30
        _sieve_case("uneven_701", 701, 2310, 7_654_321, 12_347, 11_117, 2_300_000_000),
        # a wide search of the mix: a bitset above L2, primes to 1e10
        _sieve_case("wide_1019", 1019, 2310, 31_415_926, 333_333, 24_999, 10**10),
        # few intervals: ten rows of K = 1511#/210 (a point of the speed-up
        # curve), where almost all work is per prime
        _sieve_case("few_1511", 1511, 210, 1, 44, 18_000, 10**10),
        # the largest search: around the 36,702 record gap, primes to 1e11, a
        # 4.77 GB bitset, with the autotuner's threshold and tile height
        _sieve_case("large_1019", 1019, 210, 164_000_000, 10_000_000, 25_000, 10**11, threshold=100_002,
                    tile_rows=8),
        # eight searches of the uneven mix in one captured batch over shared residue caches
        {"name": "batch_8", "kind": "batch", "n": 8, "M_lo": 1000, "M_hi": 100_000, "L_lo": 10**8, "L_hi": 10**9,
         "mix": 11},
        # eight small requests through the server, two slots
        {"name": "serve_8", "kind": "serve", "n": 8, "M_lo": 1000, "M_hi": 3000, "L_lo": 10**6, "L_hi": 10**7,
         "mix": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("sieve", "sieve", "sieve", "sieve", "few", "compact", "batch", "serve"))
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(2, 12), "M_lo": 1000, "M_hi": _log_int(rng, 3000, 200_000),
                "L_lo": 10**7, "L_hi": _log_int(rng, 3 * 10**7, 10**9), "mix": rng.randrange(1 << 30)}
    if kind == "serve":
        return {"kind": "serve", "n": rng.randint(2, 12), "M_lo": 100, "M_hi": _log_int(rng, 300, 10_000),
                "L_lo": 10**6, "L_hi": _log_int(rng, 3 * 10**6, 10**8), "mix": rng.randrange(1 << 30)}
    case = {"kind": "sieve", "P": rng.choice((503, 701, 953, 1019, 1511)), "d": rng.choice((30, 210, 2310)),
            "M_start": _log_int(rng, 10**6, 10**8), "M_inc": _log_int(rng, 100, 10**6),
            "SL": rng.randint(2000, 25_000), "L": _log_int(rng, 10**6, 10**10)}
    if kind == "few":
        case["M_inc"] = rng.randint(5, 99)
    if kind == "compact":
        case.update(d=rng.choice((30, 210)), layout=1)
    return case


# ------------------------------------------------------------------ sizes

def _shift(seed, d):
    """How far the seed moves a search's first multiplier (a multiple of d: as many rows)."""
    return d * random.Random(seed).randrange(1_000_000 // d)


def _signed(h):
    return h - (1 << 64) if h >> 63 else h


def _members(case):
    """The searches of a batch or of a server's requests: P, d, M_inc, SL, L from
    the mix's own number, every other d 2310."""
    rng = random.Random(case["mix"])
    Ps = (503, 1019) if case["kind"] == "batch" else (503, 701)
    out = []
    for k in range(case["n"]):
        out.append((Ps[k % 2], (210, 2310)[k // 2 % 2], 10**6 + rng.randrange(10**7),
                    _log_int(rng, case["M_lo"], case["M_hi"]), rng.randint(5000, 25_000 if case["kind"] == "batch" else 9000),
                    _log_int(rng, case["L_lo"], case["L_hi"])))
    return out


def _searches(case):
    if case["kind"] == "sieve":
        return [tuple(case[k] for k in ("P", "d", "M_start", "M_inc", "SL", "L"))]
    return _members(case)


def _small_primes(n):
    s = np.ones(n + 1, dtype=bool)
    s[:2] = False
    for i in range(2, int(n ** 0.5) + 1):
        if s[i]:
            s[i * i::i] = False
    return np.flatnonzero(s)


def _k_primes(P, d):
    return [int(q) for q in _small_primes(P) if d % q]


def _columns(P, d, SL):
    """x in [-SL, SL] coprime to K."""
    keep = np.ones(2 * SL + 1, dtype=bool)
    for q in _k_primes(P, d):
        keep[SL % q::q] = False
    return np.flatnonzero(keep) - SL


def work(case):
    """Bytes: the bitset and the per-row counts, written once.  Operations: one per
    enumerated factor (a hit of a prime on a stored cell, M_c W sum 1/p by
    Mertens) and one per sieving prime."""
    bytes_, ops = 0, 0.0
    for P, d, _, M_inc, SL, L in _searches(case):
        phi = 1.0
        for q in (2, 3, 5, 7, 11):
            if d % q == 0:
                phi *= 1 - 1 / q
        rows, W = M_inc * phi, len(_columns(P, d, SL))
        W_stored = W
        if case.get("layout") == 1:
            W_stored = W * phi
        bytes_ += int(rows * (8 * math.ceil(W_stored / 64) + 4))
        ops += rows * W * math.log(math.log(L) / math.log(P)) + L / math.log(L)
    return {"bytes": bytes_, "flops": ops}


# ------------------------------------------------------------------ passes

class _DeviceWords:
    """A plan's device bitset as an array other libraries read in place."""

    def __init__(self, plan):
        self.plan = plan
        self.__cuda_array_interface__ = {"shape": (int(plan.M_c), int(plan.wpr)), "typestr": "<i8", "version": 3,
                                         "data": (cs.cs_device_bitset(plan.h), False), "strides": None}


def _bitset_view(plan):
    if plan.M_c * plan.wpr == 0:
        return torch.empty((int(plan.M_c), int(plan.wpr)), dtype=torch.int64, device="cuda")
    return torch.as_tensor(_DeviceWords(plan), device="cuda")


def prepare(case, seed):
    cs.load()
    state = {"case": case}
    if case["kind"] == "sieve":
        tuning = {k: case[k] for k in ("threshold", "tile_rows", "layout") if k in case}
        P, d, M_start, M_inc, SL, L = _searches(case)[0]
        plan = cs.Plan(P, d, M_start + _shift(seed, d), M_inc, SL, L, **tuning)
        state["plan"], state["bits"] = plan, _bitset_view(plan)
    elif case["kind"] == "batch":
        members = _members(case)
        caches = {}
        for P, d, _, _, _, L in members:
            caches[P, d] = max(L, caches.get((P, d), 0))
        state["caches"] = {k: cs.Cache(k[0], k[1], L) for k, L in caches.items()}
        state["plans"] = [cs.Plan(P, d, M_start + _shift(seed, d), M_inc, SL, L, cache=state["caches"][P, d])
                          for P, d, M_start, M_inc, SL, L in members]
        state["bits"] = [_bitset_view(p) for p in state["plans"]]
        state["batch"] = cs.Batch(state["plans"])
    else:
        state["requests"] = [(P, d, M_start + _shift(seed, d), M_inc, SL, L) for P, d, M_start, M_inc, SL, L in _members(case)]
        state["server"] = cs.Server(4 << 30, max_slots=2)
    return state


def _outputs(plan, bits):
    per_row, F, h = plan.counts()
    return {"bits": bits, "per_row": per_row.view(np.int32), "F": F, "hash": _signed(h)}


def _serve(server, requests):
    results = [None] * len(requests)
    waiting, running = list(enumerate(requests)), {}
    while waiting or running:
        if waiting:
            ticket = server.submit(*waiting[0][1])
            if ticket is not None:
                running[ticket] = waiting.pop(0)[0]
                continue
        for ticket in [t for t in running if server.poll(t)]:
            plan = server.plan(ticket)
            results[running.pop(ticket)] = _outputs(plan, plan.bitset().view(np.int64))
            server.release(ticket)
    return results


def run(state):
    kind = state["case"]["kind"]
    if kind == "sieve":
        state["plan"].sieve(torch.cuda.current_stream())
        return _outputs(state["plan"], state["bits"])
    if kind == "batch":
        state["batch"].run(torch.cuda.current_stream()).sync()
        return [_outputs(p, b) for p, b in zip(state["plans"], state["bits"])]
    return _serve(state["server"], state["requests"])


# ------------------------------------------------------------------ exact

def _mix64(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def exact(case, seed):
    """The bitset, counts, F and checksum by a plain sieve of every row in numpy,
    for searches small enough to take a few seconds that way."""
    if case["kind"] != "sieve" or case.get("layout"):
        return None
    P, d, M_start, M_inc, SL, L = _searches(case)[0]
    if L > 10**7 or M_inc > 2000 or SL > 10_000:
        return None
    M_start += _shift(seed, d)
    rows = np.array([m for m in range(M_start, M_start + M_inc) if math.gcd(m, d) == 1], dtype=np.int64)
    cols = _columns(P, d, SL)
    K = math.prod(_k_primes(P, d))
    stored = np.zeros(2 * SL + 1, dtype=bool)
    stored[cols + SL] = True
    alive = np.tile(stored, (len(rows), 1))
    for q in (int(q) for q in _small_primes(P) if d % q == 0):      # the wheel of d's primes
        for i, m in enumerate(rows):
            alive[i, (SL - int(m) * K) % q::q] = False
    F = 0
    primes = [int(p) for p in _small_primes(L) if p > P]
    n_dense = sum(p <= 2 * SL for p in primes)
    for p in primes[:n_dense]:
        z = (SL - (rows % p) * (K % p)) % p                           # first offset with p | N + x
        hit = np.flatnonzero(z <= 2 * SL)
        while hit.size:
            zz = z[hit]
            F += int(np.count_nonzero(stored[zz]))
            alive[hit, zz] = False
            z[hit] += p
            hit = hit[z[hit] <= 2 * SL]
    for k in range(n_dense, len(primes), 1024):                       # at most one offset per row
        p = np.array(primes[k:k + 1024], dtype=np.int64)
        r = np.array([K % q for q in primes[k:k + 1024]], dtype=np.int64)
        z = (SL - (rows[:, None] % p) * r) % p
        i, j = np.nonzero(z <= 2 * SL)
        zz = z[i, j]
        F += int(np.count_nonzero(stored[zz]))
        alive[i, zz] = False
    bits = np.zeros((len(rows), 64 * ((len(cols) + 63) // 64)), dtype=np.uint8)
    bits[:, :len(cols)] = alive[:, cols + SL]
    words = np.packbits(bits, axis=1, bitorder="little").view("<u8")
    with np.errstate(over="ignore"):
        pos = np.arange(words.size, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        h = int(_mix64(words.reshape(-1) + pos).sum(dtype=np.uint64))
    return {"bits": torch.from_numpy(words.view(np.int64).copy()), "per_row": bits.sum(axis=1, dtype=np.int32), "F": F,
            "hash": _signed(h)}
