"""The walk's step and first-hit routines on nearest-integer Euclid steps
(cs_basis.cuh), compiled for the host, against the paper's recursion G."""
import math
import os
import random
import subprocess

import pytest

import oracle.oracle as O
from tests.conftest import ROOT

SRC = os.path.join(ROOT, "tests", "host", "basis_check.cpp")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("basis") / "basis_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", out, SRC])
    return out


@pytest.mark.parametrize("lo, hi, w_lo, accepted", [
    (1 << 17, 1 << 30, 512, 0.99),                 # 32-bit primes
    (1 << 30, 1 << 31, 1024, 0.99),                # the narrowest 64-bit ones
    (1 << 31, 1 << 36, 4000, 0.98),
    (1 << 36, 1 << 40, 20000, 0.8),
])
def test_steps_and_first_hits_equal_the_paper_recursion(exe, lo, hi, w_lo, accepted):
    """Whatever the routines return is G's answer for the two step windows and
    for the first hit's window; ordinary residues are accepted, and residues
    next to 0, p and the window are answered or refused."""
    rng = random.Random(lo)
    cases, ordinary = [], 0
    while len(cases) < 3000:
        p = rng.randrange(lo, hi) | 1
        w = min(rng.choice((w_lo, w_lo + 1, 2 * rng.randrange(w_lo // 2, 25_000), 1 << 21)), p // 4)
        edge = rng.random() < 0.1
        r = rng.choice((1, 2, p - 1, p - 2, w, w + 1, p - w, p // 2, p // 3)) if edge else rng.randrange(1, p)
        if w < w_lo or math.gcd(p, r) != 1:
            continue
        cases.append((p, r, w, rng.choice((w + 1, p - 1, rng.randrange(w + 1, p))), edge))
    text = "".join(f"{p} {r} {w} {v0}\n" for p, r, w, v0, _ in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    taken = 0
    for (p, r, w, v0, edge), line in zip(cases, out):
        ok, a, da, b, ub, hit, t, y = (int(v) for v in line.split())
        ordinary += not edge
        taken += (not edge) and ok and hit
        if ok:
            ga, gb = O.G(p, r, p - w, p - 1), O.G(p, r, 1, w)
            assert (a, da, b, ub) == (ga, p - r * ga % p, gb, r * gb % p), (p, r, w)
        if hit:
            g = O.G(p, r, p - v0, p - v0 + w)
            assert (t, y) == (g, (v0 + r * g) % p), (p, r, w, v0)
    assert taken > accepted * ordinary

