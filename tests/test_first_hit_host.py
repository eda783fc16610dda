"""The walk's first hit (near_first_hit in cs_basis.cuh), compiled for the host, on
every window the walk gives it: 2SL from 2 up, also below the 512 and 1024 from
which near_steps takes the steps, against the paper's recursion G."""
import math
import os
import random
import subprocess

import pytest

import oracle.oracle as O
from tests.conftest import ROOT

SRC = os.path.join(ROOT, "tests", "host", "first_hit_check.cpp")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("first_hit") / "first_hit_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", out, SRC])
    return out


@pytest.mark.parametrize("w_lo, w_hi, p_lo, p_hi", [
    (2, 40, 5, 1 << 16), (2, 511, 1 << 12, 1 << 30), (512, 1023, 1 << 17, 1 << 40), (1024, 1 << 21, 1 << 22, 1 << 40),
])
def test_first_hits_of_every_window_equal_the_paper_recursion(exe, w_lo, w_hi, p_lo, p_hi):
    rng = random.Random(w_lo + p_hi)
    cases = []
    while len(cases) < 2500:
        p = int(math.exp(rng.uniform(math.log(p_lo), math.log(p_hi)))) | 1
        w = min(2 * int(math.exp(rng.uniform(math.log(w_lo / 2), math.log(w_hi / 2)))), p - 3) // 2 * 2
        edge = rng.random() < 0.2
        r = rng.choice((1, 2, p - 1, p - 2, w, w + 1, p - w, p // 2, p // 3)) if edge else rng.randrange(1, p)
        if w < 2 or not 0 < r < p or math.gcd(p, r) != 1 or w + 1 >= p:
            continue
        cases.append((p, r, w, rng.choice((w + 1, p - 1, rng.randrange(w + 1, p)))))
    text = "".join(" ".join(map(str, c)) + "\n" for c in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    taken = 0
    for (p, r, w, v0), line in zip(cases, out):
        v = [int(x) for x in line.split()]
        g = O.G(p, r, p - v0, p - v0 + w)
        for k in (0, 6, 12):
            assert v[k]
            if v[k + 3]:
                taken += 1
                assert (v[k + 4], v[k + 5]) == (g, (v0 + r * g) % p), (p, r, w, v0, k)
    assert taken > 2500
