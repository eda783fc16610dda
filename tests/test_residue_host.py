"""K mod p of 64-bit primes from K's limbs (cs_residue.cuh), compiled for the
host, against exact integers."""
import math
import os
import random
import subprocess

import oracle.oracle as O
from tests.conftest import ROOT

SRC = os.path.join(ROOT, "tests", "host", "residue_check.cpp")


def test_residues_equal_exact_integers(tmp_path):
    """Odd p from 2^28 to 2^40, their edges, and low words on both sides of the
    chain's limit; K = 1, one limb and whole primorials; M to 2^40."""
    exe = str(tmp_path / "residue_check")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe, SRC])
    rng = random.Random(3)
    Ks = [[], [101], [65521, 65537], [q for q in O._simple_primes(503) if 210 % q],
          [q for q in O._simple_primes(1511) if 2310 % q]]
    edges = [(1 << 28) + 3, (1 << 32) - 5, (1 << 32) - 1, (1 << 32) + 15, (1 << 40) - 87, (1 << 40) - 1]
    edges += [(h << 32) + 0xfffff7ff + d for h in (0, 1, 255) for d in (-2, 0, 2, 0x7fe)]
    cases = []
    for k in range(4000):
        p = rng.choice(edges) if k % 4 == 0 else rng.randrange(1 << rng.randint(28, 39), 1 << 40) | 1
        cases.append((p, rng.choice((1, (1 << 20) - 1, 1 << 20, (1 << 40) - 1, rng.randrange(1, 1 << 40))),
                      rng.choice((0, 25_000, (1 << 20))), rng.choice(Ks)))
    text = "".join(f"{p} {M} {s} {len(K)} {' '.join(map(str, K))}\n" for p, M, s, K in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    ways = set()
    for (p, M, s, K), line in zip(cases, out):
        r, v, chain, v2, f = (int(x) for x in line.split())
        assert v2 == v and (f - (r << 32) // p + 2) % 2**32 <= 4, (p, M, s, len(K))
        assert (r, v) == (math.prod(K) % p, (math.prod(K) * M + s) % p), (p, M, s, len(K))
        ways.add(chain)
    assert ways == {0, 1}
