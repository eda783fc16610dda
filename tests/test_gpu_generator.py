"""The prime generator at the edges of its segments and base primes: ranges that
end inside a word, a segment of the smallest and of more than the largest size,
squares of the base primes on both sides of the warp/thread split, numbers below
the pre-sieve's primes and next to 2^40."""
import math

import numpy as np
import pytest

import paper_2012_03771_gb300 as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _primes(lo, hi):
    """Primes lo < p <= hi by a plain segmented sieve."""
    base = np.ones(math.isqrt(hi) + 1, dtype=bool)
    base[:2] = False
    for i in range(2, math.isqrt(len(base)) + 1):
        if base[i]:
            base[i * i::i] = False
    seg = np.ones(hi - lo, dtype=bool)                 # lo + 1 .. hi
    seg[:max(0, 1 - lo)] = False                       # 1
    for q in np.flatnonzero(base):
        q = int(q)
        first = max(q * q, (lo // q + 1) * q)
        seg[first - lo - 1::q] = False
    return np.flatnonzero(seg).astype(np.uint64) + np.uint64(lo + 1)


@pytest.mark.parametrize("lo, hi", [
    (0, 2), (0, 31), (0, 2047), (0, 2048), (0, 2049), (30, 3000),
    (1, 1 << 20),
    (1019 * 1019 - 4, 1021 * 1021), (1021 * 1021 - 1, 1031 * 1031 + 1),
    (1 << 30, (1 << 30) + 2048 + 62), ((1 << 31) - 5000, (1 << 31) + 5000),
    (10**10 + 1, 10**10 + 1 + 2 * 1024 * 304 + 7),     # one smallest segment per CTA, and a rest
    (9 * 10**9, 9 * 10**9 + 3 * (1 << 27) // 2 + 1),   # segments of several sizes
    ((1 << 40) - (1 << 21), 1 << 40),
])
def test_prime_list_at_segment_edges(lo, hi):
    ref = _primes(lo, hi)
    for call in (cs.cs_primes, cs.cs_primes_static):
        out = torch.zeros(len(ref) + 8, dtype=torch.int64, device="cuda")
        n = call(lo, hi, out.data_ptr(), len(out))
        assert n == len(ref)
        assert np.array_equal(np.sort(out[:n].cpu().numpy()).astype(np.uint64), ref)
