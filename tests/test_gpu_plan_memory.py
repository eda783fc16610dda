"""Device memory a plan holds for its large primes."""
import pytest

import paper_2012_03771_gb300 as cs

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M_inc, SL, per_prime", [
    (1000, 2000, 36),     # one chunk from the threshold on: p, r, v and the walker, 4 + 4 + 4 + 24 bytes
    (6, 20, 12),          # every m tried: no walkers
])
def test_large_prime_buffers_follow_the_prime_count(M_inc, SL, per_prime):
    with cs.Plan(503, 210, 1, M_inc, SL, 130_000_000) as p:
        p.sieve().sync()
        held = int(p.info.device_bytes) - int(p.info.bitset_bytes)
        n = p.stats()["n_large_primes"]
    # 3% above the count, 16 bytes for each small prime of the threshold, the tables
    assert held <= 1.03 * per_prime * n + 8_000_000
