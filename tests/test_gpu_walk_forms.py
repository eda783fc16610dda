"""The walk's forms at the edges of its tables: the column mask in shared memory
and (SL of 65,536 and more) in global memory, with direct clears and with hit
buckets, and divisors whose wheel test covers d's primes up to 11, only some of
them, or none; whole bitsets, F, counts and checksum against the oracle."""
import numpy as np
import pytest

import oracle.oracle as O
import paper_2012_03771_gb300 as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [1, 2, 3, 6, 15, 30, 77, 210, 2310, 2 * 3 * 5 * 7 * 97])
@pytest.mark.parametrize("SL", [300, 65_504, 65_536])
def test_walk_forms_match_oracle(d, SL):
    args = (101, d, 10**6 + 77, 40 if SL > 300 else 900, SL, 400_000)
    m_ref, bits_ref, F_ref = O.full_sieve(*args)
    for kw in ({}, {"hit_buckets": 2}, {"m_classes": 3, "item_hits": 4}, {"m_classes": 1}, {"large_mode": 1}):
        with cs.Plan(*args, threshold=max(2 * SL, 600), **kw) as plan:
            plan.sieve(torch.cuda.current_stream()).sync()
            counts, F, h = plan.counts()
            assert np.array_equal(plan.rows(), m_ref)
            assert np.array_equal(plan.bitset(), bits_ref), (d, SL, kw)
            assert F == int(F_ref.sum()) and h == O.bitset_hash(bits_ref)
            assert np.array_equal(counts, O.row_counts(bits_ref))


def test_walk_without_the_wheel_clears_every_hit():
    args = (101, 2310, 10**6 + 77, 900, 300, 400_000)
    m_ref, bits_ref, F_ref = O.full_sieve(*args, wheel=False)
    for kw in ({}, {"hit_buckets": 2}, {"m_classes": 3}):
        with cs.Plan(*args, threshold=600, no_wheel=True, **kw) as plan:
            plan.sieve(torch.cuda.current_stream()).sync()
            assert np.array_equal(plan.bitset(), bits_ref), kw
            assert plan.counts()[1] == int(F_ref.sum())
