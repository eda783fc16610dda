"""Searches of few rows or few primes, whose launches are cut differently: one
row per tile, columns in several pieces, light chunks at their full width, small
work items and the threshold raised over the class chunks; whole bitsets against
the oracle."""
import numpy as np
import pytest

import oracle.oracle as O
import paper_2012_03771_gb300 as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P, d, M_inc, SL, L", [
    (503, 210, 4, 9000, 3 * 10**6),          # one row, or none
    (503, 210, 44, 9000, 3 * 10**6),         # fewer rows than SMs: columns cut
    (101, 30, 700, 31, 10**6),               # one word of columns
    (503, 210, 1000, 2000, 10**6),           # every prime above T in one chunk
    (503, 2310, 3000, 7000, 5 * 10**6),      # class chunks, then one light chunk
    (97, 15, 500, 3000, 2 * 10**6),          # odd d: no classes
])
def test_small_searches_match_oracle(P, d, M_inc, SL, L):
    args = (P, d, 10**6 + 3, M_inc, SL, L)
    m_ref, bits_ref, F_ref = O.full_sieve(*args)
    for kw in ({}, {"threshold": max(2 * SL, P)}, {"hit_buckets": 2}):
        with cs.Plan(*args, **kw) as plan:
            plan.sieve(torch.cuda.current_stream()).sync()
            counts, F, h = plan.counts()
            assert np.array_equal(plan.rows(), m_ref)
            assert np.array_equal(plan.bitset(), bits_ref), kw
            assert F == int(F_ref.sum()) and h == O.bitset_hash(bits_ref)
            assert np.array_equal(counts, O.row_counts(bits_ref))
