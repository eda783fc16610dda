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


@pytest.mark.parametrize("M_inc", [1, 2, 9, 16, 17, 255, 256, 257])
@pytest.mark.parametrize("P, d, L, threshold", [(101, 6, 300_000, 700), (101, 15, 300_000, 700), (503, 210, 1_100_000_000, 0)])
def test_few_m_equal_prepared_walkers(P, d, L, threshold, M_inc):
    """Chunks over few m, where every m is tried, against the walk's prepared
    walkers: odd m and every m, 32-bit primes and some above 2^30, at the edges of
    a pass and of the range that takes this form."""
    for SL in (300, 9000):
        args = (P, d, 10**6 + 3, M_inc, SL, L)
        out = []
        for prep in (0, 2):
            with cs.Plan(*args, threshold=max(threshold, 2 * SL), walk_prep=prep) as plan:
                plan.sieve(torch.cuda.current_stream()).sync()
                # primes above M_inc S / Q (at most one expected hit) try every m
                few = M_inc <= 256 and M_inc * (2 * SL + 1) // (2 if d % 2 == 0 else 1) < L
                if few and not prep:
                    assert plan.info.prep_chunks < plan.info.n_large_chunks
                out.append((plan.bitset(), plan.counts(), plan.stats()))
        assert np.array_equal(out[0][0], out[1][0])
        assert out[0][1][1:] == out[1][1][1:]
        for k in ("F_small", "F_large", "hits_all"):
            assert out[0][2][k] == out[1][2][k]
