"""An m-range above 2^30: every prime's walk is cut into segments of at most 2^30 m,
whose offsets and clamped steps add up below 2^32."""
import numpy as np
import pytest

import oracle.oracle as O
import paper_2012_03771_gb300 as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_m_range_above_2_30_matches_oracle():
    """P = 101, d = 510510, X = 2, primes to 6e9: the light primes' steps are about p /
    5 and reach past a segment.  Rows of both segments and at their ends against the
    oracle, and the large primes' factors against M_c W sum 1/p (4e8 of them: a
    standard deviation of 5e-5)."""
    P, d, M_start, M_inc, SL, L = 101, 510510, 10**9 + 7, (1 << 30) + 5_000_001, 2, 6 * 10**9
    with cs.Plan(P, d, M_start, M_inc, SL, L) as plan:
        plan.sieve(torch.cuda.current_stream()).sync()
        m, st, T = plan.rows(), plan.stats(), int(plan.info.threshold)
        half = int(np.searchsorted(m, M_start + (M_inc + 1) // 2))
        rows = sorted({0, 1, half - 2, half - 1, half, half + 1, len(m) - 2, len(m) - 1} |
                      {int(i) for i in np.linspace(0, len(m) - 1, 50)})
        got = np.stack([plan.fetch_rows(r, 1)[0] for r in rows])
    bits, F, _ = O.sieve(P, d, SL, L, [int(m[r]) for r in rows])
    assert int(F.sum()) > 0 and np.array_equal(got, bits)
    expected = len(m) * len(O.columns(P, d, SL)) * O.prime_stats(T, L)[2]
    assert abs(st["F_large"] / expected - 1) < 5e-4
