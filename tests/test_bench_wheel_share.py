"""bench.py's share of the stored cells that the wheel leaves, which turns the walk's
stored hits into bit clears, against every cell of small searches."""
import math

import pytest

import bench
from paper_2012_03771_gb300 import workloads


@pytest.mark.parametrize("P, d, SL", [(13, 6, 40), (13, 210, 60), (31, 30, 100), (13, 1, 25), (19, 17, 50), (13, 2310, 80), (11, 15, 1)])
def test_share_is_the_mean_over_rows_and_columns(P, d, SL):
    K = math.prod(q for q in range(2, P + 1) if all(q % f for f in range(2, q)) and d % q)
    w = math.gcd(d, 2310)                         # d's primes up to 11
    cols = [x for x in range(-SL, SL + 1) if math.gcd(x, K) == 1]
    rows = [m for m in range(d) if math.gcd(m, d) == 1] or [1]
    left = sum(math.gcd(m * K + x, w) == 1 for m in rows for x in cols)
    got = bench.wheel_share(workloads.SieveParams(P=P, d=d, M_start=1, M_inc=1, SL=SL, L=100))
    assert abs(got - left / (len(rows) * len(cols))) < 1e-12
