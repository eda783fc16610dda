"""Which form the light chunks of a search over few m take: an every-m chunk solves
nothing, a prepared walker solves for its two steps."""
import statistics

import pytest

import paper_2012_03771_gb300 as cs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P, d, M_inc, SL, L, T, every_m", [
    (101, 6, 16, 300, 300_000, 10_000, True),             # 8 odd m, at most one expected hit
    (503, 210, 44, 18_000, 1_100_000_000, 0, True),       # also 64-bit primes
    (101, 6, 256, 20_000, 10_000_000, 6_000_000, False),  # 128 odd m, half a hit a prime
    (97, 15, 80, 25_000, 10_000_000, 5_000_000, False),
    (97, 15, 200, 31, 300_000, 100_000, False),           # more m than a walker costs
])
def test_form_of_few_m(P, d, M_inc, SL, L, T, every_m):
    args = (P, d, 10**6 + 3, M_inc, SL, L)
    got = {}
    for prep in (0, 2):
        with cs.Plan(*args, threshold=T or 2 * SL * M_inc, walk_prep=prep) as p:
            p.sieve(torch.cuda.current_stream()).sync()
            info, st = p.info, p.stats()
            got[prep] = p.counts()[1:]
            assert info.n_large_chunks > 0 and st["hits_all"] > 0
            if prep == 0 and every_m:
                assert info.prep_chunks == 0 and st["solves"] == 0
            else:
                assert info.prep_chunks == info.n_large_chunks and st["solves"] > 0
    assert got[0] == got[2]


@pytest.mark.parametrize("P, d, M_inc, SL, L", [
    (97, 15, 120, 20_000, 10**8),     # 120 m from low primes on (2010 us every m, 370 prepared, before warps stayed together)
    (97, 15, 256, 20_000, 10**8),     # more m than a walker costs (3490 us every m, 410 prepared)
    (953, 210, 99, 5_000, 10**8),     # 50 odd m (760 us every m, 410 prepared)
])
def test_chosen_form_is_about_as_fast_as_prepared_walkers(P, d, M_inc, SL, L):
    s = torch.cuda.current_stream()
    ms = {}
    for prep in (2, 0):
        with cs.Plan(P, d, 10**6 + 3, M_inc, SL, L, walk_prep=prep) as p:
            t = []
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(s)
                p.sieve(s)
                b.record(s)
                s.synchronize()
                t.append(a.elapsed_time(b))
            ms[prep] = statistics.median(t[3:])
    assert ms[0] < 1.4 * ms[2]
