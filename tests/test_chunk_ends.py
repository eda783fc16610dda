"""No chunk of large primes crosses 2^30 or 2^32: its primes take one kernel form."""
import os
import subprocess

import pytest

from tests.conftest import ROOT
from tests.test_plan_classes import _cuda_include

SRC = os.path.join(ROOT, "tests", "host", "chunk_check.cpp")


def test_chunk_ends(tmp_path):
    inc = _cuda_include()
    if inc is None:
        pytest.skip("CUDA headers not found (cuda_runtime.h)")
    exe = str(tmp_path / "chunk_check")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", inc, "-o", exe, SRC])
    a, b = 1 << 30, 1 << 32
    cases = {(65536, a - 1): a - 1, (65536, a): a - 1, (65536, 1 << 40): a - 1, (a - 2, b): a - 1,
             (a - 1, a + 5): a + 5, (a - 1, b - 1): b - 1, (a - 1, b): b - 1, (a, 1 << 33): b - 1,
             (b - 2, b + 1): b - 1, (b - 1, b): b, (b - 1, 1 << 40): 1 << 40, (b, 1 << 40): 1 << 40, (7, 8): 8}
    text = "".join(f"{lo} {hi}\n" for lo, hi in cases)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == list(cases.values())


@pytest.mark.gpu
@pytest.mark.parametrize("chunk", [1 << 27, (1 << 31) + 12345, 1 << 40])
def test_wide_chunks_give_the_same_bits(chunk):
    """Primes on both sides of 2^32 in chunks of any width: one cut at 2^30, one at
    2^32, and the same bitset."""
    cs = pytest.importorskip("paper_2012_03771_gb300")
    args = (503, 210, 10**6 + 3, 1000, 3000, (1 << 32) + 200_000_001)
    got = []
    for width in (0, chunk):
        with cs.Plan(*args, threshold=1 << 29, chunk_numbers=width) as p:
            p.sieve().sync()
            got.append(p.counts()[1:])
            if width == 1 << 40:
                assert p.info.n_large_chunks == 3
    assert got[0] == got[1]
