"""The apply groups of the hit buckets with the columns that become records
(record_columns in csrc/cs_buckets.h), compiled for the host, as the plan asks for
them: the wheel's cells are counted, not recorded."""
import math
import os
import subprocess

import pytest

from tests.conftest import ROOT
from tests.test_buckets_host import CTAS, L2_GB300, _chunks

SRC = os.path.join(ROOT, "tests", "host", "records_check.cpp")


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("records") / "records_check")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-o", out, SRC])
    return out


def _run(exe, rows):
    text = ""
    for M_c, wpr, W, wheel, chunks in rows:
        text += f"{M_c} {wpr} {W} {L2_GB300} {CTAS} {len(wheel)} {' '.join(map(str, wheel))} {len(chunks)} "
        text += " ".join(f"{lo} {hi}" for lo, hi in chunks) + "\n"
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
    return [tuple(int(v) for v in line.split()) for line in out]


def test_large_search_groups(exe):
    """large_1019: 3814 of 16,682 columns become records (the wheel of 210 leaves
    8/35 of them), 7 apply groups, as the plan reports on the GPU; without the
    wheel every column, 20 groups."""
    chunks = _chunks(100002, 10**11)
    wheel, plain = _run(exe, [(2285714, 261, 16682, (2, 3, 5, 7), chunks), (2285714, 261, 16682, (), chunks)])
    assert wheel == (math.ceil(16682 * 8 / 35), 7, 1)
    assert plain == (16682, 20, 1)


@pytest.mark.parametrize("wheel", [(), (2,), (3, 5), (2, 3, 5, 7, 11), (2, 3, 13), (17, 101)])
def test_record_columns(exe, wheel):
    """Primes above 11 are not in the walk's wheel test: their cells are recorded."""
    for W in (0, 1, 64, 9618):
        (cols, _, last), = _run(exe, [(5000, 200, W, wheel, [(10**6, 2 * 10**6)])])
        assert abs(cols - W * math.prod(1 - 1 / q for q in wheel if q <= 11)) < 1 + 1e-9 and last
