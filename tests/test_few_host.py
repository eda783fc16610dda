"""From which prime on the light chunks try every m (few_from in cs_classes.h),
compiled for the host, against both forms' measured times."""
import os
import subprocess

import pytest

from tests.conftest import ROOT
from tests.test_plan_classes import _cuda_include

SRC = os.path.join(ROOT, "tests", "host", "few_check.cpp")

# (M_inc, Q, S, k, every m, prepared walkers): ps a prime of one GB300 on a chunk of
# min(2^k, 2^27) numbers from 2^k on, whichever of the two the plan would take
MEASURED = [
    (5, 2, 4001, 27, 6, 22), (44, 2, 4001, 29, 7, 23), (128, 2, 4001, 27, 11, 22), (256, 2, 4001, 27, 17, 22),
    (256, 2, 4001, 29, 16, 23), (64, 2, 16001, 27, 9, 22), (128, 2, 16001, 25, 19, 28), (256, 2, 16001, 25, 31, 30),
    (256, 2, 16001, 27, 20, 23), (20, 2, 50001, 27, 8, 22), (44, 2, 50001, 27, 9, 22), (64, 2, 50001, 27, 10, 22),
    (128, 2, 50001, 24, 50, 41), (128, 2, 50001, 27, 16, 23), (192, 2, 50001, 25, 41, 31),
    (256, 2, 50001, 25, 52, 31), (256, 2, 50001, 26, 34, 27), (256, 2, 50001, 29, 20, 23), (44, 1, 4001, 27, 9, 22),
    (128, 1, 4001, 27, 17, 22), (192, 1, 4001, 27, 23, 22), (256, 1, 4001, 28, 28, 23), (44, 1, 16001, 29, 10, 22),
    (128, 1, 16001, 24, 50, 39), (128, 1, 16001, 27, 20, 23), (192, 1, 16001, 26, 33, 26), (20, 1, 50001, 27, 9, 22),
    (44, 1, 50001, 30, 11, 26), (64, 1, 50001, 27, 15, 23), (128, 1, 50001, 24, 85, 41), (256, 1, 50001, 27, 46, 26),
]


def test_the_cheaper_form_is_taken(tmp_path):
    """The form the rule takes is never more than 15% slower than the other one, and
    no prime with more than one expected hit tries every m."""
    inc = _cuda_include()
    if inc is None:
        pytest.skip("CUDA headers not found (cuda_runtime.h)")
    exe = str(tmp_path / "few_check")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-I", inc, "-o", exe, SRC])
    text = "".join(f"{M} {S} {Q}\n" for M, Q, S, *_ in MEASURED)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    for (M, Q, S, k, every, prep), start in zip(MEASURED, out):
        assert int(start) >= -(-M // Q) * S
        if 1 << k >= int(start):
            assert every <= 1.15 * prep, (M, Q, S, k)
        else:
            assert prep <= 1.15 * every, (M, Q, S, k)
