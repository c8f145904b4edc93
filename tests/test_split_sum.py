"""The FP32 read-out's sums over a tile of 64 walkers, on the host: numbers split at
2^-16 and 2^-33, so that only the last level (below 2^-28, 64 additions that round at
2^-53 at most, one conversion) is inexact: within 64 2^-53 + 2^-49, below 3 units of
2^-48, of the exact sum, at the ends of the levels' binades too."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_sums_are_exact_to_48_bits(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", os.path.join(HERE, "split_sum_check.cpp"),
                           "-o", exe])
    sums, worst = subprocess.check_output([exe], text=True).split()
    assert int(sums) == 600_000
    assert float(worst) <= 3.0
