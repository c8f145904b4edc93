"""The integer-ALU FP64 arithmetic at its rare branches: discarded bits a unit from
one half, carries through a kept part of ones, quotients and roots a few remainders
from an integer (soft_fp64_edges.h solves for the operands).  On the host here,
against its IEEE operations; test_gpu_soft_fp64.py runs the same operands on the
GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rare_branches_are_ieee(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fno-fast-math",
                           os.path.join(HERE, "soft_fp64_edges_check.cpp"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True)
    rows = [[int(x) for x in line.split()] for line in out.stdout.splitlines()]
    assert [r[1] for r in rows] == [0, 0, 0], out.stdout
    assert rows[0][0] > 500_000 and rows[1][0] > 100_000 and rows[2][0] > 100_000
