"""The integer-ALU products, quotients and roots on the GPU itself, against its
IEEE operations: the carry chain that rounds a product is assembly there, and the
classes that tell a wrong rounding -- ties, carries through a kept part of ones --
hardly ever come up in a run.  tests/soft_fp64_device_check.cu has the classes."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_device_results_are_ieee(tmp_path):
    exe = str(tmp_path / "soft_fp64_device_check")
    subprocess.check_call([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                           "-std=c++17", "-fmad=false", os.path.join(HERE, "soft_fp64_device_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
    rows = [[int(x) for x in line.split()] for line in out.stdout.splitlines()]
    assert [r[1] for r in rows] == [0, 0, 0]
    assert all(r[0] >= 4_000_000 for r in rows)
