"""The phases of the fixed-point read-out are not off together: rounded down, they
were too small by half a unit on average, which no sum over walkers averages out and
an imaginary part near zero shows.  Over 2^18 terms the mean error of the phase is
within 2^-60.5 (the steps after the phase round at 2^-62 and 2^-63) and what the
rounding of each phase leaves: a unit's 0.29 over 2^9, six times."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2012_06478_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_mean_phase_error(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC,
                           os.path.join(HERE, "readout_bias_check.cpp"), "-o", exe])
    rows = [x.split() for x in subprocess.check_output([exe], text=True).splitlines()]
    assert len(rows) == 15
    for e2, mean, unit in rows:
        # the term's own rounding: 2^-55 in the mean square over 2^9
        assert float(mean) <= 2.0 ** -60.5 + 6 * (0.29 * float(unit) + 2.0 ** -55) / 512, (e2, mean, unit)
