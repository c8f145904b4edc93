"""The integer arithmetic of the plain form's read-out and of the b-values, on
the host: every term alpha e^{-i phi} within 2^-51.8 + 2^-55 |phi|max of its
value in extended precision (the phase is within 2^-57 of the largest; cosine
and sine carry 52 to 53 fraction bits), unbiased to 2^-57 + 2^-57 |phi|max; and
additions taken 32 at a time bit for bit the ones taken one after another."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2012_06478_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_terms_and_additions(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC,
                           os.path.join(HERE, "readout_fixed_check.cpp"), "-o", exe])
    lines = [x.split() for x in subprocess.check_output([exe], text=True).splitlines()]
    terms = [x for x in lines if x[0] == "term"]
    assert len(terms) == 27
    for _, e2, largest, mean in terms:
        phi = 2.0 ** (int(e2) + 1)
        assert float(largest) <= 2.0 ** -51.8 + 2.0 ** -55 * phi, (e2, largest)
        assert abs(float(mean)) <= 2.0 ** -57 + 2.0 ** -57 * phi, (e2, mean)
    assert lines[-1] == ["chain", "0"]
