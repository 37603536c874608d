"""Block fixed-point element arithmetic of the double-precision kernels, on the
host (tests/fixedpoint/check.cpp): primitives at the edges of their ranges
within the units they promise; the element routines no further from the element
in long double than the double-precision routines, norm-wise per component (10 %
for the spread of a finite sample); data out of range left alone."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_fixed_point_arithmetic(tmp_path):
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-I" + os.path.join(HERE, "flopcount"),
                           "-o", exe, os.path.join(HERE, "fixedpoint", "check.cpp")])
    out = subprocess.check_output([exe], text=True)
    lines = [m.groups() for m in re.finditer(r"^(\S+) (\S+) (\S+)$", out, re.M)]
    assert len(lines) > 100
    bad = [(name, float(v), float(lim)) for name, v, lim in lines if not float(v) <= float(lim)]
    assert not bad, bad
