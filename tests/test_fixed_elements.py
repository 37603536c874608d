"""Fixed-point element routines on the host over elements of many kinds
(tests/fixedpoint/elements.cpp): no shift count, operand or accumulator out of
the range that the arithmetic relies on, in any formulation, and the results of
the double-precision routines."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_fixed_point_elements(tmp_path):
    exe = str(tmp_path / "elements")
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-Wno-unused-function",
                           "-I" + os.path.join(HERE, "flopcount"), "-o", exe,
                           os.path.join(HERE, "fixedpoint", "elements.cpp")])
    out = subprocess.check_output([exe], text=True)
    lines = [m.groups() for m in re.finditer(r"^(\S+) (\S+) (\S+)$", out, re.M)]
    assert len(lines) > 100
    bad = [(name, float(v), float(lim)) for name, v, lim in lines if not float(v) <= float(lim)]
    assert not bad, bad
