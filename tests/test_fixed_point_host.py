"""The block-floating-point line contractions of csrc/fxp.h on the host (the header compiles as plain
C++): conversions of the whole exponent range, every line length, both symmetries, against long
double.  The bound per result follows from the formats: an input is cut below 2^-56 of the line's
largest value, the dropped limb products and the cut of the 64-bit sum are below 2^-57 of (largest
value) x (largest row sum), together under 2^-55 of that product, and the result is rounded once to
53 bits."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_07663_gb300", "csrc")


def test_line_contractions_on_the_host(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "fixed_point_host")
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC,
                    os.path.join(HERE, "fixed_point_host.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, f"check {r.returncode} of the conversions failed"
    rows = [line.split() for line in r.stdout.splitlines()]
    assert len(rows) == 10 * 2 * 11
    for n, sym, spread, shift, worst, e_fx, e_64 in rows:
        assert float(worst) <= 1.0, (n, sym, spread, shift, worst)
        if int(spread) <= 6:  # lines of the magnitudes a field has within an element
            assert float(e_fx) <= float(e_64), (n, sym, spread, shift, e_fx, e_64)
