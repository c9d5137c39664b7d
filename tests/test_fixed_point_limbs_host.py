"""The limbs of values that are not folded (csrc/fxp.h, compiled as plain C++): a low limb of at most 2^27
of either sign, so that the products a contraction leaves out stay small, and nothing else changed."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_07663_gb300", "csrc")


def test_low_limbs_of_both_signs(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "fixed_point_limbs_host")
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC,
                    os.path.join(HERE, "fixed_point_limbs_host.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
