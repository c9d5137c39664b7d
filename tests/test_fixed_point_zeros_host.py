"""Zeros of either sign, and values that their scale shifts out, have zero limbs and contract to exactly
zero (csrc/fxp.h, compiled as plain C++): an element of zeros gives zeros."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_07663_gb300", "csrc")


def test_zeros_contract_to_zero(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "fixed_point_zeros_host")
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-I", CSRC,
                    os.path.join(HERE, "fixed_point_zeros_host.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
