"""The per-block flags of the coarse solve (csrc/coarse_flags.h) on the host: a block that polls late
finds its generation passed whatever its neighbours have published since, their last arrival
included, and no schedule leaves a block waiting."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_07663_gb300", "csrc")


def test_flags_and_schedules_on_the_host(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    exe = str(tmp_path / "coarse_flags_host")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, os.path.join(HERE, "coarse_flags_host.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, f"{r.returncode}: {r.stdout}"
