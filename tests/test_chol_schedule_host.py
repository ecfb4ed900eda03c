"""The launch order of the tile Cholesky on a stream and its side stream (paper_1208_6387_gb300/csrc/chol_schedule.cuh),
compiled for the host with g++: no access to a tile may overtake an earlier conflicting one, also where a tile column is
empty below its diagonal (pinned or decoupled dofs); no GPU needed."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1208_6387_gb300", "csrc")


def test_no_tile_access_overtakes_another(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "chol_schedule")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(HERE, "host", "chol_schedule.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
