"""The index arithmetic of the 3 x 3 layers' tiles (gmmsp_grid3.cuh), checked on the host against 64-bit
divisions: small grids cell by cell, and every row length at the most rows that a network call accepts."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_tile_positions_match_divisions(tmp_path):
    exe = str(tmp_path / "grid3_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1612_08792_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "grid3_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr
