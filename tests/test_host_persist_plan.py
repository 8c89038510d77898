"""Host check of the persistent solve's division of the grid: block runs, tile
chunks and every gather index (tests/host/persist_checks.cpp, built here with
the host compiler)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_16037_gb300", "csrc")


def test_persistent_solve_indices(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "persist_checks")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "host", "persist_checks.cpp"),
                    os.path.join(CSRC, "graph.cpp"), os.path.join(CSRC, "persist_plan.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
    assert "64x64x32 R2 K 4 bytes: planned" in out.stdout
