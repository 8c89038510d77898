"""Which driver the automatic solve takes on a GPU of 152 SMs (the plans of
persist_plan.h, computed by tests/host/plan_report.cpp): the persistent solve
for scenes that stay on the chip and in L2, passes in rounds beyond, a block
per group where a haloed row of the grid is too long for either."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_16037_gb300", "csrc")

P, R, S = "persistent", "rounds", "passes"
# shape, radius: K in FP32 and FP64, K^T in FP32 and FP64
EXPECTED = {
    (5, 5, 1, 1): (P, P, P, P), (8, 8, 8, 1): (P, P, P, P), (16, 16, 16, 2): (P, P, P, P),
    (21, 19, 9, 2): (P, P, P, P), (45, 37, 29, 2): (P, P, P, P), (48, 48, 32, 2): (P, P, P, P),
    (64, 64, 32, 2): (P, P, P, P), (130, 61, 12, 2): (P, P, P, P),
    (96, 96, 32, 2): (P, S, P, S), (104, 104, 34, 2): (P, S, R, S), (130, 125, 36, 2): (R, S, R, S), (128, 128, 40, 2): (R, S, R, S),
    (512, 8, 40, 2): (S, S, S, S), (1000, 10, 32, 2): (S, S, S, S),
}


def test_drivers_of_the_automatic_solve(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = str(tmp_path / "plan_report")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "host", "plan_report.cpp"),
                    os.path.join(CSRC, "graph.cpp"), os.path.join(CSRC, "persist_plan.cpp"), "-o", exe], check=True)
    args = [str(v) for shape in EXPECTED for v in shape]
    out = subprocess.run([exe] + args, capture_output=True, text=True, timeout=300, check=True).stdout
    got = {}
    for line in out.splitlines():
        head, tail = line.split(":")
        dims, radius = head.split(" R")
        got[tuple(int(v) for v in dims.split("x")) + (int(radius),)] = tuple(w.split("=")[1] for w in tail.split())
    assert got == EXPECTED
