"""Host checks of the serving loop's batcher of solves (tests/host/batch_checks.cpp,
built here with the host compiler against a stand-in for the CUDA runtime)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_16037_gb300", "csrc")
CUDA = next((d for d in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
             if os.path.exists(os.path.join(d, "include", "cuda_runtime.h"))), None)


def test_which_solves_are_batched_and_when(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or CUDA is None:
        pytest.skip("no host C++ compiler or no CUDA headers")
    exe = str(tmp_path / "batch_checks")
    src = [os.path.join(ROOT, "tests", "host", "batch_checks.cpp")] + [os.path.join(CSRC, f) for f in (
        "batch.cu", "persist_plan.cpp", "graph.cpp")]
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(CUDA, "include"), "-x", "c++"] + src + ["-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
