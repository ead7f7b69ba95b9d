"""The conversions between FP64 and FP32 expansions (expansion.cuh), compiled with
the host compiler and compared with FP64 arithmetic (expansion_check.cpp); no GPU
needed."""
import os
import shutil
import subprocess
from pathlib import Path

import pytest

HERE = Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2212_11024_gb300" / "csrc"


def test_conversions_round_to_nearest(tmp_path):
    cxx = shutil.which("g++")
    inc = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda")) / "include"
    if cxx is None or not (inc / "cuda_runtime.h").exists():
        pytest.skip("needs g++ and the CUDA headers")
    exe = tmp_path / "expansion_check"
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", f"-I{inc}", f"-I{CSRC}",
                    str(HERE / "expansion_check.cpp"), "-o", str(exe)], check=True, capture_output=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
