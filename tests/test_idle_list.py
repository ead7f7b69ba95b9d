"""The list of idle FFT plans (idle_list.h), compiled with the host compiler and run
against an account of what is alive (idle_list_check.cpp); and that the plans' pool
keeps them by it.  No GPU needed."""
import shutil
import subprocess
from pathlib import Path

import pytest

HERE = Path(__file__).resolve().parent
CSRC = HERE.parent / "paper_2212_11024_gb300" / "csrc"


def test_idle_objects_are_bounded_and_none_is_lost(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    exe = tmp_path / "idle_list_check"
    subprocess.run([cxx, "-O1", "-std=c++17", f"-I{CSRC}", str(HERE / "idle_list_check.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, timeout=120)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout


def test_the_pool_destroys_what_the_list_drops():
    code = (CSRC / "plans.cu").read_text()
    give = code[code.index("void plan_give("):]
    assert "drop = p.idle.give(" in give and "if (drop) cufftDestroy(old);" in give
