"""A context whose stream has only some of the device's SMs: lattices that take
several steps in one launch on the whole device do not fit there, and are stepped
launch by launch."""
import ctypes
import os
import shutil
import subprocess
from pathlib import Path

import pytest
import torch

from gpu_helpers import turbulence

pytestmark = pytest.mark.gpu

HERE = Path(__file__).resolve().parent


@pytest.fixture(scope="module")
def part(tmp_path_factory):
    cuda = Path(os.environ.get("CUDA_HOME", "/usr/local/cuda"))
    so = tmp_path_factory.mktemp("green") / "green_stream.so"
    if shutil.which("g++") is None or not (cuda / "include" / "cuda.h").exists():
        pytest.skip("needs g++ and the CUDA headers")
    subprocess.run(["g++", "-shared", "-fPIC", "-std=c++17", f"-I{cuda / 'include'}", str(HERE / "green_stream.cpp"),
                    f"-L{cuda / 'lib64' / 'stubs'}", "-lcuda", "-o", str(so)], check=True, capture_output=True,
                   timeout=120)
    torch.zeros(1, device="cuda")
    lib, p = ctypes.CDLL(str(so)), ctypes.c_void_p()
    sms = lib.green_stream(16, ctypes.byref(p))
    if not 0 < sms <= 32:
        pytest.skip("no stream of a part of the SMs to be had")
    return torch.cuda.ExternalStream(p.value)


@pytest.mark.parametrize("shape,storage", [((32, 32, 32), "fp32"), ((40, 40, 40), "fp16"), ((4, 5, 33), "fp32")])
def test_several_steps_on_a_part_of_the_sms(part, shape, storage):
    """32^3 and 40^3 need more resident threads than 32 SMs hold, 4 x 5 x 33 not."""
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    u, B = turbulence(shape, 81, 0.04)
    states = []
    for stream in (None, part):
        sim = Flame(nx, ny, nz, 0.56, 0.6, 1.0, storage=storage, stream=stream)
        sim.init(None, u, B)
        sim.step(7)
        sim.step(4)
        sim.sync()
        states.append(sim.get_state()[0].cpu())
        assert sim.info()["step"] == 11
        sim.close()
    assert torch.equal(*states)
