"""The step kernels launched one step at a time, which is how lattices beyond the
several-step launch's run: staged rows, half rows and windows of every kind against
the unstaged pair kernel, bit for bit, and chains of small launches against graph
replays.  The kernel that ran is checked by its name."""
import numpy as np
import pytest
import torch

from gpu_helpers import turbulence
from test_gpu_step_launches import launched

pytestmark = pytest.mark.gpu

B0 = np.array([0.0, 0.02, 0.05])


@pytest.fixture(scope="module")
def recorded():
    x = torch.zeros(1024, device="cuda")
    launched(lambda: x.add_(1.0))  # the profiler's first use only starts it
    return bool(launched(lambda: x.add_(1.0)))


def _sim(shape, storage, variant, kernel, **kw):
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    sim = Flame(nx, ny, nz, 0.52, 0.55, 1.5, storage=storage, B_ref=tuple(B0), kernel=kernel, variant=variant, **kw)
    u, B = turbulence(shape, 61, 0.05)
    sim.init(None, u, B + B0[:, None, None, None])
    return sim


def _equal_steps(shape, storage, variant, kernel, name, recorded):
    a, b = _sim(shape, storage, variant, kernel), _sim(shape, storage, variant, "pair")
    if recorded:
        names = launched(lambda: a.step(1))
        assert any(name in s for s in names), names
    else:
        a.step(1)
    b.step(1)
    for _ in range(6):
        assert torch.equal(a.state, b.state)
        a.step(1)
        b.step(1)
    assert torch.equal(a.state, b.state) and a.sync() is None
    assert torch.isfinite(a.moments()["u"]).all()
    a.close()
    b.close()


# (nz, ny, nx): pitch 216, pitch 280 (a full and a hardly filled last warp), pitches
# read from the grid (N3 no multiple of 8, and rows beyond 256 sites)
WINDOWS = [(4, 1, 190), (2, 4, 222), (2, 4, 250), (4, 2, 254), (3, 1, 254), (1, 2, 318), (3, 1, 446), (2, 1, 1022)]


@pytest.mark.parametrize("shape", WINDOWS)
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("variant", ["flame", "bgk", "emhd"])
def test_windows(shape, storage, variant, recorded):
    _equal_steps(shape, storage, variant, "auto", "step_window_kernel", recorded)


# compile-time lengths 64, 128, 192, 256, 384, 512; the general ones with three
# stages and two, partly filled last warps among them
ROWS = [(3, 2, 64), (2, 2, 128), (2, 3, 192), (2, 2, 256), (1, 3, 384), (2, 1, 512), (2, 2, 72), (2, 1, 136),
        (1, 3, 200), (1, 2, 328), (2, 1, 456), (2, 1, 960), (1, 1, 1000), (1, 2, 1024)]


@pytest.mark.parametrize("shape", ROWS)
@pytest.mark.parametrize("storage,variant", [("fp16", "flame"), ("bf16", "flame"), ("fp16", "bgk"), ("bf16", "emhd")])
def test_whole_rows(shape, storage, variant, recorded):
    _equal_steps(shape, storage, variant, "row", "step_row_kernel", recorded)


@pytest.mark.parametrize("shape", [(2, 2, 320), (2, 1, 512), (1, 2, 608), (2, 1, 1024), (1, 2, 400)])
@pytest.mark.parametrize("storage,variant", [("fp16", "flame"), ("bf16", "flame"), ("fp16", "bgk"), ("bf16", "emhd")])
def test_half_rows(shape, storage, variant, recorded):
    _equal_steps(shape, storage, variant, "row_half", "step_row_kernel", recorded)


@pytest.mark.parametrize("shape,storage,variant,kernel", [
    ((6, 5, 64), "fp32", "flame", "site"), ((41, 40, 33), "fp32", "bgk", "auto"), ((7, 8, 129), "fp16", "emhd", "auto"),
    ((33, 32, 64), "fp16", "flame", "auto"), ((31, 5, 250), "bf16", "flame", "auto"), ((9, 8, 100), "fp16", "bgk", "pair")])
@pytest.mark.parametrize("own_stream", [False, True])
def test_chains_of_small_launches(shape, storage, variant, kernel, own_stream):
    s = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    with torch.cuda.stream(s):
        a = _sim(shape, storage, variant, kernel, stream=s)
        for _ in range(40):
            a.step(1)
        a.sync()
    b = _sim(shape, storage, variant, kernel, graph_steps=20)
    b.step(40)
    assert b.sync() is None and torch.equal(a.state, b.state)
    a.close()
    b.close()
