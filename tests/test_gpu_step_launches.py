"""Which kernels flame_step launches, by their names as the profiler records them:
a forced tiling runs whatever the number of steps; several steps of a small
lattice are one launch by the automatic choice."""
import numpy as np
import pytest
import torch

from gpu_helpers import turbulence

pytestmark = pytest.mark.gpu


def launched(fn):
    """Names of the kernels that fn() launches."""
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        fn()
        torch.cuda.synchronize()
    return [e.name for e in prof.events() if "kernel" in e.name]


def _sim(shape, storage, variant="flame", kernel="auto"):
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    sim = Flame(nx, ny, nz, 0.56, 0.6, 1.0, storage=storage, variant=variant, kernel=kernel)
    sim.init(None, *turbulence(shape, 81, 0.04))
    return sim


@pytest.fixture(autouse=True, scope="module")
def _profiler_records():
    x = torch.zeros(1024, device="cuda")
    launched(lambda: x.add_(1.0))  # its first use only starts it
    if not launched(lambda: x.add_(1.0)):
        pytest.skip("the profiler records no kernels here")


@pytest.mark.parametrize("variant", ["flame", "bgk", "emhd"])
@pytest.mark.parametrize("kernel,shape", [("row", (4, 3, 64)), ("row", (2, 2, 200)), ("row", (1, 2, 384)),
                                          ("row_half", (2, 3, 320)), ("row_half", (1, 2, 1024))])
def test_forced_staged_rows_run_at_every_number_of_steps(kernel, shape, variant):
    sim = _sim(shape, "fp16", variant, kernel)
    for n in (1, 2, 7):
        names = launched(lambda: sim.step(n))
        assert len(names) == n and all("step_row_kernel" in s for s in names), names
    sim.close()


@pytest.mark.parametrize("shape,storage,kernel,one,several", [
    ((4, 3, 64), "fp16", "auto", "step_row_kernel", "step_pairs_kernel"),
    ((2, 4, 250), "bf16", "auto", "step_window_kernel", "step_pairs_kernel"),
    ((4, 3, 64), "fp16", "pair", "step_pair_kernel", "step_pairs_kernel"),
    ((4, 3, 64), "fp16", "site", "step_kernel", "step_sites_kernel"),
    ((4, 3, 66), "fp16", "row", "step_kernel", "step_sites_kernel"),  # a tiling that does not apply
    ((4, 3, 64), "fp32", "auto", "step_kernel", "step_sites_kernel")])
def test_several_steps_of_a_small_lattice_are_one_launch(shape, storage, kernel, one, several):
    sim = _sim(shape, storage, kernel=kernel)
    names = launched(lambda: sim.step(1))
    assert len(names) == 1 and one in names[0], names
    names = launched(lambda: sim.step(7))
    assert len(names) == 1 and several in names[0], names
    sim.close()
