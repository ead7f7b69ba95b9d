"""flame_step_adjoint against FP64 autograd at the edges of its blocks, for every
storage and parity, with lambda aligned and not."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_helpers import turbulence
from oracle import torch_ref as R

pytestmark = pytest.mark.gpu

# (nz, ny, nx): blocks of one row and of two, partly filled last blocks; a row that
# is its own neighbour in y and z; more partial sums than one block adds
SHAPES = [(2, 3, 7), (3, 5, 32), (1, 1, 40), (2, 3, 64), (3, 2, 65), (2, 3, 129), (40, 33, 34)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("parity", [0, 1])
def test_step_adjoint_matches_autograd(shape, storage, parity):
    """lambda_t to 1e-5 of its largest component, and the same bits and
    dL/d(d_i) whatever lambda's alignment, and on a second call."""
    from paper_2212_11024_gb300 import Flame
    from paper_2212_11024_gb300.flame import library
    nz, ny, nx = shape
    u, B = turbulence(shape, 13, 0.05)
    B[2] += 0.05
    sim = Flame(nx, ny, nz, 0.57, 0.62, 1.3, storage=storage, B_ref=(0, 0, 0.05))
    sim.init(None, u, B)
    sim.step(2 + parity)
    blob, _, par = sim.get_state()
    pop = sim.populations().cpu().numpy()
    n3 = nx * ny * nz
    lam = np.random.default_rng(3).standard_normal((48, n3)).astype(np.float32)
    buf = torch.zeros(48 * n3 + 1, dtype=torch.float32, device="cuda")
    res = []
    for off in (0, 1, 0):
        lin = buf[off:off + 48 * n3]
        lin.copy_(torch.from_numpy(lam.reshape(-1)))
        lout = torch.full((48, n3), float("nan"), dtype=torch.float32, device="cuda")
        ddi = torch.zeros(1, dtype=torch.float64, device="cuda")
        rc = library().flame_step_adjoint(sim._ctx, ctypes.c_void_p(blob.data_ptr()), par,
                                          ctypes.c_void_p(lin.data_ptr()), ctypes.c_void_p(lout.data_ptr()),
                                          ctypes.c_void_p(ddi.data_ptr()))
        assert rc == 0
        torch.cuda.synchronize()
        res.append((lout.cpu().numpy().reshape((48,) + shape), float(ddi[0])))
    sim.close()
    x = torch.tensor(pop, requires_grad=True)
    d = torch.tensor(1.3, dtype=torch.float64, requires_grad=True)
    ref, gd = torch.autograd.grad((R.step(x, 0.57, 0.62, d, 1) * torch.tensor(lam.reshape((48,) + shape), dtype=torch.float64)).sum(), [x, d])
    ref = ref.numpy()
    top = np.abs(ref).max()
    out, d0 = res[0]
    assert np.abs(out - ref).max() < 1e-5 * top
    assert all(np.array_equal(out, o) and d0 == d1 for o, d1 in res[1:])
    # the d_i terms are of the order of lambda times the fields' ~0.1
    assert abs(d0 - float(gd)) < 1e-5 * abs(float(gd)) + 3e-6 * np.sqrt(n3)
