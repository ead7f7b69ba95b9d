"""Steps launched one by one on a stream, each kernel brought to the SMs while
the one before it still ends, against the same steps as graph replays, whose
kernels start one after the other: the same kernels on the same state, so the
results are the same bits."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2212_11024_gb300 import Flame

pytestmark = pytest.mark.gpu


def _run(shape, storage, variant, graph_steps, kernel="auto", stream=None):
    rng = np.random.default_rng(9)
    nx, ny, nz = shape
    u, B = (0.03 * rng.standard_normal((3, nz, ny, nx)) for _ in range(2))
    s = Flame(nx, ny, nz, 0.6, 0.6, 1.0, storage=storage, variant=variant, graph_steps=graph_steps, kernel=kernel,
              stream=stream)
    s.init(None, u, B)
    s.step(40)
    out = [v.cpu().numpy() for v in s.moments().values()]
    s.close()
    return out


# one-site kernel in row blocks and flat blocks, row kernel (whole rows, halves,
# x windows), window kernel, pair kernel; grids of less than a wave and of many
@pytest.mark.parametrize("shape,storage,variant,kernel", [
    ((64, 5, 6), "fp32", "flame", "site"), ((129, 63, 65), "fp16", "flame", "auto"),
    ((128, 96, 96), "fp32", "flame", "auto"), ((33, 40, 41), "fp32", "bgk", "auto"),
    ((64, 32, 33), "fp16", "flame", "row"), ((256, 48, 40), "bf16", "emhd", "auto"),
    ((512, 24, 20), "fp16", "flame", "auto"), ((250, 30, 31), "bf16", "flame", "auto"),
    ((64, 64, 64), "fp16", "flame", "pair"), ((64, 40, 40), "fp16", "fd_current", "auto")])
def test_chained_steps_equal_graph_steps(shape, storage, variant, kernel):
    for a, b in zip(_run(shape, storage, variant, 0, kernel), _run(shape, storage, variant, 20, kernel)):
        assert np.array_equal(a, b)


def test_chain_on_a_stream_of_the_caller():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a = _run((96, 40, 40), "fp16", "flame", 0, stream=s)
    b = _run((96, 40, 40), "fp16", "flame", 20)
    assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("shape,storage", [((64, 64, 64), "fp32"), ((33, 20, 21), "fp16"), ((16, 4, 4), "bf16"),
                                           ((128, 64, 96), "fp16")])
def test_chained_adjoint_steps_equal_single_ones(shape, storage):
    nx, ny, nz = shape
    g = torch.Generator(device="cuda").manual_seed(3)
    u, B = (0.03 * torch.randn((3, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    lam0 = torch.randn((48, nz, ny, nx), generator=g, device="cuda")
    s = Flame(nx, ny, nz, 0.6, 0.6, 1.0, storage=storage)
    s.init(None, u, B)
    states = []
    for _ in range(4):
        states.append(s.get_state())
        s.step(1)

    def sweep(sync):
        lam, out = lam0.clone(), torch.empty_like(lam0)
        ddi = torch.zeros(12, dtype=torch.float64, device="cuda")
        for i in range(12):
            blob, _, par = states[3 - i % 4]
            rc = s._lib.flame_step_adjoint(s._ctx, ctypes.c_void_p(blob.data_ptr()), par,
                                           ctypes.c_void_p(lam.data_ptr()), ctypes.c_void_p(out.data_ptr()),
                                           ctypes.c_void_p(ddi.data_ptr() + 8 * i))
            assert rc == 0
            if sync:
                torch.cuda.synchronize()
            lam, out = out, lam
        torch.cuda.synchronize()
        return lam, ddi

    a, b = sweep(False), sweep(True)
    assert torch.isfinite(a[0]).all() and torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    s.close()
