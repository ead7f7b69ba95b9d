"""flame_step_adjoint whose first call on a context is captured into a graph (in
relaxed mode, which lets it allocate): the calls that run before the graph does,
and the graph's replays, write the same dL/d(d_i)."""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(n, stream=None):
    from paper_2212_11024_gb300 import Flame
    g = torch.Generator(device="cuda").manual_seed(3)
    u, B = (0.03 * torch.randn((3, n, n, n), generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    lam = torch.randn((48, n, n, n), generator=g, device="cuda")
    sim = Flame(n, n, n, 0.6, 0.6, 1.0, stream=stream)
    sim.init(None, u, B)
    out = torch.empty_like(lam)

    def call(ddi):
        rc = sim._lib.flame_step_adjoint(sim._ctx, ctypes.c_void_p(sim.state.data_ptr()), 0, ctypes.c_void_p(lam.data_ptr()),
                                         ctypes.c_void_p(out.data_ptr()), ctypes.c_void_p(ddi.data_ptr()))
        assert rc == 0
    return sim, call


def _dirty_memory():
    """Device memory of the sizes of small workspaces, filled with ones and freed:
    what the next allocation finds is not zero."""
    try:
        rt = ctypes.CDLL("libcudart.so.13")
    except OSError:
        return
    ptrs = []
    for size in range(4096, 8192, 8):
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
        assert rt.cudaMemset(p, 255, ctypes.c_size_t(size)) == 0
        ptrs.append(p)
    torch.cuda.synchronize()
    for p in ptrs:
        assert rt.cudaFree(p) == 0


def test_first_call_captured():
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ddi = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(4)]
        sim, call = _run(24, s)
        call(ddi[0])
        s.synchronize()
        sim.close()
        sim, call = _run(24, s)
        s.synchronize()
        _dirty_memory()
        g = torch.cuda.CUDAGraph()
        g.capture_begin(capture_error_mode="relaxed")
        call(ddi[1])
        g.capture_end()
        call(ddi[2])
        g.replay()
        call(ddi[3])
        s.synchronize()
    assert float(ddi[0]) != 0.0 and len({float(d) for d in ddi}) == 1, [float(d) for d in ddi]
    sim.close()
