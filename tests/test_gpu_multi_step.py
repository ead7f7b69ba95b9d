"""Several steps of a small lattice in one launch against single steps of the
same context type: bit for bit, for every kernel body, parity and count, at
lattices of one thread's work up to the resident limit, and beyond it."""
import numpy as np
import pytest

from gpu_helpers import turbulence

pytestmark = pytest.mark.gpu

B0 = np.array([0.0, 0.02, 0.05])


def _sim(shape, storage, variant, **kw):
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    sim = Flame(nx, ny, nz, 0.56, 0.6, 1.0, storage=storage, B_ref=tuple(B0), variant=variant, **kw)
    u, B = turbulence(shape, 81, 0.04)
    sim.init(None, u, B + B0[:, None, None, None])
    return sim


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 2), (3, 5, 33), (9, 7, 64), (32, 32, 32), (48, 50, 48), (49, 50, 48)])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("variant", ["flame", "bgk", "emhd"])
def test_many_steps_equal_single_steps(shape, storage, variant):
    import torch
    a, b = _sim(shape, storage, variant), _sim(shape, storage, variant)
    for n in (2, 7, 16):
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert torch.equal(a.state, b.state), n
        assert a.info()["step"] == b.info()["step"] and a.info()["parity"] == b.info()["parity"]
    assert a.sync() is None
    a.close()
    b.close()


def test_many_steps_with_checks_forced_kernel_and_capture():
    """check_every in the middle of a call, more steps than one launch takes,
    the one-site kernel forced on 16-bit storage, and a stream under capture."""
    import torch
    shape = (6, 10, 34)
    a, b = _sim(shape, "fp16", "flame", kernel="site", check_every=7), _sim(shape, "fp16", "flame", kernel="site")
    a.step(600)
    for _ in range(600):
        b.step(1)
    assert torch.equal(a.state, b.state) and a.info()["step"] == 600
    a.close()
    b.close()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        a, b = _sim(shape, "fp32", "flame"), _sim(shape, "fp32", "flame")
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            a.step(6)
        g.replay()
        b.step(6)
    s.synchronize()
    assert torch.equal(a.state, b.state)
    a.close()
    b.close()


def test_nonfinite_seen_by_many_steps():
    import torch
    from paper_2212_11024_gb300 import flame as F
    sim = _sim((4, 4, 4), "fp32", "flame")
    sim.state.view(torch.float32)[5] = float("nan")
    sim.step(4)
    with pytest.raises(F.FlameError) as e:
        sim.sync()
    assert e.value.status == F.FLAME_ERR_NONFINITE
    sim.close()
