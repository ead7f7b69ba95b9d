"""flame_step_between against flame_step: the same arithmetic into another
buffer, so every state is the same bits, and the buffer it reads is unchanged."""
import numpy as np
import pytest
import torch

from paper_2212_11024_gb300 import Flame
from paper_2212_11024_gb300.flame import FlameError

pytestmark = pytest.mark.gpu


def _sim(shape, storage, **kw):
    rng = np.random.default_rng(5)
    nx, ny, nz = shape
    u, B = (0.03 * rng.standard_normal((3, nz, ny, nx)) for _ in range(2))
    s = Flame(nx, ny, nz, 0.6, 0.6, 1.0, storage=storage, **kw)
    s.init(None, u, B)
    return s


# row blocks, flat blocks, a single row of sites, the packed kernels' lengths
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("shape", [(64, 12, 9), (33, 7, 5), (257, 3, 2), (16, 1, 1), (250, 5, 4), (128, 6, 7)])
def test_states_equal_steps_in_place(shape, storage):
    a, b = _sim(shape, storage), _sim(shape, storage)
    blob, step, par = b.get_state()
    for t in range(5):
        before = blob.clone()
        after = torch.empty_like(blob) if t < 4 else b.state
        b.step_between(blob, after)
        assert torch.equal(blob, before)
        a.step(1)
        assert torch.equal(after, a.get_state()[0])
        blob = after
    assert b.info()["step"] == a.info()["step"] and b.get_state()[2] == a.get_state()[2]
    assert torch.equal(a.moments()["u"], b.moments()["u"])
    a.close(), b.close()


def test_refused_calls():
    s = _sim((32, 8, 8), "fp32")
    one = torch.empty_like(s.state)
    with pytest.raises(FlameError):
        s.step_between(one, one)
    with pytest.raises(ValueError):
        s.step_between(s.state, one[:-256])
    s.close()
    s = _sim((32, 8, 8), "fp32", variant="emhd")
    with pytest.raises(FlameError):
        s.step_between(s.state, one)
    s.close()
