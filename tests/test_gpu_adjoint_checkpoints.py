"""The differentiable run's two ways of keeping its forward states -- all of
them, or sqrt(N) checkpoints with replay -- give the same gradients, bit for
bit."""
import pytest

from gpu_helpers import turbulence

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,nsteps", [("fp32", 1), ("fp32", 7), ("fp32", 12), ("fp16", 10)])
def test_kept_and_replayed_states_agree(storage, nsteps, monkeypatch):
    import torch
    from paper_2212_11024_gb300 import adjoint as A
    u, B = turbulence((6, 8, 10), 23, 0.04)
    B[2] += 0.03
    got = []
    for share in (1.0, 0.0):
        monkeypatch.setattr(A, "KEEP_ALL", share)
        got.append(A.band_energy_gradient(u, B, 1.5, 0.6, 0.65, nsteps, (1, 2), storage=storage))
    a, b = got
    assert a[3] == b[3]  # (the loss itself is summed by atomics, in no fixed order, before any of this)
    assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
