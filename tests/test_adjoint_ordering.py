"""The backward sweep of a differentiable run is queued on the run's stream after
what torch's current stream has queued for it (the seed's copy, the zeroed sums):
the order of the calls, on the CPU, and gradients from another, busy stream."""
import numpy as np
import pytest
import torch

from paper_2212_11024_gb300 import adjoint as A


def test_the_sweep_waits_for_torchs_stream(monkeypatch):
    calls = []

    class Lib:
        def __getattr__(self, name):
            return lambda *a: calls.append(name) or 0

    class Sim:
        device, _ctx = torch.device("cpu"), None

        def _before(self):
            calls.append("before")

        def __getattr__(self, name):
            return lambda *a: calls.append(name)

    monkeypatch.setattr(A, "library", Lib)
    for name in ("zeros", "empty"):
        fn = getattr(torch, name)
        monkeypatch.setattr(A.torch, name, lambda *a, fn=fn, name=name, **k: calls.append(name) or fn(*a, **k))
    run = A._Run.__new__(A._Run)
    run.sim, run.shape, run.k, run.nsteps = Sim(), (2, 2, 2), 1, 2
    run.ckpt = {t: (torch.zeros(4), t, t & 1) for t in range(2)}
    calls.clear()
    f = torch.zeros(3, 2, 2, 2, dtype=torch.float64)
    run.backward(f, f, torch.zeros(48, 8))
    lib = [i for i, c in enumerate(calls) if c.startswith("flame_")]
    assert [calls[i] for i in lib] == ["flame_step_adjoint"] * 2 + ["flame_init_adjoint"]
    for i in lib:
        before = max([j for j in range(i) if calls[j] == "before"], default=-1)
        wrote = max(j for j in range(i) if calls[j] in ("zeros", "empty"))
        assert before > wrote, calls


@pytest.mark.gpu
@pytest.mark.parametrize("keep", [1.0, 0.0])
def test_gradients_from_a_busy_stream(keep, monkeypatch):
    from gpu_helpers import turbulence
    monkeypatch.setattr(A, "KEEP_ALL", keep)
    shape, n = (6, 8, 34), 7
    u, B = (torch.tensor(f, device="cuda") for f in turbulence(shape, 23, 0.04))
    got = []
    for other in (False, True):
        run = A._Run(shape, 0.6, 0.65, 1.5, "fp32", (0.0, 0.0, 0.0), u.device)
        _, seed = run.forward(u, B, n, (1, 2))
        torch.cuda.synchronize()
        s = torch.cuda.Stream() if other else torch.cuda.current_stream()
        with torch.cuda.stream(s):
            if other:
                torch.cuda._sleep(200_000_000)  # what the sweep's buffers come after
            got.append([t.cpu().numpy() for t in run.backward(u, B, seed)])
        torch.cuda.synchronize()
        run.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)
