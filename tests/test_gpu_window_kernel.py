"""Rows of even lengths that are no multiple of 8, staged as aligned windows
(the automatic choice for 16-bit storage where a block's lanes are filled),
against the unstaged pair kernel, whose arithmetic is the same: bit for bit."""
import numpy as np
import pytest

from gpu_helpers import turbulence
from paper_2212_11024_gb300 import flame as F

B0 = np.array([0.0, 0.02, 0.05])
# (nz, ny, nx): two compile-time row lengths (staged by the same rule), then windows:
# N3 a multiple of 8 and not, compile-time and run-time pitches,
# single rows (windows at both ends of the state), partly filled last warps
SHAPES = [(2, 3, 192), (1, 2, 384), (1, 4, 182), (3, 1, 182), (4, 1, 190), (2, 3, 222), (2, 4, 250), (1, 1, 250),
          (3, 2, 254), (1, 2, 318), (3, 1, 446), (2, 1, 1022)]


def _run(shape, storage, variant, kernel, n, graph=0):
    import torch
    nz, ny, nx = shape
    u, B = turbulence(shape, 61, 0.05)
    sim = F.Flame(nx, ny, nz, 0.52, 0.55, 1.5, storage=storage, B_ref=tuple(B0), kernel=kernel, variant=variant,
                  graph_steps=graph)
    sim.init(None, u, B + B0[:, None, None, None])
    sim.step(n)
    sim.sync()
    blob = sim.get_state()[0]
    assert torch.isfinite(sim.moments()["u"]).all()
    return sim, blob


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("storage", ["fp16", "bf16"])
@pytest.mark.parametrize("variant", ["flame", "bgk", "emhd", "fd_current"])
def test_windows_equal_the_pair_kernel(shape, storage, variant):
    import torch
    a, x = _run(shape, storage, variant, "auto", 7)
    b, y = _run(shape, storage, variant, "pair", 7)
    assert torch.equal(x, y)
    # the windows' copies have waits to stall, the pair kernel has none; auto takes
    # the pairs too where lanes idle and the pitch is not fixed at compile time
    pairs = [b]
    if shape in ((3, 1, 182), (2, 3, 222)):
        pairs.append(a)
    else:
        a.debug_stall_next_step(64)
    for s in pairs:
        with pytest.raises(F.FlameError) as e:
            s.debug_stall_next_step(64)
        assert e.value.status == F.FLAME_ERR_PARAM
    a.close()
    b.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(3, 2, 250), (4, 2, 254)])
def test_windows_in_graphs_and_slabs(shape):
    """Graph replay, and the lattice split into slabs (whose states have other
    sizes, so other window alignments)."""
    import torch

    from paper_2212_11024_gb300.slab import SlabGroup
    nz, ny, nx = shape
    a, x = _run(shape, "fp16", "flame", "pair", 8)
    b, y = _run(shape, "fp16", "flame", "auto", 8, graph=4)
    assert torch.equal(x, y)
    u, B = turbulence(shape, 61, 0.05)
    grp = SlabGroup(nx, ny, nz, 2, 0.52, 0.55, 1.5, storage="fp16", B_ref=tuple(B0))
    grp.init(None, u, B + B0[:, None, None, None])
    grp.step(8)
    assert torch.equal(grp.populations(), a.populations())
    a.close()
    b.close()
    grp.close()


@pytest.mark.gpu
@pytest.mark.parametrize("nx", [174, 198, 258, 340, 514, 1026, 250])
def test_lengths_that_are_not_windows(nx):
    """Where the block's lanes would idle, and with the kernel forced."""
    sim = F.Flame(nx, 2, 2, 0.52, 0.55, 1.5, storage="fp16", kernel="pair" if nx == 250 else "auto")
    u, B = turbulence((2, 2, nx), 61, 0.05)
    sim.init(None, u, B)
    with pytest.raises(F.FlameError) as e:
        sim.debug_stall_next_step(64)
    assert e.value.status == F.FLAME_ERR_PARAM
    sim.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(2, 4, 250), (1, 2, 318)])
def test_windows_whose_waits_run_out(shape):
    """Barriers armed but never fed: the step reports a timeout and leaves the
    state as it was."""
    import torch
    sim, before = _run(shape, "fp16", "flame", "auto", 3)
    sim.debug_stall_next_step(256)
    with pytest.raises(F.FlameError) as e:
        sim.step(1)
    assert e.value.status == F.FLAME_ERR_TIMEOUT
    assert torch.equal(sim.state, before)
    sim.close()
