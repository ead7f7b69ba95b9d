"""The scalar reductions hold FP64: a site's terms, and a thread's sums over many
sites, to units of FP64 rounding.  Single sites and rows that give every thread
the same numbers, so that no rounding averages out."""
import numpy as np
import pytest
import torch

from test_gpu_diag64 import EPS, _pre_collision, _slots, _sums

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [0.05, 1e-33])
def test_terms_of_one_site_of_fp32_storage(scale):
    """One site is its own sum: every raw sum within 16 roundings of the magnitude
    of its terms (the velocity 3, a square twice its factors' and 3 more, the
    scaled sums 2), for ordinary fields and for ones whose squares FP32 lacks."""
    from paper_2212_11024_gb300 import Flame
    Bref, shape, f = (0.0, 0.03, 0.1), (1, 1, 1), np.float32
    sim = Flame(1, 1, 1, 0.625, 0.625, 1.5, storage="fp32", B_ref=Bref)
    for seed in range(64):
        blob = (scale * np.random.default_rng(seed).standard_normal((48,) + shape)).astype(f)
        sim.set_state(torch.from_numpy(blob.reshape(-1).view(np.uint8).copy()).cuda(), 0, 0)
        got = sim.reduce_sums()
        ref, mag = _sums(_pre_collision(blob, 0), float(f(1 / 0.625)), 1.5, [float(f(b)) for b in Bref])
        off = np.abs(got - ref)
        assert (off <= 16 * EPS * mag).all(), (seed, (off / (EPS * mag + 1e-300)).astype(float).round(1).tolist())
    sim.close()


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
def test_sums_of_one_block_over_many_sites(storage):
    """One block, each of whose threads sums the same 4096 sites, all moving the same
    way: the momentum is the exact sum of the sites' terms but for 10 roundings (a
    thread's sum to FP64, seven additions of equal numbers, the rest density's
    share)."""
    from paper_2212_11024_gb300 import Flame
    nx, ny, nz = 256, 64, 64
    dt = torch.float16 if storage == "fp16" else torch.bfloat16
    sim = Flame(nx, ny, nz, 0.625, 0.625, 1.5, storage=storage)
    v = 0.05 * torch.rand((48, nz, ny, 1), generator=torch.Generator().manual_seed(5))
    for slot, c, _, _ in _slots():
        v[slot] *= float(np.prod(1.0 + 0.7 * c))
    v = v.to(dt)
    sim.set_state(v.expand(48, nz, ny, nx).contiguous().reshape(-1).view(torch.uint8).cuda(), 0, 0)
    got = sim.reduce_static(nblocks=1).cpu().numpy()
    m = {k: x.cpu().numpy()[..., 0].astype(np.longdouble) for k, x in sim.moments().items()}
    sim.close()
    for a in range(3):
        t = m["rho"] * m["u"][a]
        assert abs(got[1 + a] - nx * t.sum()) <= 10 * EPS * nx * np.abs(t).sum(), a


def test_momentum_of_tiny_velocities():
    """BF16 storage holds velocities down to FP32's smallest numbers beside ordinary
    densities: their momentum, one site's, is rho u to three roundings."""
    from paper_2212_11024_gb300 import Flame
    rest = next(slot for slot, c, _, _ in _slots() if slot < 27 and not np.any(c))
    sim = Flame(1, 1, 1, 0.625, 0.625, 1.5, storage="bf16")
    g = torch.Generator().manual_seed(6)
    for amp in (1e-20, 1e-30, 1e-36):
        v = amp * torch.randn(48, generator=g)
        v[rest] = 0.37
        sim.set_state(v.to(torch.bfloat16).view(torch.uint8).cuda(), 0, 0)
        got = sim.reduce_sums()
        m = {k: x.cpu().numpy().astype(np.longdouble).reshape(-1) for k, x in sim.moments().items()}
        for a in range(3):
            t = m["rho"][0] * m["u"][a]
            assert abs(got[1 + a] - t) <= 3 * EPS * abs(t), (amp, a)
    sim.close()
