"""The initial populations of FP32 storage hold what FP64 holds of them where FP32
pairs would not: small deviations from a mean field, values left by cancellation;
and the speed of fields whose squares FP32 lacks."""
import numpy as np
import pytest

from test_gpu_diag64 import EPS, _slots

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _exact(u, B, Bref, omega, omegaB, d_i, gradB=None):
    """(stored values [48, ...] in extended precision of FP64 fields and their FP64
    differences, the sums of their terms' magnitudes)."""
    def diffs(f):
        return np.stack([0.5 * (np.roll(f, -1, 3 - a) - np.roll(f, 1, 3 - a)) for a in range(3)])
    du = diffs(u).astype(LD)  # [a, b]: d_a u_b
    dB = (gradB.reshape((3, 3) + u.shape[1:]) if gradB is not None else diffs(B)).astype(LD)
    u, B, r = u.astype(LD), B.astype(LD), np.asarray(Bref, dtype=np.float32).astype(LD)
    b = (B - r[:, None, None, None]).astype(np.float64).astype(LD)
    J = np.stack([dB[1, 2] - dB[2, 1], dB[2, 0] - dB[0, 2], dB[0, 1] - dB[1, 0]])
    V, mV = u - d_i * J, np.abs(u) + d_i * np.abs(dB).sum((0, 1))
    N = np.stack([np.stack([r[a] * b[c] + b[a] * r[c] + b[a] * b[c] for c in range(3)]) for a in range(3)])
    P = -(du + du.transpose(1, 0, 2, 3, 4)) / (3 * LD(omega))
    miso = sum(r[a] * b[a] + b[a] * b[a] / 2 for a in range(3))
    trN, trP = (N[0, 0] + N[1, 1] + N[2, 2]) / 3, (P[0, 0] + P[1, 1] + P[2, 2]) / 3
    out, mag = np.empty((48,) + u.shape[1:], LD), np.empty((48,) + u.shape[1:], LD)
    mfl = 18 * (np.abs(b) * (np.abs(B) + np.abs(r)[:, None, None, None])).sum(0) + 9 * np.abs(P).sum((0, 1))
    for slot, c, w, _ in _slots():
        if slot < 27:
            E, mE = LD(1), LD(1)
            for a in range(3):
                E = E * (1 + (-1.5 * u[a] ** 2 if c[a] == 0 else 3 * u[a] ** 2 + 3 * c[a] * u[a]))
                mE = mE * (1 + 3 * u[a] ** 2 + 3 * np.abs(u[a]))
            cNc = sum(int(c[a] * c[e]) * N[a, e] for a in range(3) for e in range(3))
            cPc = sum(int(c[a] * c[e]) * P[a, e] for a in range(3) for e in range(3))
            c2 = int((np.asarray(c) ** 2).sum())
            out[slot] = (E - 1) + 4.5 * (miso * (c2 - 1) - cNc + trN) + 4.5 * (cPc - trP)
            mag[slot] = (mE - 1) + mfl
        else:
            i, k = divmod(slot - 27, 3)
            out[slot], mag[slot] = b[k], np.abs(b[k])
            for a in range(3):
                if c[a]:
                    out[slot] = out[slot] + int(c[a]) * (4 * (V[a] * B[k] - B[a] * V[k]) - dB[a, k] / LD(omegaB))
                    mag[slot] = mag[slot] + np.abs(dB[a, k]) / omegaB
                    if a != k:
                        mag[slot] = mag[slot] + 4 * (mV[a] * np.abs(B[k]) + np.abs(B[a]) * mV[k])
    return out, mag


def _init(u, B, Bref, tau, d_i, gradB=None):
    import torch
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = u.shape[1:]
    sim = Flame(nx, ny, nz, tau, tau, d_i, storage="fp32", B_ref=Bref)
    gradu = None if gradB is None else np.zeros_like(gradB)
    sim.init(None, u, B, gradu, gradB)
    got = sim.state.view(torch.float32).cpu().numpy().reshape((48,) + u.shape[1:]).astype(LD)
    speed = sim.info()["max_speed"]
    sim.close()
    return got, speed


@pytest.mark.parametrize("amp", [1e-9, 1e-6, 0.03])
def test_small_deviations_from_a_mean_field(amp):
    """Half a unit of the stored value's last place, and FP64's 16 roundings of its
    terms -- deviations and differences, not the mean field they are taken from."""
    r = np.random.default_rng(31)
    shape, Bref, tau, d_i = (6, 7, 65), (0.0, 0.03, 0.1), 0.625, 1.5
    u = amp * r.standard_normal((3,) + shape)
    B = amp * r.standard_normal((3,) + shape) + np.array(Bref, np.float32).astype(float)[:, None, None, None]
    got, _ = _init(u, B, Bref, tau, d_i)
    om = float(np.float32(1 / tau))
    ref, mag = _exact(u, B, Bref, om, om, d_i)
    tol = 0.5 * np.spacing(np.abs(ref).astype(np.float32)).astype(LD) + 16 * EPS * mag
    off = np.abs(got - ref) / tol
    assert (off <= 1).all(), (float(off.max()), int((off > 1).sum()))


def test_values_left_by_cancellation():
    """d_a B_b / omega_B within 1e-9 of b_b, no flow and no Hall term: of the magnetic
    populations of one direction a 1e-9th of their terms is left, to three roundings
    (b, the quotient, the sum)."""
    r = np.random.default_rng(32)
    shape, tau = (5, 6, 65), 0.625
    om = float(np.float32(1 / tau))
    B = 0.05 * r.standard_normal((3,) + shape)
    gB = np.stack([B * om * (1 + 1e-9 * r.standard_normal(B.shape)) for _ in range(3)]).reshape((9,) + shape)
    u = np.zeros_like(B)
    got, _ = _init(u, B, (0.0, 0.0, 0.0), tau, 0.0, gB)
    ref, mag = _exact(u, B, (0.0, 0.0, 0.0), om, om, 0.0, gB)
    tol = 0.5 * np.spacing(np.abs(ref).astype(np.float32)).astype(LD) + 3 * EPS * mag
    off = (np.abs(got - ref) / tol)[27:]
    assert (off <= 1).all(), (float(off.max()), int((off > 1).sum()))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("amp", [1e-15, 1e-21, 1e-30, 1e-37])
def test_speed_of_tiny_fields(amp, dtype):
    """max(|u|, |B|) rounded to FP32 (half a unit of it, and two-term arithmetic)."""
    r = np.random.default_rng(33)
    shape = (3, 4, 33)
    for ku, kB in ((1.0, 0.5), (0.5, 1.0)):
        u = (ku * amp * r.standard_normal((3,) + shape)).astype(dtype)
        B = (kB * amp * r.standard_normal((3,) + shape)).astype(dtype)
        _, speed = _init(u, B, (0.0, 0.0, 0.0), 0.625, 1.5)
        top = max(np.sqrt((f.astype(LD) ** 2).sum(0)).max() for f in (u, B))
        assert abs(LD(speed) - top) <= 0.51 * np.spacing(np.float32(top))
