"""FP64 diagnostics of FP32 storage (moments and reductions), whose sums run
in FP32 expansions, against extended-precision sums of the same stored
values, at the edges of a warp and a block, for zero, tiny, ordinary and
overflowing values and for both AA parities."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53
C27, W27, XI7, W7 = (np.asarray(v) for v in O.lattice())


def _slots():
    """(storage slot, velocity, weight, opposite's storage slot) per natural slot (flame.h)."""
    fl = [int((c[0] + 1) + 3 * (c[1] + 1) + 9 * (c[2] + 1)) for c in C27]
    out = [(fl[q], C27[q], W27[q], 26 - fl[q]) for q in range(27)]
    opp = [0, 2, 1, 4, 3, 6, 5]
    return out + [(27 + 3 * i + b, XI7[i], W7[i], 27 + 3 * opp[i] + b) for b in range(3) for i in range(7)]


def _blob(shape, scale, seed):
    g = np.random.default_rng(seed).standard_normal((48,) + shape)
    return (scale * g).astype(np.float32)


def _pre_collision(blob, parity):
    s = np.empty(blob.shape, dtype=np.longdouble)
    for q, (slot, c, _, opp) in enumerate(_slots()):
        src = blob[slot] if parity == 0 else np.roll(blob[opp], (int(c[2]), int(c[1]), int(c[0])), (0, 1, 2))
        s[q] = src
    return s


def _reference(s, omB, aH, Bref):
    """(moments, their rounding scales) in extended precision."""
    w = np.array([v[2] for v in _slots()], dtype=np.longdouble)[:, None, None, None]
    t = w * s
    a = np.abs(t)
    drho = t[:27].sum(0)
    rho = 1 + drho
    j = np.stack([(C27[:, k, None, None, None] * t[:27]).sum(0) for k in range(3)])
    U = j / rho
    sU = a[:27].sum(0) / np.abs(rho) * (1 + np.abs(U) * a[:27].sum(0))
    g = t[27:].reshape(3, 7, *s.shape[1:])
    dB, sB = g.sum(1), np.abs(g).sum(1)
    B = dB + np.asarray(Bref)[:, None, None, None]
    lam = np.stack([np.stack([g[b, 2 * k + 1] - g[b, 2 * k + 2] for b in range(3)]) for k in range(3)])
    A = np.stack([lam[1, 2] - lam[2, 1], lam[2, 0] - lam[0, 2], lam[0, 1] - lam[1, 0]])
    gq = 4 * omB
    sH = 2 * aH * gq
    y = -gq * (A - 2 * np.cross(U, B, axis=0))
    den = 1 + sH ** 2 * (B * B).sum(0)
    J = (y - sH * np.cross(y, B, axis=0) + sH ** 2 * (y * B).sum(0) * B) / den
    mB, mU = np.abs(B).max(0) + sB.max(0), np.abs(U).max(0) + sU
    sy = gq * (np.abs(g).sum((0, 1)) + 4 * mU * mB)
    sJ = sy * (1 + 2 * sH * mB + 3 * (sH * mB) ** 2) / den
    return (dict(rho=rho, u=U, B=B, J=J),
            dict(rho=1 + a[:27].sum(0), u=sU, B=sB + np.abs(B), J=sJ * (1 + (sH * mB) ** 2 / den)))


@pytest.mark.parametrize("shape", [(2, 3, 5), (1, 2, 32), (3, 2, 129)])
@pytest.mark.parametrize("scale", [0.0, 1e-28, 0.05])
@pytest.mark.parametrize("parity", [0, 1])
def test_moments_of_fp32_storage_are_fp64(shape, scale, parity):
    """Each moment within 64 units of FP64 rounding of its terms' magnitude
    (the sums have at most 27 terms, the current's solve about 40 operations)."""
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    Bref = (0.0, 0.03, 0.1)
    sim = Flame(nx, ny, nz, 0.625, 0.625, 1.5, storage="fp32", B_ref=Bref)
    blob = _blob(shape, scale, 5)
    sim.set_state(torch.from_numpy(blob.reshape(-1).view(np.uint8).copy()).cuda(), parity, parity)
    m = {k: v.cpu().numpy() for k, v in sim.moments().items()}
    only = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
    sim.moments(dict(B=only))
    uB = {k: torch.empty((3,) + shape, dtype=torch.float64, device="cuda") for k in ("u", "B")}
    sim.moments(uB)
    f32 = {k: v.cpu().numpy() for k, v in sim.moments(dtype=torch.float32).items()}
    sim.close()
    f = np.float32
    ref, tol = _reference(_pre_collision(blob, parity), float(f(1 / 0.625)), 1.5, [float(f(b)) for b in Bref])
    for k in ref:
        err = np.abs(m[k] - ref[k])
        assert (err <= 64 * EPS * tol[k]).all(), (k, float((err / (EPS * tol[k] + 1e-300)).max()))
        assert np.array_equal(f32[k], m[k].astype(np.float32))
    assert np.array_equal(only.cpu().numpy(), m["B"])
    assert all(np.array_equal(uB[k].cpu().numpy(), m[k]) for k in uB)
    if scale == 0.0:
        assert not m["u"].any() and not m["J"].any() and (m["rho"] == 1.0).all()


def test_moments_of_overflowing_and_nonfinite_sites():
    """Sites whose sums leave FP32's range keep their FP64 moments, and a
    non-finite population makes its own site non-finite only."""
    from paper_2212_11024_gb300 import Flame
    shape = (2, 2, 33)
    blob = _blob(shape, 0.05, 6)
    blob[:27, 0, 1, 7] = 3e37
    blob[5, 1, 0, 32] = np.inf
    blob[30, 1, 1, 0] = np.nan
    sim = Flame(33, 2, 2, 0.625, 0.625, 1.5, storage="fp32")
    sim.set_state(torch.from_numpy(blob.reshape(-1).view(np.uint8).copy()).cuda(), 0, 0)
    m = {k: v.cpu().numpy() for k, v in sim.moments().items()}
    sim.close()
    with np.errstate(all="ignore"):
        ref, tol = _reference(_pre_collision(blob, 0), float(np.float32(1 / 0.625)), 1.5, (0, 0, 0))
        off = {k: np.abs(m[k] - ref[k]) for k in ref}
    bad = np.zeros(shape, bool)
    bad[1, 0, 32] = bad[1, 1, 0] = True
    for k in ref:
        ok = np.broadcast_to(~bad, ref[k].shape)
        assert (off[k][ok] <= 64 * EPS * np.broadcast_to(tol[k], ref[k].shape)[ok]).all(), k
    assert not np.isfinite(m["rho"][1, 0, 32]) and not np.isfinite(m["B"][:, 1, 1, 0]).all()
    assert np.isfinite(m["u"][:, 1, 1, 0]).all()


def _sums(s, omB, aH, Bref):
    """(flame_reduce_sums, the magnitudes of their terms) in extended precision."""
    m, tol = _reference(s, omB, aH, Bref)
    w = np.array([v[2] for v in _slots()], dtype=np.longdouble)[:, None, None, None]
    t = w * s
    lam = sum(t[27 + 7 * a + 2 * a + 1] - t[27 + 7 * a + 2 * a + 2] for a in range(3))
    slam = sum(np.abs(t[27 + 7 * a + 2 * a + 1]) + np.abs(t[27 + 7 * a + 2 * a + 2]) for a in range(3))
    b = m["B"] - np.asarray(Bref)[:, None, None, None]
    sb, su, sJ = tol["B"], tol["u"] + np.abs(m["u"]), tol["J"] + np.abs(m["J"])
    u, J, rho = m["u"], m["J"], m["rho"]
    dv, sd = 4 * omB * lam, 4 * omB * slam
    out = [rho.sum()] + [(rho * u[a]).sum() for a in range(3)] + [m["B"][a].sum() for a in range(3)]
    out += [(u * u).sum(), (b * b).sum(), (u * b).sum()] + [u[a].sum() for a in range(3)]
    out += [(J * J).sum(), np.sqrt((u * u).sum(0).max()), (dv * dv).sum(), 0.0, rho.size]
    mag = [tol["rho"].sum()] + [(np.abs(rho) * su[a]).sum() for a in range(3)] + [sb[a].sum() for a in range(3)]
    mag += [(su * su).sum(), (sb * sb).sum(), (su * sb).sum()] + [su[a].sum() for a in range(3)]
    mag += [(sJ * sJ).sum(), su.max() * 2, (sd * sd).sum(), 0.0, 0.0]
    return np.array(out, dtype=np.longdouble), np.array(mag, dtype=np.longdouble)


@pytest.mark.parametrize("shape", [(1, 1, 5), (1, 2, 128), (3, 5, 129), (41, 32, 64)])
@pytest.mark.parametrize("scale", [0.0, 1e-20, 0.05, 1e20])
def test_sums_of_fp32_storage(shape, scale):
    """flame_reduce_sums within 2^-43 of the magnitude of the terms (two-term
    arithmetic of about 40 operations a site), the maximum speed to FP64
    rounding; 1e20 leaves the expansions' range, so blocks sum in FP64."""
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    Bref = (0.0, 0.03, 0.1)
    sim = Flame(nx, ny, nz, 0.625, 0.625, 1.5, storage="fp32", B_ref=Bref)
    blob = _blob(shape, scale, 8)
    sim.set_state(torch.from_numpy(blob.reshape(-1).view(np.uint8).copy()).cuda(), 1, 1)
    got = sim.reduce_sums()
    stat = sim.reduce_static().cpu().numpy()
    red = sim.reduce()
    sim.close()
    f = np.float32
    ref, mag = _sums(_pre_collision(blob, 1), float(f(1 / 0.625)), 1.5, [float(f(b)) for b in Bref])
    assert (np.abs(got - ref) <= 2.0 ** -43 * mag).all(), ((np.abs(got - ref) / (mag + 1e-300)).tolist())
    assert abs(got[14] - ref[14]) <= 64 * EPS * mag[14]
    assert np.allclose(stat, [red[k] for k in list(red)[:14]], rtol=1e-12, atol=0)


@pytest.mark.parametrize("storage", ["fp16", "bf16"])
def test_sums_of_16_bit_storage(storage):
    """The sums against FP64 sums of flame_moments' fields: the per-site
    arithmetic is the same FP32 arithmetic, the sums are exact to 2^-43 of
    their terms' magnitude (2^-22 for the squares, which flame_moments'
    caller forms from the rounded fields)."""
    from paper_2212_11024_gb300 import Flame
    shape = (5, 7, 129)
    sim = Flame(129, 7, 5, 0.6, 0.7, 1.5, storage=storage, B_ref=(0.0, 0.03, 0.1))
    gen = torch.Generator().manual_seed(3)
    vals = 0.05 * torch.randn(48 * 5 * 7 * 129, generator=gen)
    dt = torch.float16 if storage == "fp16" else torch.bfloat16
    sim.set_state(vals.to(dt).view(torch.uint8).cuda(), 0, 0)
    got = sim.reduce_sums()
    m = {k: v.cpu().numpy() for k, v in sim.moments().items()}
    sim.close()
    f = np.float32
    b = m["B"] - np.array([0.0, f(0.03), f(0.1)], dtype=np.float64)[:, None, None, None]
    u, J = m["u"], m["J"]
    exact = 2.0 ** -43
    for v, t, tol in [(0, m["rho"], exact)] + [(1 + a, m["rho"] * u[a], exact) for a in range(3)] + \
            [(4 + a, m["B"][a], exact) for a in range(3)] + [(10 + a, u[a], exact) for a in range(3)] + \
            [(7, u * u, 2.0 ** -22), (8, b * b, 2.0 ** -22), (9, u * b, 2.0 ** -22), (13, J * J, 2.0 ** -22)]:
        assert abs(got[v] - t.sum()) <= tol * np.abs(t).sum(), v
    assert abs(got[14] - np.sqrt((u * u).sum(0).max())) <= 2.0 ** -22 * got[14]
    assert got[16] == 0 and got[17] == 5 * 7 * 129


def test_sums_with_nonfinite_sites():
    """Non-finite sites are counted and left out; the other blocks' and the
    same block's finite sites are still summed."""
    from paper_2212_11024_gb300 import Flame, flame
    shape = (2, 20, 64)
    for dt, storage in ((torch.float32, "fp32"), (torch.float16, "fp16")):
        vals = (0.05 * torch.randn((48,) + shape, generator=torch.Generator().manual_seed(4))).to(dt)
        clean = vals.clone()
        clean[:, 0, 3, 5] = 0
        clean[:, 1, 19, 63] = 0
        vals[3, 0, 3, 5] = float("nan")
        vals[9, 1, 19, 63] = float("inf")
        sums = []
        for v in (vals, clean):
            sim = Flame(64, 20, 2, 0.6, 0.7, 1.5, storage=storage)
            sim.set_state(v.reshape(-1).view(torch.uint8).cuda(), 0, 0)
            sums.append(sim.reduce_sums())
            sim.close()
        bad, ok = sums
        assert bad[16] == 2 and ok[16] == 0
        # the cleared sites are at rest: rho = 1, everything else zero
        assert abs(bad[0] + 2 - ok[0]) < 1e-9 and np.allclose(bad[1:16], ok[1:16], rtol=1e-6, atol=1e-9)


def _stored(f, Bref):
    """Deviations from rest over the weight of oracle populations f [48, ...]."""
    s = np.empty(f.shape)
    feq = O.feq_hermite(1.0, np.zeros(3)) + O.lorentz(np.array(Bref, dtype=float))
    geq = O.geq_hall(np.array(Bref, dtype=float), np.zeros(3), np.zeros(3), 0.0).reshape(21)
    rest = np.concatenate([feq, geq])
    for q, (slot, _, w, _) in enumerate(_slots()):
        s[slot] = (f[q] - rest[q]) / w
    return s


@pytest.mark.parametrize("shape", [(3, 4, 5), (2, 3, 129), (9, 8, 32)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("given", ["u B", "rho", "gradients", "no noneq"])
def test_initial_populations_of_fp32_storage(shape, dtype, given):
    """Every stored value is the oracle's FP64 value rounded to FP32: within
    0.501 units of its last place (half a unit of rounding and the two-term
    arithmetic's 2^-44) and 1e-12 (the oracle's FP64 rounding of populations
    of order one, divided by weights down to 1/216)."""
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    r = np.random.default_rng(11)
    u, B = (0.05 * r.standard_normal((3,) + shape)).astype(dtype), (0.05 * r.standard_normal((3,) + shape)).astype(dtype)
    u[:, 0, 0, 1] = 0.0
    B[:, 0, 1, 2] = 0.0
    u[:, 1, 1, 0] = 1e-30
    rho = (1 + 0.01 * r.standard_normal(shape)).astype(dtype) if given == "rho" else None
    gu, gB = ((0.01 * r.standard_normal((9,) + shape)).astype(dtype) if given == "gradients" else None for _ in range(2))
    Bref, tau, d_i = (0.0, 0.03125, 0.125), 0.625, 1.5
    noneq = given != "no noneq"
    sim = Flame(nx, ny, nz, tau, tau, d_i, storage="fp32", B_ref=Bref, init_noneq=noneq)
    sim.init(rho, u, B, gu, gB)
    got = sim.state.view(torch.float32).cpu().numpy().reshape((48,) + shape)
    speed = sim.info()["max_speed"]
    sim.close()
    f64 = [None if a is None else a.astype(np.float64) for a in (rho, u, B, gu, gB)]
    stored_tau = 1.0 / float(np.float32(1.0 / tau))  # the library holds the rates 1 / tau in FP32
    p = O.Params(nx, ny, nz, stored_tau, stored_tau, d_i)
    ref = _stored(O.init(p, *f64, noneq), Bref)
    tol = 0.501 * np.spacing(np.abs(ref).astype(np.float32)).astype(np.float64) + 1e-12
    assert (np.abs(got - ref) <= tol).all(), float((np.abs(got - ref) / tol).max())
    rr = 1.0 if rho is None else f64[0]
    top = max(np.sqrt((f64[2] ** 2).sum(0) / rr).max(), np.sqrt((f64[1] ** 2).sum(0)).max())
    assert abs(speed - top) <= 0.51 * np.spacing(np.float32(top))


def test_initial_populations_beside_rounding_ties():
    """Fields a unit of the FP64 last place beside the middle of two FP32 values
    (further out than the two terms' 48 bits): the stored rest populations of the
    magnetic field are B rounded to FP32, every one of them."""
    from paper_2212_11024_gb300 import Flame
    shape = (4, 5, 33)
    r = np.random.default_rng(12)
    n = r.integers(2 ** 23, 2 ** 24 - 1, (3,) + shape).astype(np.float64) + 0.5
    n *= 2.0 ** -28
    B = r.choice([-1.0, 1.0], n.shape) * np.where(r.random(n.shape) < 0.5, np.nextafter(n, 1), np.nextafter(n, 0))
    sim = Flame(33, 5, 4, 0.6, 0.6, 1.0, storage="fp32")
    sim.init(None, np.zeros_like(B), B)
    got = sim.state.view(torch.float32).cpu().numpy().reshape((48,) + shape)[27:30]
    sim.close()
    assert np.array_equal(got, B.astype(np.float32))


def test_initial_populations_beyond_two_term_range():
    """Fields of 1e13 take the FP64 path: rounded FP64 values there too, and
    a non-finite field is reported."""
    from paper_2212_11024_gb300 import Flame, flame
    shape = (3, 4, 33)
    r = np.random.default_rng(12)
    u, B = 0.05 * r.standard_normal((3,) + shape), 0.05 * r.standard_normal((3,) + shape)
    B[:, 1, 2, 20] = 1e13
    sim = Flame(33, 4, 3, 0.625, 0.625, 0.0, storage="fp32")
    sim.init(None, u, B)
    got = sim.state.view(torch.float32).cpu().numpy().reshape((48,) + shape)
    ref = _stored(O.init(O.Params(33, 4, 3, 0.625, 0.625, 0.0), None, u, B), (0, 0, 0))
    mag = np.abs(ref).max(0)
    assert (np.abs(got - ref) <= 1e-6 * mag + 1e-9).all()
    u[0, 0, 0, 0] = np.nan
    B[0, 0, 0, 0] = np.inf
    with pytest.raises(flame.FlameError) as e:
        sim.init(None, u, B)
    assert e.value.status == flame.FLAME_ERR_NONFINITE
    sim.close()


@pytest.mark.parametrize("shape", [(5, 6, 4), (3, 4, 33), (2, 3, 129)])
@pytest.mark.parametrize("scale", [1.0, 1e36])
def test_init_adjoint_is_fp64(shape, scale):
    """flame_init_adjoint against FP64 autograd with rates that FP32 holds
    exactly (tau = 0.8): 2^-44 of the largest component (sums of up to 48
    terms and ~200 operations in FP64), also where sums of lambda leave
    FP32's range."""
    import ctypes

    from oracle import torch_ref as R
    from paper_2212_11024_gb300 import Flame
    from paper_2212_11024_gb300.flame import library
    nz, ny, nx = shape
    r = np.random.default_rng(13)
    u, B = 0.05 * r.standard_normal((3,) + shape), 0.05 * r.standard_normal((3,) + shape)
    lam = (scale * r.standard_normal((48,) + shape)).astype(np.float32)
    sim = Flame(nx, ny, nz, 0.8, 0.8, 1.5)
    ud, Bd, l0 = torch.tensor(u, device="cuda"), torch.tensor(B, device="cuda"), torch.tensor(lam, device="cuda")
    ub, Bb = torch.empty_like(ud), torch.empty_like(Bd)
    ddi = torch.zeros(1, dtype=torch.float64, device="cuda")
    rc = library().flame_init_adjoint(sim._ctx, *(ctypes.c_void_p(t.data_ptr()) for t in (ud, Bd, l0, ub, Bb, ddi)))
    assert rc == 0
    torch.cuda.synchronize()
    sim.close()
    ut, Bt = torch.tensor(u, requires_grad=True), torch.tensor(B, requires_grad=True)
    d = torch.tensor(1.5, dtype=torch.float64, requires_grad=True)
    g = torch.autograd.grad((R.init(ut, Bt, 0.8, 0.8, d) * torch.tensor(lam.astype(np.float64))).sum(), [ut, Bt, d])
    for got, ref in ((ub.cpu().numpy(), g[0].numpy()), (Bb.cpu().numpy(), g[1].numpy())):
        assert np.abs(got - ref).max() <= 2.0 ** -44 * np.abs(ref).max()
    assert abs(float(ddi[0]) - float(g[2])) <= 2.0 ** -40 * np.abs(g[1].numpy()).sum()


@pytest.mark.parametrize("shape,nshell", [((5, 3, 1), 3), ((3, 4, 2), 4), ((9, 7, 33), 9), ((16, 12, 130), 60),
                                          ((4, 3, 9000), 4096)])
def test_shell_binning(shape, nshell):
    """flame_spectra_fields of given fields against numpy's transform binned
    mode by mode: rows shorter and longer than a warp, Nyquist modes, shells
    dropped at nshell, modes above 2^24 in |m|^2; 1e-12 (FP64 throughout)."""
    from oracle import spectra as S
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    r = np.random.default_rng(14)
    u, B = r.standard_normal((3,) + shape), r.standard_normal((3,) + shape)
    sim = Flame(nx, ny, nz, 0.6, 0.6, 0.5, storage="fp16", fields_only=True)
    Eu, Eb = sim.spectra(nshell, u, B)
    sim.close()
    Bp = B - B.reshape(3, -1).mean(1)[:, None, None, None]
    for got, ref in ((Eu, S.shell_spectrum(u, nshell)), (Eb, S.shell_spectrum(Bp, nshell))):
        assert np.abs(got - ref).max() <= 1e-12 * ref.max()
