"""The work a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" says which public entry points
one pass goes through:

  steps     Flame.step(n) on a running lattice; the state it leaves
  adjoint   flame_step_adjoint of one stored state; lambda_t and dL/d(d_i)
  gradient  a whole differentiable run (FlameBandEnergy): forward with
            checkpoints, loss, backward to u0, B0 and d_i
  record    what a decaying-turbulence run records every so many steps:
            Flame.reduce and Flame.spectra
  fields    the start of a run and the reading of its fields: Flame.init,
            then Flame.moments
  job       a run whose fields live in host memory: Flame.init_host, n steps,
            Flame.moments_host with the scalars

Fields are seeded random-phase solenoidal u and B (shells 1..4), the mean
field b0 along z is the reference field of the encoding.  The relaxation
times, amplitudes and d_i keep the runs bounded for thousands of steps.
Lattices are nx x ny x nz; rows (x) are the contiguous axis.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

DTYPE = {"fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def _case(name, kind, shape, storage, **more):
    nx, ny, nz = shape
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, storage=storage, variant="flame", n=1, graph=0, tau=0.6, d_i=2.0,
             rms=0.03, b0=0.0, parity=0)
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # the damped Hall wave's validation lattice: few sites, so launches and latency count
        _case("steps_32_fp32", "steps", (32, 32, 32), "fp32", n=10, rms=1e-3, b0=0.1),
        # decaying turbulence in plain FP32, 128^3
        _case("steps_128_fp32", "steps", (128, 128, 128), "fp32", n=10, tau=0.55, d_i=6.4, rms=0.04),
        # the benchmark's lattice and storage, replayed as graphs of 20 steps
        _case("steps_256_fp16", "steps", (256, 256, 256), "fp16", n=20, graph=20, tau=0.55, d_i=2.56, rms=0.04),
        # the largest production lattice, 12.9 GB of populations
        _case("steps_512_fp16", "steps", (512, 512, 512), "fp16", n=2, tau=0.55, d_i=2.56, rms=0.04),
        # a box whose rows are even but no multiple of 8
        _case("steps_250_bf16", "steps", (250, 124, 132), "bf16", n=10, graph=10, rms=0.03),
        # an odd box (odd rows, odd planes)
        _case("steps_129_fp16", "steps", (129, 127, 131), "fp16", n=10),
        # the current from the central-difference curl of B
        _case("steps_192_fd_fp16", "steps", (192, 192, 192), "fp16", variant="fd_current", n=10, graph=10, d_i=0.25),
        # one reverse step of a differentiable run with 16-bit states
        _case("adjoint_128_fp16", "adjoint", (128, 128, 128), "fp16", d_i=3.2, parity=1),
        # the differentiable run: 64^3, FP32, loss in shells 8..16
        _case("gradient_64_fp32", "gradient", (64, 64, 64), "fp32", n=32, d_i=3.2),
        # the scalars and shell spectra a turbulence run records
        _case("record_128_fp32", "record", (128, 128, 128), "fp32", n=4, tau=0.55, d_i=6.4),
        # the start of an FP32 run and its fields read back
        _case("fields_128_fp32", "fields", (128, 128, 128), "fp32", d_i=6.4),
        # the benchmark's job from and to host memory: fields in, 20 steps, fields and scalars out
        _case("job_256_fp16", "job", (256, 256, 256), "fp16", n=20, graph=20, tau=0.55, d_i=2.56, rms=0.04),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _length(rng, lo, hi):
    """A lattice length: as drawn (odd ones among them), or a multiple of 8 or 32 as most lattices have."""
    v = _log(rng, lo, hi)
    m = rng.choice((1, 1, 2, 8, 32))
    return min(hi, max(lo, (v + m - 1) // m * m))


def draw(rng):
    kind = rng.choice(("steps", "steps", "steps", "steps", "adjoint", "gradient", "record", "fields", "job"))
    storage = rng.choice(("fp32", "fp16", "bf16", "fp16"))
    lo, hi = {"steps": (16, 512), "adjoint": (24, 224), "gradient": (24, 72), "record": (32, 224),
              "fields": (32, 224), "job": (48, 256)}[kind]
    nx = _length(rng, lo, hi)
    # boxes of up to 2:1 in y and z; FP32 storage, whose fields are read and written in FP64, up to 128^3 or so
    ny, nz = (max(16, min(_length(rng, max(16, nx // 2), 2 * nx), hi)) for _ in range(2))
    most = 40_000_000 if kind in ("steps", "adjoint") else 3_000_000 if storage == "fp32" else 17_000_000
    while nx * ny * nz > most and ny * nz > 256:
        ny, nz = max(16, ny * 3 // 4), max(16, nz * 3 // 4)
    n, graph, variant, d_i = 1, 0, "flame", rng.choice((0.0, 0.5, 2.0, round(rng.uniform(0.1, 4.0), 2)))
    if kind in ("steps", "job"):
        # as many steps as keep the pass below the largest listed one
        n = _log(rng, 1, max(2, min(40, 100_000_000 // (nx * ny * nz))))
        if rng.random() < 0.5:
            n += n % 2
            graph = n
    if kind == "steps":
        variant = rng.choice(("flame", "flame", "flame", "bgk", "emhd", "fd_current"))
    if kind == "gradient":
        n, storage = _log(rng, 4, 40), rng.choice(("fp32", "fp32", "fp16"))
    if kind == "record":
        n = rng.randrange(0, 7)
        while nx * ny * nz > 8_000_000:
            ny, nz = max(16, ny * 3 // 4), max(16, nz * 3 // 4)
    if variant == "fd_current":
        d_i = min(d_i, 0.25)
    return _case(None, kind, (nx, ny, nz), storage, n=n, graph=graph, variant=variant, d_i=d_i,
                 tau=round(rng.uniform(0.56, 0.8), 3), rms=round(rng.uniform(0.01, 0.035), 4),
                 b0=rng.choice((0.0, 0.05)), parity=rng.randrange(2) if kind == "adjoint" else 0)


# --------------------------------------------------------------------- inputs
def _band_field(c, rng, hi=4):
    """[3, nz, ny, nx] FP64 solenoidal random-phase field on the GPU, modes 1 <= round|m| <= hi."""
    m = np.arange(-hi, hi + 1)
    K = 2 * hi + 1
    V = rng.standard_normal((3, K, K, K)) + 1j * rng.standard_normal((3, K, K, K))  # [component, mz, my, mx]
    mz, my, mx = np.meshgrid(m, m, m, indexing="ij")
    shell = np.rint(np.sqrt(mx * mx + my * my + mz * mz))
    k = np.stack([np.sin(2 * np.pi * mx / c["nx"]), np.sin(2 * np.pi * my / c["ny"]), np.sin(2 * np.pi * mz / c["nz"])])
    kk = (k * k).sum(0)
    V = V - k * ((k * V).sum(0) / np.where(kk > 0, kk, 1.0))
    V = V * np.where((shell >= 1) & (shell <= hi), 1.0 / np.maximum(shell, 1.0), 0.0)
    e = [np.exp(2j * np.pi * np.outer(m, np.arange(c[a])) / c[a]) for a in ("nx", "ny", "nz")]
    out = torch.empty((3, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda")
    for a in range(3):
        t = np.einsum("zyx,xi,yj->zji", V[a], e[0], e[1]).reshape(K, -1)  # [mz, y x]
        tr, ti = torch.from_numpy(t.real.copy()).cuda(), torch.from_numpy(t.imag.copy()).cuda()
        zr, zi = torch.from_numpy(e[2].real.T.copy()).cuda(), torch.from_numpy(e[2].imag.T.copy()).cuda()
        flat = out[a].view(c["nz"], -1)
        torch.mm(zr, tr, out=flat)
        flat.addmm_(zi, ti, alpha=-1.0)
    scale = 0.0
    for a in range(3):
        scale += float((out[a] * out[a]).mean())
    return out.mul_(c["rms"] / math.sqrt(scale / 3.0))


def _fields(c, seed):
    """u, B of the case as its program holds them: FP64 for FP32 storage, FP32 for 16-bit storage and host jobs."""
    rng = np.random.default_rng(seed)
    dt = torch.float64 if c["storage"] == "fp32" and c["kind"] != "job" else torch.float32
    u = _band_field(c, rng).to(dt)
    B = _band_field(c, rng)
    B[2] += c["b0"]
    return u, B.to(dt)


def _lambda(c, seed):
    """A seeded FP32 lambda_{t+1} [48, N3] in natural slot order: low moments of smooth fields, as adjoint states are."""
    rng = np.random.default_rng([int(seed), 1])
    p, a = (_band_field(c, rng).float().view(3, -1) for _ in range(2))
    lam = torch.empty((48, p.shape[1]), dtype=torch.float32, device="cuda")
    for q, v in enumerate(NATURAL):
        lam[q] = sum((v[k] * p[k] + 0.5 * v[k] * v[k] * a[k] for k in range(3) if v[k]), 0.25 * a[0])
    for b in range(3):
        for i, v in enumerate(D7):
            lam[27 + 7 * b + i] = sum((v[k] * p[(k + b) % 3] for k in range(3) if v[k]), a[b])
    return lam


BAND = (8, 16)  # shells of the gradient runs' loss


def _band(c):
    """The loss's shells: 8..16, or the upper half of what a smaller lattice resolves."""
    top = min(c["nx"], c["ny"], c["nz"]) // 2
    return BAND if top >= 16 else (top // 2, top)


def _nshell(c):
    return max(c["nx"], c["ny"], c["nz"]) // 2 + 1


# ------------------------------------------------------------- the library's
def prepare(c, seed):
    from paper_2212_11024_gb300 import Flame

    torch.cuda.set_device(0)
    u, B = _fields(c, seed)
    s = dict(c=c)
    if c["kind"] == "gradient":
        # FP32 parameters, as an optimiser over initial fields holds them
        s["u"], s["B"] = (t.float().requires_grad_() for t in (u, B))
        s["d_i"] = torch.tensor(c["d_i"], dtype=torch.float32, device="cuda", requires_grad=True)
        return s
    sim = s["sim"] = Flame(c["nx"], c["ny"], c["nz"], c["tau"], c["tau"], c["d_i"], storage=c["storage"],
                           B_ref=(0.0, 0.0, c["b0"]), graph_steps=c["graph"], variant=c["variant"])
    if c["kind"] == "fields":
        s["u"], s["B"] = u, B
    elif c["kind"] == "job":
        s["u"], s["B"] = (torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (u, B))
        shape = (3, c["nz"], c["ny"], c["nx"])
        s["out"] = {k: torch.empty(shape, dtype=torch.float32, pin_memory=True) for k in ("u", "B", "J")}
    else:
        sim.init(None, u, B)
        if c["kind"] == "record":
            sim.step(c["n"])
        if c["kind"] == "adjoint":
            sim.step(c["parity"])
            s["blob"], _, s["par"] = sim.get_state()
            s["lam"] = _lambda(c, seed)
            s["out"] = torch.empty_like(s["lam"])
            s["ddi"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    return s


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def run(s):
    from paper_2212_11024_gb300 import flame

    c = s["c"]
    if c["kind"] == "gradient":
        from paper_2212_11024_gb300.adjoint import FlameBandEnergy

        L = FlameBandEnergy.apply(s["u"], s["B"], s["d_i"], c["tau"], c["tau"], c["n"], _band(c), c["storage"])
        gu, gB, gd = torch.autograd.grad(L, (s["u"], s["B"], s["d_i"]))
        return {"L": L.detach().float(), "u": gu, "B": gB, "d_i": gd}
    sim = s["sim"]
    if c["kind"] == "steps":
        sim.step(c["n"])
        return sim.state.view(DTYPE[c["storage"]])
    if c["kind"] == "adjoint":
        flame._check(flame.library().flame_step_adjoint(sim._ctx, _ptr(s["blob"]), s["par"], _ptr(s["lam"]),
                                                        _ptr(s["out"]), _ptr(s["ddi"])), "flame_step_adjoint")
        return {"lambda": s["out"], "d_i": s["ddi"].float()}
    if c["kind"] == "record":
        r = sim.reduce()
        Eu, Eb = sim.spectra(_nshell(c))
        return {"scalars": np.array([r[k] for k in flame.SCALAR_NAMES]), "Eu": Eu, "Eb": Eb}
    if c["kind"] == "fields":
        sim.init(None, s["u"], s["B"])
        m = sim.moments(dtype=s["u"].dtype)
        return {"state": sim.state.view(DTYPE[c["storage"]]), "rho": m["rho"], "u": m["u"], "B": m["B"], "J": m["J"]}
    sim.init_host(None, s["u"], s["B"])
    sim.step(c["n"])
    m, r = sim.moments_host(s["out"], scalars=True)
    return {"u": m["u"], "B": m["B"], "J": m["J"], "scalars": np.array([r[k] for k in flame.SCALAR_NAMES])}


def work(c):
    """Bytes and operations one pass cannot do without.  A step reads and writes the 48 populations of every site
    (a lattice step is one pass: nothing else carries the state from one step to the next) and takes about 900
    operations per site; its adjoint about 3000."""
    n3 = c["nx"] * c["ny"] * c["nz"]
    e = 4 if c["storage"] == "fp32" else 2
    step = 96.0 * e * n3
    if c["kind"] == "steps":
        return {"bytes": step * c["n"], "flops": 900.0 * n3 * c["n"]}
    vjp = (48.0 * e + 2 * 48 * 4) * n3
    if c["kind"] == "adjoint":
        return {"bytes": vjp, "flops": 3000.0 * n3}
    fft = 2.5 * n3 * math.log2(n3)  # operations of one real transform
    if c["kind"] == "gradient":
        return {"bytes": (step + vjp) * c["n"] + (6 * 4 * 2 + 48 * e) * n3,
                "flops": 3900.0 * n3 * c["n"] + 6 * fft}
    if c["kind"] == "record":
        return {"bytes": 48.0 * e * n3, "flops": 300.0 * n3 + 6 * fft}
    if c["kind"] == "fields":
        f = 8 if c["storage"] == "fp32" else 4
        return {"bytes": (2 * 48.0 * e + (6 + 10) * f) * n3, "flops": 900.0 * n3}
    return {"bytes": step * c["n"] + (6 + 9) * 4.0 * n3, "flops": (900.0 * c["n"] + 900.0) * n3}


# -------------------------------------------------------- the same in 64 bits
# Fluid velocities in the order of the state's fluid slots, (cx+1) + 3 (cy+1) + 9 (cz+1), the magnetic ones (rest,
# +x, -x, +y, -y, +z, -z), and the fluid velocities in natural order (flame.h), which the adjoint vectors have.
CUBE = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
D7 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
_HALF = [(-1, 0, 0), (0, -1, 0), (0, 0, -1), (-1, -1, 0), (-1, 1, 0), (-1, 0, -1), (-1, 0, 1), (0, -1, -1),
         (0, -1, 1), (-1, -1, -1), (-1, -1, 1), (-1, 1, -1), (-1, 1, 1)]
NATURAL = [(0, 0, 0)] + _HALF + [tuple(-a for a in v) for v in _HALF]
W1 = {0: 2.0 / 3.0, 1: 1.0 / 6.0, -1: 1.0 / 6.0}


def _w(v):
    return W1[v[0]] * W1[v[1]] * W1[v[2]]


def _w7(i):
    return 0.25 if i == 0 else 0.125


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _lorentz(v, B, b2):
    cb = sum(v[a] * B[a] for a in range(3) if v[a]) if any(v) else 0.0
    c2 = sum(abs(a) for a in v)
    return 4.5 * _w(v) * (0.5 * b2 * (c2 - 1.0 / 3.0) - cb * cb)


def _psi(U):
    return [{0: 2.0 / 3.0 - u * u, 1: 0.5 * (1.0 / 3.0 + u * u + u), -1: 0.5 * (1.0 / 3.0 + u * u - u)} for u in U]


def _hall(B, V, b, i):
    """g^Hall(0) of component b on D3Q7 velocity i."""
    a = next((k for k in range(3) if D7[i][k]), None)
    if a is None:
        return 0.25 * B[b]
    return 0.125 * (B[b] + 4.0 * D7[i][a] * (V[a] * B[b] - B[a] * V[b]))


def _moments(c, f, g, di, curl=None):
    """rho, U, B, J, V = U - d_i J and Lambda of populations f [27 of [S]] (cube order), g [3][7]."""
    rho = sum(f)
    U = [sum(v[a] * x for v, x in zip(CUBE, f) if v[a]) / rho for a in range(3)]
    B = [sum(g[b]) for b in range(3)]
    lam = [[g[b][2 * a + 1] - g[b][2 * a + 2] for b in range(3)] for a in range(3)]
    q = 4.0 / c["tau"]
    Ue = [torch.zeros_like(x) for x in U] if c["variant"] == "emhd" else U
    if curl is None:
        A = [lam[1][2] - lam[2][1], lam[2][0] - lam[0][2], lam[0][1] - lam[1][0]]
        y = [-q * (x - 2.0 * z) for x, z in zip(A, _cross(Ue, B))]
        s = 2.0 * q * di
        yb, yx, den = _dot(y, B), _cross(y, B), 1.0 + s * s * _dot(B, B)
        J = [(y[a] - s * yx[a] + s * s * yb * B[a]) / den for a in range(3)]
    else:
        J = curl
    return rho, U, B, J, [Ue[a] - di * J[a] for a in range(3)], lam


def _collide(c, f, g, di, curl=None):
    rho, U, B, _, V, _ = _moments(c, f, g, di, curl)
    w = 1.0 / c["tau"]
    b2, psi = _dot(B, B), _psi(U)
    fe = [rho * psi[0][v[0]] * psi[1][v[1]] * psi[2][v[2]] + _lorentz(v, B, b2) for v in CUBE]
    if c["variant"] == "bgk":
        fs = [x - w * (x - e) for x, e in zip(f, fe)]
    else:
        S = [[sum(v[a] * v[b] * x for v, x in zip(CUBE, f) if v[a] * v[b]) - rho * U[a] * U[b] + B[a] * B[b]
              for b in range(3)] for a in range(3)]
        tr = (S[0][0] + S[1][1] + S[2][2]) / 3.0
        D = [[(1.0 - w) * (S[a][b] - tr if a == b else S[a][b]) for b in range(3)] for a in range(3)]
        # the population whose central moments are zero but the second-order ones D: inverse-moment maps per axis
        F0 = [{0: 1.0 - u * u, 1: 0.5 * (u * u + u), -1: 0.5 * (u * u - u)} for u in U]
        F1 = [{0: -2.0 * u, 1: u + 0.5, -1: u - 0.5} for u in U]
        F2 = {0: -1.0, 1: 0.5, -1: 0.5}
        fs = []
        for v, e in zip(CUBE, fe):
            x, y, z = v
            p = F0[2][z] * (D[0][0] * F2[x] * F0[1][y] + D[1][1] * F2[y] * F0[0][x] + D[0][1] * F1[0][x] * F1[1][y])
            p = p + F1[2][z] * (D[0][2] * F1[0][x] * F0[1][y] + D[1][2] * F0[0][x] * F1[1][y])
            fs.append(e + p + F2[z] * D[2][2] * F0[0][x] * F0[1][y])
    gs = [[g[b][i] - w * (g[b][i] - _hall(B, V, b, i)) for i in range(7)] for b in range(3)]
    return fs, gs


def _cdiff(F, a):
    return 0.5 * (torch.roll(F, -1, 2 - a) - torch.roll(F, 1, 2 - a))


def _curl(B):
    return [_cdiff(B[2], 1) - _cdiff(B[1], 2), _cdiff(B[0], 2) - _cdiff(B[2], 0), _cdiff(B[1], 0) - _cdiff(B[0], 1)]


def _start(c, u, B, di):
    """Initial populations: 27 fluid (cube order) and [3][7] magnetic fields."""
    w = 1.0 / c["tau"]
    U, Bl = [u[0], u[1], u[2]], [B[0], B[1], B[2]]
    b2, psi, J = _dot(Bl, Bl), _psi(U), _curl(Bl)
    P = [[None] * 3 for _ in range(3)]
    for a in range(3):
        for b in range(a, 3):
            P[a][b] = P[b][a] = -(_cdiff(U[b], a) + _cdiff(U[a], b)) / (3.0 * w)
    tr = (P[0][0] + P[1][1] + P[2][2]) / 3.0
    f = []
    for v in CUBE:
        x = psi[0][v[0]] * psi[1][v[1]] * psi[2][v[2]] + _lorentz(v, Bl, b2)
        ne = sum(v[a] * v[b] * P[a][b] for a in range(3) for b in range(3) if v[a] * v[b]) if any(v) else 0.0
        f.append(x + 4.5 * _w(v) * (ne - tr))
    V = [U[a] - di * J[a] for a in range(3)]
    g = [[_hall(Bl, V, b, i) for i in range(7)] for b in range(3)]
    for b in range(3):
        for i in range(1, 7):
            a = (i - 1) // 2
            g[b][i] = g[b][i] - 0.125 / w * D7[i][a] * _cdiff(Bl[b], a)
    return f, g


def _stream(x, v):
    return torch.roll(x, (v[2], v[1], v[0]), (0, 1, 2)) if any(v) else x


def _step(c, f, g, di):
    fs, gs = _collide(c, f, g, di, _curl([sum(g[b]) for b in range(3)]) if c["variant"] == "fd_current" else None)
    return [_stream(x, v) for x, v in zip(fs, CUBE)], [[_stream(x, v) for x, v in zip(r, D7)] for r in gs]


def _march(c, pop, n):
    """n steps of pop [48, nz, ny, nx] FP64 (storage slot order) in slabs of planes; pop is overwritten."""
    planes = max(1, 4_000_000 // (c["nx"] * c["ny"]))
    vel = CUBE + [D7[i] for i in range(7) for _ in range(3)]
    for _ in range(n):
        curl = None
        if c["variant"] == "fd_current":
            curl = _curl([pop[27 + b::3].sum(0) for b in range(3)])
        for z in range(0, c["nz"], planes):
            p = pop[:, z:z + planes]
            f, g = [p[q] for q in range(27)], [[p[27 + 3 * i + b] for i in range(7)] for b in range(3)]
            fs, gs = _collide(c, f, g, c["d_i"], [j[z:z + planes] for j in curl] if curl else None)
            p[:] = torch.stack(fs + [gs[b][i] for i in range(7) for b in range(3)])
        for q in range(48):
            pop[q] = _stream(pop[q], vel[q])
    return pop


def _storage(f, g):
    return torch.stack(f + [g[b][i] for i in range(7) for b in range(3)])


def _rest(c):
    """(weight, rest population) per storage slot."""
    B = (0.0, 0.0, c["b0"])
    w = [_w(v) for v in CUBE] + [_w7(i) for i in range(7) for _ in range(3)]
    r = [_w(v) + _lorentz(v, B, c["b0"] ** 2) for v in CUBE] + [_w7(i) * B[b] for i in range(7) for b in range(3)]
    return w, r


def _encoded(c, pop, parity):
    """The state's values: deviations from rest over the weight, at their place for the AA parity.  Overwrites pop."""
    w, r = _rest(c)
    for q in range(48):
        pop[q].sub_(r[q]).div_(w[q])
    if not parity:
        return pop
    vel = CUBE + [D7[i] for i in range(7) for _ in range(3)]
    opp = [26 - q for q in range(27)] + [27 + 3 * (0 if i == 0 else (i - 1 ^ 1) + 1) + b for i in range(7)
                                         for b in range(3)]
    out = torch.empty_like(pop)
    for q in range(48):
        out[opp[q]] = _stream(pop[q], tuple(-a for a in vel[q]))
    return out


def _stored(c, pop):
    """pop as the storage type holds it."""
    w, r = _rest(c)
    for q in range(48):
        x = ((pop[q] - r[q]) / w[q]).float()
        pop[q] = x.to(DTYPE[c["storage"]]).double() * w[q] + r[q]
    return pop


def _spectrum(F, nshell, zero_mean):
    nz, ny, nx = F.shape[1:]
    m = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda") for n in (nz, ny, nx)]
    shell = torch.sqrt(m[0][:, None, None] ** 2 + m[1][None, :, None] ** 2 + m[2] ** 2).round().long().flatten()
    p = sum((torch.fft.fftn(F[b]) / F[b].numel()).abs().square() for b in range(3))
    if zero_mean:
        p[0, 0, 0] = 0.0
    return 0.5 * torch.zeros(int(shell.max()) + 1, dtype=torch.float64, device="cuda").index_add_(
        0, shell, p.flatten())[:nshell]


def _scalars(c, pop):
    f, g = [pop[q] for q in range(27)], [[pop[27 + 3 * i + b] for i in range(7)] for b in range(3)]
    rho, U, B, J, _, lam = _moments(c, f, g, c["d_i"])
    Bm = [x.mean() for x in B]
    d = [x - m for x, m in zip(B, Bm)]
    div = (4.0 / c["tau"]) * (lam[0][0] + lam[1][1] + lam[2][2])
    s = [rho.sum()] + [(rho * x).sum() for x in U] + Bm
    s += [0.5 * _dot(U, U).mean(), 0.5 * _dot(d, d).mean(), _dot(U, d).mean(), _dot(J, J).mean(),
          _dot(U, U).max().sqrt(), (div * div).mean().sqrt(), torch.zeros((), dtype=torch.float64, device="cuda")]
    return torch.stack(s), torch.stack(U), torch.stack(B), torch.stack(J), rho


def _exact_adjoint(c, pop, seed):
    shape = (c["nz"], c["ny"], c["nx"])
    lam = _lambda(c, seed).double().view((48,) + shape)
    order = [CUBE.index(v) for v in NATURAL]  # natural slot -> cube slot
    out, ddi = torch.empty_like(lam), 0.0
    vel = NATURAL + [D7[i] for _ in range(3) for i in range(7)]
    for q in range(48):  # dL/df* at x is lambda_{t+1} at x + c_q
        lam[q] = _stream(lam[q], tuple(-a for a in vel[q]))
    planes = max(1, 500_000 // (c["nx"] * c["ny"]))
    for z in range(0, c["nz"], planes):
        with torch.enable_grad():
            x = pop[:, z:z + planes].clone().requires_grad_()
            di = torch.tensor(c["d_i"], dtype=torch.float64, device="cuda", requires_grad=True)
            f, g = [x[q] for q in range(27)], [[x[27 + 3 * i + b] for i in range(7)] for b in range(3)]
            fs, gs = _collide(c, f, g, di)
            y = torch.stack([fs[order[q]] for q in range(27)] + [gs[b][i] for b in range(3) for i in range(7)])
            gx, gd = torch.autograd.grad(y, (x, di), lam[:, z:z + planes])
        ddi += float(gd)
        for q in range(27):
            out[q, z:z + planes] = gx[order[q]]
        for b in range(3):
            for i in range(7):
                out[27 + 7 * b + i, z:z + planes] = gx[27 + 3 * i + b]
    return {"lambda": out.view(48, -1), "d_i": torch.tensor([ddi], dtype=torch.float64, device="cuda")}


def _exact_gradient(c, u, B):
    from torch.utils.checkpoint import checkpoint

    u, B = (t.float().double().requires_grad_() for t in (u, B))
    di = torch.tensor(c["d_i"], dtype=torch.float32, device="cuda").double().requires_grad_()

    def one(pop, di):
        return _storage(*_step(c, [pop[q] for q in range(27)],
                               [[pop[27 + 3 * i + b] for i in range(7)] for b in range(3)], di))

    with torch.enable_grad():
        pop = checkpoint(lambda u, B, di: _storage(*_start(c, u, B, di)), u, B, di, use_reentrant=False)
        for _ in range(c["n"]):
            pop = checkpoint(one, pop, di, use_reentrant=False)
        Bf = torch.stack([pop[27 + b::3].sum(0) for b in range(3)])
        lo, hi = _band(c)
        m = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda") for n in Bf.shape[1:]]
        shell = torch.sqrt(m[0][:, None, None] ** 2 + m[1][None, :, None] ** 2 + m[2] ** 2).round()
        p = sum((torch.fft.fftn(Bf[b]) / Bf[b].numel()).abs().square() for b in range(3))
        L = 0.5 * (p * ((shell >= lo) & (shell <= hi))).sum()
        gu, gB, gd = torch.autograd.grad(L, (u, B, di))
    return {"L": L.detach(), "u": gu, "B": gB, "d_i": gd}


def exact(c, seed):
    n3 = c["nx"] * c["ny"] * c["nz"]
    if n3 * c["n"] > 400_000_000 or (c["kind"] == "gradient" and n3 * c["n"] > 12_000_000):
        return None  # too long
    torch.cuda.set_device(0)
    u, B = _fields(c, seed)
    if c["kind"] == "gradient":
        return _exact_gradient(c, u, B)
    with torch.no_grad():
        pop = _storage(*_start(c, u.double(), B.double(), c["d_i"]))
        del u, B
        if c["kind"] == "steps":
            return _encoded(c, _march(c, pop, c["n"]), c["n"] % 2).flatten()
        if c["kind"] == "adjoint":
            pop = _stored(c, pop)
            return _exact_adjoint(c, _stored(c, _march(c, pop, 1)) if c["parity"] else pop, seed)
        if c["kind"] == "record":
            s, U, Bf, _, _ = _scalars(c, _march(c, pop, c["n"]))
            return {"scalars": s, "Eu": _spectrum(U, _nshell(c), False), "Eb": _spectrum(Bf, _nshell(c), True)}
        if c["kind"] == "fields":
            _, U, Bf, J, rho = _scalars(c, pop)
            return {"state": _encoded(c, pop, 0).flatten(), "rho": rho, "u": U, "B": Bf, "J": J}
        s, U, Bf, J, _ = _scalars(c, _march(c, pop, c["n"]))
        return {"u": U, "B": Bf, "J": J, "scalars": s}
