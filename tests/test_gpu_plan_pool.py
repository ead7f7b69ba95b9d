"""cuFFT plans that pass from one context to the next: the same results from a
fresh plan and from one that another context, stream and thread has used, and
more lattices than the pool keeps."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _spectra(shape, seed, stream=None):
    import torch
    from paper_2212_11024_gb300 import Flame
    nz, ny, nx = shape
    g = np.random.default_rng(seed)
    u, B = g.standard_normal((3,) + shape), g.standard_normal((3,) + shape)
    sim = Flame(nx, ny, nz, 0.6, 0.6, 0.5, storage="fp16", fields_only=True, stream=stream)
    Eu, Eb = sim.spectra(5, u, B)
    L, dLdB, _ = sim.band_energy(1, 3, B=torch.from_numpy(B).cuda(), grad=True)
    torch.cuda.synchronize()
    d = dLdB.cpu().numpy()
    sim.close()
    return np.concatenate([Eu, Eb, [L]]), d


def test_plans_from_context_to_context():
    import torch
    shapes = [(8, 6, 10 + 2 * i) for i in range(12)]  # more than the pool keeps, twice over
    first = [_spectra(s, 3) for s in shapes]
    again = [_spectra(s, 3, torch.cuda.Stream()) for s in shapes]
    for (a, da), (b, db) in zip(first, again):
        assert np.allclose(a, b, rtol=1e-13, atol=0)
        assert np.abs(da - db).max() <= 1e-13 * np.abs(da).max()
    out = {}

    def work(i):
        out[i] = _spectra(shapes[i % 3], 3, torch.cuda.Stream())

    threads = [threading.Thread(target=work, args=(i,)) for i in range(9)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for i in range(9):
        assert np.allclose(out[i][0], first[i % 3][0], rtol=1e-13, atol=0)
        assert np.abs(out[i][1] - first[i % 3][1]).max() <= 1e-13 * np.abs(first[i % 3][1]).max()
