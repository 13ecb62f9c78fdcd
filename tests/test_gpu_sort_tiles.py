"""Sort order, segment offsets and work items at the edges of their tiles: particle
counts around the radix tiles (1024 and 4096 keys) and the switch between them,
spaxel counts around the work items' scan tiles (1024 spaxels). Bit for bit
against the stable order of the oracle's keys."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nx,ny", [(1, 1, 1), (31, 3, 2), (1023, 32, 32), (1024, 31, 33), (1025, 1023, 1),
                                     (4097, 1024, 1), (5000, 205, 5), (40_000, 300, 301), (1_245_184, 64, 64),
                                     (1_245_185, 64, 64), (1_300_001, 257, 129)])
def test_sort_and_items(n, nx, ny):
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(3, 2, 120, 4500.0, 4648.75)
    tel = synth.Telescope(nx=nx, ny=ny, spaxel_size=1.0, n_lambda=33, lambda0=4540.0, dlambda=1.25, psf_fwhm=0.0,
                          lsf_sigma=0.0)
    rng = np.random.default_rng(n)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    one = f(np.ones(n))
    p = synth.Particles(x=f(rng.uniform(-0.55, 0.55, n) * nx), y=f(rng.uniform(-0.55, 0.55, n) * ny), mass=one,
                        age=one, Z=f(0.01 * np.ones(n)), v_los=f(np.zeros(n)))
    model = CubeModel(ssp, tel, "f32", max_particles=n)
    assert model.stats()["n_bands"] == 1  # so the order is the spaxel order
    for _ in range(2):  # the second pass finds the first one's scan state
        cube = model.forward(p)
        perm, seg = (t.cpu().numpy() for t in model.sorted())
        key = oracle.spaxel_keys(p.x.astype(np.float64), p.y.astype(np.float64), tel)
        assert np.array_equal(perm, np.argsort(key, kind="stable"))
        count = np.bincount(key, minlength=nx * ny + 1)
        assert np.array_equal(seg, np.concatenate([[0], np.cumsum(count)]))
        # every particle has the same spectrum: each row is its count times it
        c = cube.cpu().numpy().reshape(nx * ny, -1).astype(np.float64)
        s = count[:-1] > 0
        unit = (c[s] / count[:-1][s][:, None])[0]
        assert np.allclose(c, count[:-1][:, None] * unit, rtol=2e-5, atol=0.0)
    assert model.stats()["device_error"] == 0
