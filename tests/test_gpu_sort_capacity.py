"""One handle for galaxies of different sizes: capacities above the sort's switch
from short to long tiles (two long tiles per SM) and calls on both sides of it,
with keys of 13 to 18 bits; and a handle of the default capacity that grows to
above the switch for a call below it. Order and segment offsets bit for bit
against the stable order of the oracle's keys."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu


def _galaxy(n, nx, ny):
    rng = np.random.default_rng(n)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    one = f(np.ones(n))
    return synth.Particles(x=f(rng.uniform(-0.55, 0.55, n) * nx), y=f(rng.uniform(-0.55, 0.55, n) * ny), mass=one, age=one,
                           Z=f(0.01 * np.ones(n)), v_los=f(np.zeros(n)))


# (capacity; None: the default handle, which grows)
@pytest.mark.parametrize("cap,nx,ny", [(2_000_000, 150, 150), (2_000_000, 450, 450), (4_000_000, 250, 250),
                                       (4_000_000, 300, 300), (2_000_000, 64, 64), (None, 150, 150), (None, 450, 450)])
def test_one_handle_many_sizes(cap, nx, ny):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    switch = 2 * torch.cuda.get_device_properties(0).multi_processor_count * 4096
    ssp = synth.ssp_grid(3, 2, 120, 4500.0, 4648.75)
    tel = synth.Telescope(nx=nx, ny=ny, spaxel_size=1.0, n_lambda=33, lambda0=4540.0, dlambda=1.25, psf_fwhm=0.0,
                          lsf_sigma=0.0)
    kw = {} if cap is None else {"max_particles": cap}
    model = CubeModel(ssp, tel, "f32", **kw)
    assert model.stats()["n_bands"] == 1  # so the order is the spaxel order
    sizes = [switch - 7, 1] if cap is None else [switch - 7, cap, switch, 300_001, switch + 1, 1, switch - 1024]
    for n in sizes:
        p = _galaxy(n, nx, ny)
        cube = model.forward(p)
        perm, seg = (t.cpu().numpy() for t in model.sorted())
        key = oracle.spaxel_keys(p.x.astype(np.float64), p.y.astype(np.float64), tel)
        assert np.array_equal(perm, np.argsort(key, kind="stable")), n
        count = np.bincount(key, minlength=nx * ny + 1)
        assert np.array_equal(seg, np.concatenate([[0], np.cumsum(count)])), n
        # every particle has the same spectrum: each row is its count times it
        c = cube.cpu().numpy().reshape(nx * ny, -1).astype(np.float64)
        s = count[:-1] > 0
        unit = (c[s] / count[:-1][s][:, None])[0]
        assert np.allclose(c, count[:-1][:, None] * unit, rtol=2e-5, atol=0.0), n
    assert model.stats()["device_error"] == 0
