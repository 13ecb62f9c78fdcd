"""Wavelength grids around and above 4096 bins, where the deposit's fixed-point Doppler
shifts are taken at bin 4096, for bin steps of every kind, bin centres and means,
with line-of-sight speeds up to the slab's halo and past it. Against the FP64 oracle,
at the tolerances of the other parity tests (1e-5 of the cube's maximum, 1e-4 of each
gradient's)."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu
NT = 8


def _galaxy(n, seed, v_max):
    rng = np.random.default_rng(seed)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    return synth.Particles(x=f(rng.normal(0, 0.8, n)), y=f(rng.normal(0, 0.8, n)), mass=f(np.exp(rng.normal(0, 0.5, n))),
                           age=f(np.exp(rng.uniform(np.log(0.08), np.log(15), n))),
                           Z=f(np.exp(rng.uniform(np.log(8e-5), np.log(0.05), n))), v_los=f(rng.uniform(-v_max, v_max, n)))


@pytest.mark.parametrize("resample", [0, 1])
@pytest.mark.parametrize("n_lambda,a0", [(4096, 0.99), (4097, 0.99), (8192, 0.99), (8192, 1.0005), (4097, 0.7),
                                         (8192, 0.7), (4096, 1.6), (4097, 1.6), (8192, 1.6)])
def test_many_bins(n_lambda, a0, resample):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    n_ls = min(16384, int(n_lambda * a0) + 200)
    ssp = synth.ssp_grid(9, 4, n_ls, 4500.0, 4500.0 + 0.7 * (n_ls - 1))
    tel = synth.Telescope(nx=3, ny=2, spaxel_size=1.0, n_lambda=n_lambda, lambda0=4550.3, dlambda=0.7 * a0, psf_fwhm=0.0,
                          lsf_sigma=0.0, resample=resample)
    p = _galaxy(500, n_lambda, 1500.0)
    model = CubeModel(ssp, tel, "f32", max_particles=p.n)
    got = model.forward(p).cpu().numpy()
    ref = oracle.forward(p, ssp, tel, n_threads=NT)
    assert float(np.abs(got - ref).max()) <= 1e-5 * float(np.abs(ref).max())
    # a smooth positive cotangent, as in the tests of the bin steps
    G = np.ones(model.cube_shape, dtype=np.float32) * (1.0 + 0.3 * np.sin(np.arange(n_lambda) / 40.0)).astype(np.float32)
    grads = [g.cpu().numpy() for g in model.backward(torch.from_numpy(G).cuda())[:4]]
    assert model.stats()["device_error"] == 0
    key = oracle.spaxel_keys(p.x.astype(np.float64), p.y.astype(np.float64), tel)
    want = oracle.gradient(key, p.v_los.astype(np.float64), p, ssp, tel, G.astype(np.float64), n_threads=NT)
    for name, g, o in zip(("mass", "age", "Z"), grads, want):
        assert float(np.abs(g - o).max()) <= 1e-4 * float(np.abs(o).max()), name
    # the velocity gradient: a bin on a node takes the slope on either side
    d = np.abs(grads[3] - want[3]) / np.abs(want[3]).max()
    assert np.mean(d > 1e-4) <= 0.02 and float(d.max()) <= 2e-2
