"""The deposit's and the adjoint's rounds for every bin step dt/dj (output bins
per template step), at the edges of their ranges: steps near 1 on both sides,
below and above 1, and beyond the two-read edges of bin means; grids of one age
or one metallicity; tiles with a ragged end; Doppler shifts up to the slab's
halo and past it. Against the FP64 oracle, at the tolerances of the other
parity tests (1e-5 of the cube's maximum, 1e-4 of each gradient's)."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu
NT = 8


def _galaxy(n, seed, v_max):
    rng = np.random.default_rng(seed)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    return synth.Particles(x=f(rng.normal(0, 1.5, n)), y=f(rng.normal(0, 1.5, n)),
                           mass=f(np.exp(rng.normal(0, 0.5, n))), age=f(np.exp(rng.uniform(np.log(0.08), np.log(15), n))),
                           Z=f(np.exp(rng.uniform(np.log(8e-5), np.log(0.05), n))),
                           v_los=f(rng.uniform(-v_max, v_max, n)))


# template steps are 1.25 A: dt/dj = dlambda / 1.25
STEPS = [0.3, 0.501, 0.7, 0.9676, 0.968, 0.99, 1.0, 1.01, 1.033, 1.4, 1.99, 2.0, 2.7]


@pytest.mark.parametrize("resample", [0, 1])
@pytest.mark.parametrize("a0", STEPS)
def test_bin_steps(a0, resample):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(9, 5, 1801, 4500.0, 6750.0)
    assert abs(ssp.dlambda - 1.25) < 1e-12
    n_lambda = min(1187, int(1900.0 / (1.25 * a0)))
    tel = synth.Telescope(nx=7, ny=5, spaxel_size=1.0, n_lambda=n_lambda, lambda0=4550.3, dlambda=1.25 * a0,
                          psf_fwhm=0.0, lsf_sigma=0.0, resample=resample)
    p = _galaxy(1500, 5, 900.0)  # the slab's halo covers 800 km/s
    model = CubeModel(ssp, tel, "f32", max_particles=p.n)
    got = model.forward(p)
    ref = oracle.forward(p, ssp, tel, n_threads=NT)
    assert float(np.abs(got.cpu().numpy() - ref).max()) <= 1e-5 * float(np.abs(ref).max())
    # a smooth positive cotangent: no bin decides a gradient by itself, so that a
    # bin within rounding of a template node (where the slope jumps) cannot
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


@pytest.mark.parametrize("n_age,n_Z", [(1, 1), (1, 4), (6, 1), (2, 2)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_bin_steps_degenerate_grids(n_age, n_Z, dtype):
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(n_age, n_Z, 900, 4500.0, 5623.75)
    if dtype == "bf16":  # the oracle on the rounded templates
        import torch
        ssp.spectra = torch.from_numpy(ssp.spectra).float().to(torch.bfloat16).double().numpy()
    tel = synth.Telescope(nx=6, ny=6, spaxel_size=1.0, n_lambda=401, lambda0=4600.0, dlambda=1.9, psf_fwhm=0.0,
                          lsf_sigma=0.0)
    p = _galaxy(700, 6, 300.0)
    model = CubeModel(ssp, tel, dtype, max_particles=p.n)
    got = model.forward(p).cpu().numpy()
    ref = oracle.forward(p, ssp, tel, n_threads=NT)
    assert float(np.abs(got - ref).max()) <= 1e-5 * float(np.abs(ref).max())
    assert model.stats()["device_error"] == 0
