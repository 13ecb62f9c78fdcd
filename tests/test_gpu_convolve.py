"""rubix_convolve on dense cubes of any alignment and size, against the oracle's
direct PSF and LSF: rows that start anywhere in a 16-byte granule, fewer bins
than a tile and tiles with a ragged end, cubes narrower than the PSF, a buffer
that ends inside a granule. Cubes with few occupied spaxels through the forward.
Tolerance of the other parity tests (1e-5 of the cube's maximum)."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu
NT = 8


@pytest.mark.parametrize("dlambda", [1.25, 3.0])  # LSF radii 4 and 2
@pytest.mark.parametrize("nx,ny,nl,shift", [(1, 1, 1, 0), (3, 2, 3, 1), (7, 9, 5, 2), (8, 30, 120, 3), (9, 5, 121, 0),
                                            (17, 40, 250, 1), (33, 12, 1001, 2), (16, 601, 7, 3), (40, 21, 400, 0)])
def test_convolve_dense(nx, ny, nl, shift, dlambda):
    import torch
    from paper_2412_08265_gb300 import capi
    from paper_2412_08265_gb300.model import CubeModel
    tel = synth.Telescope(nx=nx, ny=ny, spaxel_size=1.0, n_lambda=nl, lambda0=5000.0, dlambda=dlambda)
    rng = np.random.default_rng(nx + nl)
    cube = rng.normal(0.0, 1.0, (ny, nx, nl)).astype(np.float32)
    # the cube inside a larger buffer of NaN, `shift` floats past a 16-byte boundary
    buf = torch.full((cube.size + 8,), float("nan"), device="cuda")
    buf[shift:shift + cube.size] = torch.from_numpy(cube.reshape(-1)).cuda()
    out = torch.full((ny, nx, nl), float("nan"), device="cuda")
    capi.rubix_convolve(CubeModel.c_telescope(tel), buf.data_ptr() + 4 * shift, out.data_ptr(), ny, 0)
    torch.cuda.synchronize()
    ref = oracle.lsf(oracle.psf(cube.astype(np.float64), tel, NT), tel, NT)
    assert float(np.abs(out.cpu().numpy() - ref).max()) <= 1e-5 * float(np.abs(ref).max())


@pytest.mark.parametrize("n_lambda", [331, 400])
@pytest.mark.parametrize("where", ["corner", "centre", "scattered", "none"])
def test_forward_few_occupied_spaxels(where, n_lambda):
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(4, 3, 700, 4500.0, 5375.0)
    tel = synth.Telescope(nx=61, ny=53, spaxel_size=1.0, n_lambda=n_lambda, lambda0=4600.0, dlambda=1.25)
    rng = np.random.default_rng(3)
    n = 40
    x, y = rng.uniform(-30, 30, n), rng.uniform(-26, 26, n)
    if where == "corner":
        x, y = rng.uniform(-30.5, -29.5, n), rng.uniform(25.4, 26.4, n)
    elif where == "centre":
        x, y = rng.normal(0, 0.4, n), rng.normal(0, 0.4, n)
    elif where == "none":
        x += 1000.0
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    p = synth.Particles(x=f(x), y=f(y), mass=f(np.ones(n)), age=f(rng.uniform(0.2, 12, n)),
                        Z=f(rng.uniform(1e-3, 0.03, n)), v_los=f(rng.normal(0, 100, n)))
    model = CubeModel(ssp, tel, "f32", max_particles=n)
    for _ in range(2):  # the second pass finds the first one's rows in the scratch cube
        got = model.forward(p).cpu().numpy()
        ref = oracle.forward(p, ssp, tel, n_threads=NT)
        assert float(np.abs(got - ref).max()) <= 1e-5 * max(float(np.abs(ref).max()), 1e-30)
        p.x, p.y = f(-p.x), f(-p.y)
