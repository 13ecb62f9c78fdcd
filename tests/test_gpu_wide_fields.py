"""Fields of more than 65535 * 8 spaxels along x (the argument checks allow nx * ny
up to 2^24): the convolution, the forward (16-byte rows and others) and the
gradient through both, against the oracle at the tolerances of the other parity
tests (1e-5 of the cube's maximum, 1e-4 of each gradient's)."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu
NT = 8


def test_convolve_wide():
    import torch
    from paper_2412_08265_gb300 import capi
    from paper_2412_08265_gb300.model import CubeModel
    nx, ny, nl = 524_281 + 7_000, 2, 9
    tel = synth.Telescope(nx=nx, ny=ny, spaxel_size=1.0, n_lambda=nl, lambda0=5000.0, dlambda=1.25)
    cube = np.random.default_rng(1).normal(0.0, 1.0, (ny, nx, nl)).astype(np.float32)
    d = torch.from_numpy(cube).cuda()
    out = torch.full_like(d, float("nan"))
    capi.rubix_convolve(CubeModel.c_telescope(tel), d.data_ptr(), out.data_ptr(), ny, 0)
    torch.cuda.synchronize()
    ref = oracle.lsf(oracle.psf(cube.astype(np.float64), tel, NT), tel, NT)
    assert float(np.abs(out.cpu().numpy() - ref).max()) <= 1e-5 * float(np.abs(ref).max())


@pytest.mark.parametrize("nl", [8, 9])
def test_forward_and_backward_wide(nl):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    nx = 530_000
    ssp = synth.ssp_grid(4, 3, 40, 4990.0, 5038.75)
    tel = synth.Telescope(nx=nx, ny=1, spaxel_size=1.0, n_lambda=nl, lambda0=5005.0, dlambda=1.25)
    rng = np.random.default_rng(nl)
    n = 3000
    x = rng.uniform(-0.5, 0.5, n) * nx
    x[: n // 3] = 0.5 * nx - rng.uniform(0.01, 30.0, n // 3)  # the last columns
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    p = synth.Particles(x=f(x), y=f(np.zeros(n)), mass=f(rng.uniform(0.5, 2.0, n)), age=f(rng.uniform(0.2, 12, n)),
                        Z=f(rng.uniform(1e-3, 0.03, n)), v_los=f(rng.normal(0, 100, n)))
    model = CubeModel(ssp, tel, "f32", max_particles=n)
    got = model.forward(p).cpu().numpy()
    ref = oracle.forward(p, ssp, tel, n_threads=NT)
    assert float(np.abs(got - ref).max()) <= 1e-5 * float(np.abs(ref).max())
    G = (1.0 + 0.3 * np.sin(np.arange(nx * nl) / 40.0)).astype(np.float32).reshape(1, nx, nl)
    grads = [g.cpu().numpy() for g in model.backward(torch.from_numpy(G).cuda())[:4]]
    assert model.stats()["device_error"] == 0
    G0 = oracle.psf(oracle.lsf(G.astype(np.float64), tel, NT), tel, NT)
    key = oracle.spaxel_keys(p.x.astype(np.float64), p.y.astype(np.float64), tel)
    want = oracle.gradient(key, p.v_los.astype(np.float64), p, ssp, tel, G0, n_threads=NT)
    for name, g, o in zip(("mass", "age", "Z"), grads, want):
        assert float(np.abs(g - o).max()) <= 1e-4 * float(np.abs(o).max()), name
