"""The one-launch scans when every wait in them runs out (RUBIX_FAULT_SCAN keeps the
blocks from publishing their sums). 1, the sort's: each block counts the tiles
before its own itself; order, offsets, cube and gradients are bit for bit those
of the scans that wait, and nothing is reported. 2, the work items': items are
lost, which the device error word says; forward and gradient still stay within
their buffers, and the context serves the next model."""
import os

import numpy as np
import pytest

from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nx,ny", [(700, 3, 2), (40_000, 61, 53), (300_000, 150, 150)])
def test_expired_scan_waits_change_nothing(n, nx, ny):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(12, 5, 200, 4500.0, 4748.75)
    tel = synth.Telescope(nx=nx, ny=ny, spaxel_size=0.3, n_lambda=65, lambda0=4560.0, dlambda=1.25)
    rng = np.random.default_rng(n)
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    x, y = rng.uniform(-0.16, 0.16, n) * nx, rng.uniform(-0.16, 0.16, n) * ny
    x[: n // 2], y[: n // 2] = 0.05, 0.05  # one spaxel of many work items
    p = synth.Particles(x=f(x), y=f(y), mass=f(rng.uniform(0.5, 2.0, n)), age=f(np.exp(rng.uniform(-2.0, 2.5, n))),
                        Z=f(np.exp(rng.uniform(-9.0, -3.0, n))), v_los=f(rng.normal(0.0, 150.0, n)))
    G = torch.from_numpy(rng.standard_normal((ny, nx, 65)).astype(np.float32)).cuda()
    got = {}
    for fault in ("0", "1"):
        os.environ["RUBIX_FAULT_SCAN"] = fault
        try:
            model = CubeModel(ssp, tel, "f32", max_particles=n)
        finally:
            del os.environ["RUBIX_FAULT_SCAN"]
        for _ in range(2):
            cube = model.forward(p)
            got[fault] = [t.cpu() for t in (cube, *model.sorted(), *model.backward(G)[:4])]
        assert model.stats()["device_error"] == 0
        model.close()
    for a, b in zip(got["0"], got["1"]):
        assert torch.equal(a, b)


@pytest.mark.parametrize("n_bands_grid", [(12, 5), (3, 2)])  # several age bands, and one
def test_expired_item_scan_is_reported(n_bands_grid):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    ssp = synth.ssp_grid(*n_bands_grid, 200, 4500.0, 4748.75)
    tel = synth.Telescope(nx=61, ny=53, spaxel_size=0.3, n_lambda=65, lambda0=4560.0, dlambda=1.25)
    rng = np.random.default_rng(8)
    n = 30_000
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    p = synth.Particles(x=f(rng.uniform(-9, 9, n)), y=f(rng.uniform(-8, 8, n)), mass=f(rng.uniform(0.5, 2.0, n)),
                        age=f(np.exp(rng.uniform(-2.0, 2.5, n))), Z=f(np.exp(rng.uniform(-9.0, -3.0, n))),
                        v_los=f(rng.normal(0.0, 150.0, n)))
    G = torch.ones((53, 61, 65), device="cuda")
    ref = CubeModel(ssp, tel, "f32", max_particles=n)
    want = ref.forward(p).clone()
    os.environ["RUBIX_FAULT_SCAN"] = "2"
    try:
        model = CubeModel(ssp, tel, "f32", max_particles=n)
    finally:
        del os.environ["RUBIX_FAULT_SCAN"]
    model.forward(p)
    model.backward(G)
    torch.cuda.synchronize()
    assert model.stats()["device_error"] & 1
    model.close()
    assert torch.equal(ref.forward(p), want) and ref.stats()["device_error"] == 0
