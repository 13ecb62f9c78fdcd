"""Requests at the edge of a server's budget. What one request may hold is what it
needs with work items of 256 particles: 85 bytes per particle, the cubes, two
partial rows per item and some integers per spaxel. A budget of that size accepts
the request (with smaller items it needs up to twice as much); its cube is the
oracle's, and the same alone and in a mix."""
import numpy as np
import pytest

import oracle
from paper_2412_08265_gb300 import synth

pytestmark = pytest.mark.gpu


def _bytes_with_items_of_256(n, side, n_lambda, n_bands):
    n_s, up = side * side, lambda b: (b + 255) // 256 * 256
    counts = -(-n // 4096) * 512
    items = n // 256
    return sum(up(b) for b in (
        *(5 * [4 * n]), 16 * n, 32 * n, 16 * n,                        # keys, order, particles, records
        4 * (2 * counts + -(-counts // 4096) + 17),                    # sort
        16 * (n_s + items + 2), 4 * (2 * items + 2) * n_lambda,        # items, partial rows
        4 * (n_s * n_bands + 2), *(4 * [4 * (n_s + 1)]), 4 * (-(-(n_s + 1) // 4096) + 17), 520,
        4 * n_s * (-(-n_lambda // 4) * 4)))                            # cube before the PSF


@pytest.mark.parametrize("n,side", [(400_000, 40), (900_000, 40), (200_000, 150), (1_000_000, 150), (3000, 8)])
def test_budget_of_one_request(n, side):
    import torch
    from paper_2412_08265_gb300.model import CubeModel
    from paper_2412_08265_gb300.serve import Server
    ssp = synth.mid_galaxy(n=1).ssp
    tel = synth.serving_telescope(side)
    p = synth.disk_3d(n, 11, inclination=0.6)
    p.x[: n // 4], p.y[: n // 4], p.z[: n // 4] = 0.0, 0.05, 0.0  # a spaxel of many items
    d = {k: torch.from_numpy(np.ascontiguousarray(getattr(p, k), dtype=np.float32)).cuda()
         for k in ("x", "y", "z", "vx", "vy", "vz", "mass", "age", "Z")}
    d.update(preprojected=False, inclination=p.inclination)
    model = CubeModel(ssp, tel, "f32", max_particles=n)
    want = model.forward(d)
    budget = _bytes_with_items_of_256(n, side, tel.n_lambda, model.stats()["n_bands"])
    cubes = []
    for copies in (1, 3):
        srv = Server(ssp, synth.serving_telescope(16), hbm_budget_bytes=budget, max_slots=4, max_batch=4)
        outs = [torch.full_like(want, float("nan")) for _ in range(copies)]
        assert srv.footprint(tel, d, outs[0]) <= budget
        torch.cuda.synchronize()
        tickets = [srv.submit(tel, d, o) for o in outs]
        for t in tickets:
            assert srv.wait(t, 120.0) == 0
        assert srv.stats()["peak_bytes"] <= budget
        cubes += outs
        srv.close()
    assert all(torch.equal(c, cubes[0]) for c in cubes[1:])
    # the same sums in another grouping: FP32 rounding of sums of up to 256 terms
    assert float((cubes[0] - want).abs().max()) <= 1e-5 * float(want.abs().max())
    # spaxels against the oracle
    s = np.array([(side // 2) * side + side // 2, side * side // 3, 1], dtype=np.int64)
    xp, yp, v = oracle.orient(p)
    ref = oracle.psf_lsf_at(oracle.deposit(oracle.spaxel_keys(xp, yp, tel), v, p, ssp, tel), tel, s)
    got = cubes[0].reshape(side * side, -1)[torch.from_numpy(s).cuda()].cpu().numpy()
    assert float(np.abs(got - ref).max()) <= 1e-5 * float(np.abs(ref).max())
