"""Forward and backward cases that take the rounds for every bin step dt/dj, run with
one build of the library and saved for comparison with another: the shuffle rounds
below 1, the two-read rounds just above 1 and at any step, the rounds that gather
consecutive nodes (CTAs with many work items), the two-read edges of bin means in all
three kinds, more than 4096 bins, shifts past the slab's halo (some tiles, then all),
16-bit templates, grids of one age or one metallicity.

    python tests/_debug_rounds.py debug|release OUT.npz

Run as a separate process by tests/test_gpu_debug_rounds.py: a process loads one
build of the library only."""
import os
import sys

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
sys.path.insert(0, ROOT)

# name: (ages, metallicities, dt/dj, bins, particles, top speed km/s, resample, dtype)
CASES = {
    "below1": (9, 5, 0.95, 1500, 6000, 700.0, 0, "f32"),
    "below1_means": (9, 5, 0.95, 1500, 6000, 700.0, 1, "f32"),
    "half": (9, 5, 0.51, 1999, 6000, 700.0, 0, "f16"),
    "above1_kind0": (9, 5, 1.0012, 1500, 6000, 700.0, 0, "f32"),
    "above1_kind0_means": (9, 5, 1.0012, 1500, 6000, 700.0, 1, "f32"),
    "two_read": (9, 5, 1.6, 950, 6000, 700.0, 0, "bf16"),
    "two_read_means": (9, 5, 1.6, 950, 6000, 700.0, 1, "f32"),
    "gather": (9, 5, 1.58, 950, 400_000, 700.0, 0, "f32"),
    "coarse": (9, 5, 2.7, 600, 6000, 700.0, 0, "f32"),
    "coarse_means": (9, 5, 2.7, 600, 6000, 700.0, 1, "f32"),
    "fine": (9, 5, 0.3, 1999, 6000, 700.0, 0, "f32"),
    "many_bins": (9, 4, 0.99, 8192, 3000, 700.0, 0, "f32"),
    "many_bins_means": (9, 4, 1.6, 8192, 3000, 700.0, 1, "f32"),
    "fast_below1": (9, 5, 0.95, 1500, 6000, 3000.0, 0, "bf16"),
    "fast_above1": (9, 5, 1.6, 950, 6000, 3000.0, 0, "f32"),
    "fast_means": (9, 5, 0.7, 1500, 3000, 3000.0, 1, "f32"),
    "fast_kind0": (30, 10, 0.98, 2500, 6000, 2500.0, 0, "f32"),
    "one_age": (1, 4, 0.8, 700, 3000, 700.0, 0, "f32"),
    "one_metallicity": (6, 1, 1.3, 700, 3000, 700.0, 1, "bf16"),
}


def _case(name):
    from paper_2412_08265_gb300 import synth
    n_age, n_Z, a0, n_lambda, n, v_max, resample, dtype = CASES[name]
    n_ls = min(16384, int(n_lambda * a0) + 150)
    ssp = synth.ssp_grid(n_age, n_Z, n_ls, 4500.0, 4500.0 + 1.25 * (n_ls - 1))
    tel = synth.Telescope(nx=11, ny=9, spaxel_size=0.7, n_lambda=n_lambda, lambda0=4570.3, dlambda=1.25 * a0,
                          resample=resample)
    rng = np.random.default_rng(list(CASES).index(name))
    f = lambda a: np.ascontiguousarray(a, dtype=np.float32)
    p = synth.Particles(x=f(rng.normal(0, 2.0, n)), y=f(rng.normal(0, 2.0, n)), mass=f(np.exp(rng.normal(0, 0.5, n))),
                        age=f(np.exp(rng.uniform(np.log(0.08), np.log(15), n))),
                        Z=f(np.exp(rng.uniform(np.log(8e-5), np.log(0.05), n))), v_los=f(rng.uniform(-v_max, v_max, n)))
    return ssp, tel, p, dtype


def run(debug: bool, path: str):
    import torch
    from paper_2412_08265_gb300 import build as B
    from paper_2412_08265_gb300 import capi
    capi.load(B.build(debug=debug))
    from paper_2412_08265_gb300.model import CubeModel
    torch.cuda.set_device(0)
    res = {}
    for name in CASES:
        ssp, tel, p, dtype = _case(name)
        model = CubeModel(ssp, tel, dtype, max_particles=p.n)
        cube = model.forward(p)
        G = torch.from_numpy(np.random.default_rng(5).standard_normal(model.cube_shape).astype(np.float32)).cuda()
        grads = model.backward(G)[:4]
        torch.cuda.synchronize()
        st = model.stats()
        for k, t in zip(("cube", "dm", "dage", "dZ", "dv"), (cube, *grads)):
            res[f"{name}/{k}"] = t.cpu().numpy()
        res[f"{name}/err"] = np.array([st["device_error"]], dtype=np.int64)
        res[f"{name}/slow"] = np.array([st["slow_particle_tiles"]], dtype=np.int64)
        model.close()
    np.savez(path, **res)


if __name__ == "__main__":
    run(sys.argv[1] == "debug", sys.argv[2])
