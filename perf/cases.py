"""The work this library is measured on: forward models, gradient steps, the
convolution of a row block and a burst of served requests, each through the
public entry points (CubeModel, RubixCube, Server, rubix_convolve), over the
sizes, data types and options users run.

    listed()            the cases, a dict of plain values each
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the state a user's program holds before the call
    run(state)          one pass, returning its outputs whole
    work(case)          bytes and operations one pass cannot do without
    exact(case, seed)   the outputs in 64 bits, by plain torch
"""
from __future__ import annotations

import functools
import math
from dataclasses import replace

import numpy as np
import torch

from paper_2412_08265_gb300 import capi, synth
from paper_2412_08265_gb300.model import CubeModel, RubixCube
from paper_2412_08265_gb300.serve import Server

C_KMS = 299792.458
PSF_FWHM, LSF_SIGMA = 1.5, 1.2


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _case(name, kind, n, nx, ny, field, grid="muse", **kw):
    """`field`: side of the field along x in kpc; `grid`: wavelength grids."""
    c = dict(name=name, kind=kind, n=n, nx=nx, ny=ny, spaxel=field / nx, grid=grid, galaxy="disk", dtype="f32",
             resample=0, z=0.0, incl=0.0, azim=0.0, pa=0.0, s2n=0.0, requests=0)
    c.update(kw)
    return c


def listed():
    return [
        # one small galaxy on a survey IFU whose bins are coarser than the
        # templates' (12x6x2000 grid, 3 A bins): the smallest call, latency
        _case("small", "forward", 10_000, 25, 25, 12.5, "survey"),
        # one iteration of a fit to a small galaxy: forward and gradients
        _case("small_step", "step", 10_000, 25, 25, 12.5, "survey"),
        # a small galaxy in a wide field (most of the field empty), the light
        # end of a survey's requests
        _case("sparse_field", "forward", 10_000, 300, 300, 60.0),
        # the mid-size galaxy: 50x10x3721 FP32 templates, MUSE-like bins
        _case("mid", "forward", 1_000_000, 150, 150, 30.0),
        # the same with flux-conserving bin means
        _case("mid_means", "forward", 1_000_000, 150, 150, 30.0, resample=1),
        # one iteration of a fit to the mid-size galaxy
        _case("mid_step", "step", 1_000_000, 150, 150, 30.0),
        # a simulated galaxy oriented by three angles, placed at a redshift,
        # observed with noise, FP16 templates, odd sizes
        _case("oriented_z", "forward", 300_000, 101, 97, 30.3, "muse_z", galaxy="disk3d", dtype="f16", z=0.03,
              incl=0.9, azim=0.4, pa=-0.7, s2n=40.0),
        # fitting the orientation of a galaxy with bin means (gradients of the
        # shared parameters too)
        _case("oriented_step", "step", 200_000, 75, 75, 30.0, galaxy="disk3d", resample=1, incl=0.7, azim=0.3, pa=0.2),
        # many particles on the survey grid (bins coarser than the templates')
        _case("survey", "forward", 500_000, 72, 72, 18.0, "survey"),
        # the large galaxy: bulge and disk, 2e7 particles, BF16 templates
        _case("large", "forward", 20_000_000, 300, 300, 30.0, galaxy="bulge", dtype="bf16"),
        # PSF and LSF of one shard's rows (row-sharded galaxies)
        _case("convolve", "convolve", 0, 150, 81, 30.0),
        # a burst of requests through the server
        _case("serve", "serve", 1_000_000, 150, 150, 30.0, galaxy="disk3d", requests=12),
    ]


def draw(rng):
    def logu(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["forward"] * 5 + ["step"] * 3 + ["convolve", "serve"])
    grid = rng.choice(["muse"] * 3 + ["muse_z", "survey"])
    galaxy = rng.choice(["disk", "disk3d", "bulge"])
    dtype = rng.choice(["f32", "f32", "bf16", "f16"])
    nx = logu(25, 300)
    ny = max(20, min(300, nx + rng.randint(-9, 9)))
    kw = dict(galaxy=galaxy, dtype=dtype, resample=rng.choice([0, 0, 1]))
    if grid == "muse_z":
        kw["z"] = rng.uniform(0.015, 0.03)
    if galaxy == "disk3d":
        kw.update(incl=rng.uniform(0.0, 1.5), azim=rng.uniform(-3.0, 3.0), pa=rng.uniform(-3.0, 3.0))
    if kind == "forward":
        n = logu(1e4, 1e7 if grid == "muse" else 1e6)
        kw["s2n"] = rng.choice([0.0, 0.0, 0.0, 50.0])
    elif kind == "step":
        n = logu(1e4, 1e6 if grid == "muse" else 3e5)
    elif kind == "serve":
        n, grid, kw["z"], kw["galaxy"], kw["requests"] = logu(1e5, 2e6), "muse", 0.0, "disk3d", rng.randint(4, 16)
        kw.update(incl=0.0, azim=0.0, pa=0.0)
    else:
        n, kw = 0, {}
        ny = rng.randint(max(8, nx // 8), nx)
    c = _case("", kind, n, nx, ny, rng.uniform(12.0, 30.0) if grid == "survey" else rng.uniform(24.0, 60.0), grid, **kw)
    del c["name"]
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _ssp(grid):
    if grid == "survey":
        return synth.ssp_grid(12, 6, 2000, 3600.0, 7400.0)
    return synth.ssp_grid(50, 10, 3721, 4700.0, 9450.0)


def _telescope(case):
    wl = {"survey": (1000, 4001.5, 3.0), "muse": (3721, 4750.0, 1.25), "muse_z": (3501, 4900.0, 1.25)}[case["grid"]]
    return synth.Telescope(nx=case["nx"], ny=case["ny"], spaxel_size=case["spaxel"], n_lambda=wl[0], lambda0=wl[1],
                           dlambda=wl[2], psf_fwhm=PSF_FWHM, lsf_sigma=LSF_SIGMA, z_cosmo=case["z"],
                           resample=case["resample"])


def _populations(n, gen, dev):
    def u():
        return torch.rand(n, generator=gen, device=dev)

    age = torch.exp(math.log(0.1) + (math.log(13.5) - math.log(0.1)) * u())
    Z = torch.exp(math.log(1e-4) + (math.log(0.04) - math.log(1e-4)) * u())
    mass = torch.exp(math.log(1e5) + 0.5 * torch.randn(n, generator=gen, device=dev))
    return dict(mass=mass, age=age, Z=Z)


def _galaxy(kind, n, seed, dev):
    """Particles of one galaxy, drawn on the GPU: the disk, bulge and 3-D disk
    of the package's synthetic workloads."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    if kind == "disk3d":
        return dict(synth.disk_3d_device(n, int(seed), dev), preprojected=False)
    nb = int(0.3 * n) if kind == "bulge" else 0
    nd = n - nb

    def u(m):
        return torch.rand(m, generator=gen, device=dev).clamp_(1e-7, 1.0 - 1e-6)

    R = -3.0 * (torch.log(u(nd)) + torch.log(u(nd)))
    phi = 2.0 * math.pi * u(nd)
    x, y = R * torch.cos(phi), R * torch.sin(phi)
    v = 200.0 * math.sin(math.pi / 4) * torch.tanh(R / 2.0) * torch.cos(phi) \
        + 50.0 * torch.randn(nd, generator=gen, device=dev)
    if nb:
        s = torch.sqrt(u(nb))
        r = s / (1.0 - s)
        ct = 2.0 * u(nb) - 1.0
        rs, ph = r * torch.sqrt(1.0 - ct * ct), 2.0 * math.pi * u(nb)
        x, y = torch.cat([rs * torch.cos(ph), x]), torch.cat([rs * torch.sin(ph), y])
        v = torch.cat([150.0 * torch.randn(nb, generator=gen, device=dev), v])
    return dict(_populations(n, gen, dev), x=x, y=y, v_los=v, preprojected=True)


def _requests(case, seed):
    """(telescope, seed, particle count, inclination) of each request of a
    burst: counts log-uniform over two decades, cubes of 40 spaxels and more."""
    rng = np.random.Generator(np.random.PCG64(case["requests"]))
    out = []
    for i in range(case["requests"]):
        n = max(1000, int(case["n"] * math.exp(-rng.uniform(0.0, math.log(100.0)))))
        side = int(rng.integers(40, max(case["nx"], 60) + 1))
        tel = replace(_telescope(case), nx=side, ny=side, spaxel_size=0.2)
        out.append((tel, int(seed) * 1000 + i, n, float(rng.uniform(0.0, 0.5 * math.pi))))
    return out


def _particles(case, seed, dev):
    p = _galaxy(case["galaxy"], case["n"], seed, dev)
    if case["galaxy"] == "disk3d":
        p.update(inclination=case["incl"], azimuth=case["azim"], position_angle=case["pa"])
    return p


def _cotangent(shape, seed, dev):
    """dL/dcube of a chi-square-like loss: noise around a smooth positive part."""
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 77)
    return 0.3 + torch.randn(shape, generator=gen, device=dev)


def _block(case, seed, dev):
    """Deposited rows of a shard before its PSF: positive, falling outwards."""
    tel = _telescope(case)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) + 5)
    y = torch.linspace(-1, 1, tel.ny, device=dev)[:, None, None]
    x = torch.linspace(-1, 1, tel.nx, device=dev)[None, :, None]
    return 1e6 * torch.exp(-4.0 * torch.sqrt(x * x + y * y)) * torch.rand((tel.ny, tel.nx, tel.n_lambda),
                                                                            generator=gen, device=dev)


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    kind, tel, ssp = case["kind"], _telescope(case), _ssp(case["grid"])
    st = dict(kind=kind, tel=tel, dev=dev)
    if kind == "convolve":
        st["cube"] = _block(case, seed, dev)
        st["c_tel"] = CubeModel.c_telescope(tel)
        return st
    if kind == "serve":
        st["server"] = Server(ssp, tel, 32 << 30, max_slots=8, max_batch=16, template_dtype=case["dtype"])
        st["jobs"] = []
        for rt, s, n, incl in _requests(case, seed):
            p = dict(_galaxy("disk3d", n, s, dev), inclination=incl, azimuth=0.0, position_angle=0.0)
            st["jobs"].append((rt, p, torch.empty((rt.ny, rt.nx, rt.n_lambda), device=dev)))
        torch.cuda.synchronize()
        return st
    st["model"] = CubeModel(ssp, tel, case["dtype"], max_particles=case["n"])
    st["p"] = _particles(case, seed, dev)
    st["s2n"], st["seed"] = case["s2n"], int(seed)
    if kind == "step":
        st["G"] = _cotangent(st["model"].cube_shape, seed, dev)
        st["shared"] = case["galaxy"] == "disk3d"
        if not st["shared"]:
            st["leaf"] = [st["p"][k].requires_grad_() for k in ("mass", "age", "Z", "v_los")]
    return st


def run(state):
    kind = state["kind"]
    if kind == "convolve":
        out = torch.empty_like(state["cube"])
        capi.rubix_convolve(state["c_tel"], state["cube"].data_ptr(), out.data_ptr(), state["tel"].ny,
                            torch.cuda.current_stream(state["dev"]).cuda_stream)
        return out
    if kind == "serve":
        srv = state["server"]
        tickets = [srv.submit(tel, p, out) for tel, p, out in state["jobs"]]
        for t in tickets:
            capi.check(srv.wait(t))
        return [out for _, _, out in state["jobs"]]
    model, p = state["model"], state["p"]
    if kind == "forward":
        return model.forward(p, noise_seed=state["seed"], noise_s2n=state["s2n"])
    if state["shared"]:
        # a fit of the orientation: float32 parameters, so float32 gradients
        cube = model.forward(p)
        dm, da, dz, dv, glob = model.backward(state["G"], want_global=True)
        return [cube, dm, da, dz, dv, glob.float()]
    cube = RubixCube.apply(*state["leaf"], p["x"], p["y"], model)
    return [cube.detach(), *torch.autograd.grad(cube, state["leaf"], grad_outputs=state["G"])]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _in_field(galaxy, wx, wy, incl):
    """Share of a galaxy's particles inside a wx x wy kpc field."""
    rng = np.random.Generator(np.random.PCG64(1))
    m = 200_000
    R, phi = rng.gamma(2.0, 3.0, m), rng.uniform(0.0, 2.0 * math.pi, m)
    x, y = R * np.cos(phi), R * np.sin(phi)
    if galaxy == "disk3d":
        y = y * math.cos(incl) - rng.laplace(0.0, 0.3, m) * math.sin(incl)
    if galaxy == "bulge":
        nb = int(0.3 * m)
        s = np.sqrt(rng.uniform(0.0, 1.0, nb))
        r, ct, ph = s / np.maximum(1.0 - s, 1e-9), rng.uniform(-1.0, 1.0, nb), rng.uniform(0.0, 2.0 * math.pi, nb)
        x[:nb], y[:nb] = r * np.sqrt(1 - ct * ct) * np.cos(ph), r * np.sqrt(1 - ct * ct) * np.sin(ph)
    return float(np.mean((np.abs(x) < wx / 2) & (np.abs(y) < wy / 2)))


def _work_forward(tel, n, galaxy, incl, ssp, dtype):
    vox = tel.nx * tel.ny * tel.n_lambda
    deposits = n * _in_field(galaxy, tel.nx * tel.spaxel_size, tel.ny * tel.spaxel_size, incl) * tel.n_lambda
    rp = math.ceil(4.0 * tel.psf_fwhm / (2.0 * math.sqrt(2.0 * math.log(2.0))))
    rl = math.ceil(4.0 * tel.lsf_sigma / tel.dlambda)
    b = n * 4 * (9 if galaxy == "disk3d" else 6) + 4 * vox + ssp.spectra.size * (4 if dtype == "f32" else 2)
    # per deposit: four corners at two wavelength neighbours, a multiply-add each
    return b, 16.0 * deposits + 2.0 * vox * (2 * (2 * rp + 1) + 2 * rl + 1), deposits


def work(case):
    tel, ssp = _telescope(case), _ssp(case["grid"])
    if case["kind"] == "convolve":
        b, f, _ = _work_forward(tel, 0, "disk", 0.0, ssp, "f32")
        vox = tel.nx * tel.ny * tel.n_lambda
        return {"bytes": 8.0 * vox, "flops": f}
    if case["kind"] == "serve":
        total = [0.0, 0.0]
        for rt, _, n, incl in _requests(case, 0):
            b, f, _ = _work_forward(rt, n, "disk3d", round(incl, 1), ssp, case["dtype"])
            total[0] += b
            total[1] += f
        return {"bytes": total[0], "flops": total[1]}
    b, f, deposits = _work_forward(tel, case["n"], case["galaxy"], case["incl"], ssp, case["dtype"])
    if case["kind"] == "step":
        # the gradient cube read, four gradients written; per deposit the four
        # corners interpolated and two multiply-adds into each corner's sums
        b += 4 * tel.nx * tel.ny * tel.n_lambda + 16 * case["n"]
        f += f - 16.0 * deposits + 24.0 * deposits
    return {"bytes": float(b), "flops": float(f)}


# --------------------------------------------------------------------------
# the outputs in 64 bits
# --------------------------------------------------------------------------
def _conv64(cube, tel):
    def gauss(sigma):
        r = math.ceil(4.0 * sigma)
        w = [math.exp(-d * d / (2.0 * sigma * sigma)) for d in range(-r, r + 1)]
        return r, [v / sum(w) for v in w]

    rp, gp = gauss(tel.psf_fwhm / (2.0 * math.sqrt(2.0 * math.log(2.0))))
    rl, gl = gauss(tel.lsf_sigma / tel.dlambda)
    for dim, r, w in ((0, rp, gp), (1, rp, gp), (2, rl, gl)):
        size = cube.shape[dim]
        out = torch.zeros_like(cube)
        for d in range(-r, r + 1):
            m = size - abs(d)
            if m > 0:
                out.narrow(dim, max(0, -d), m).add_(cube.narrow(dim, max(0, d), m), alpha=w[d + r])
        cube = out
    return cube


def _orientation(incl, azim, pa):
    ca, sa, ci, si, cq, sq = (f(a) for a in (azim, incl, pa) for f in (math.cos, math.sin))
    R = [cq * ca - sq * (ci * sa), -(cq * sa) - sq * (ci * ca), sq * si,
         sq * ca + cq * (ci * sa), cq * (ci * ca) - sq * sa, -(cq * si), si * sa, si * ca, ci]
    return R, (ci * sa, ci * ca, -si), (si * ca, -(si * sa))


class _Exact:
    """The forward model and its gradients in float64, particles in chunks."""

    def __init__(self, tel, ssp, dtype, p, dev):
        self.tel, self.ssp, self.dev = tel, ssp, dev
        sp = torch.from_numpy(np.ascontiguousarray(ssp.spectra)).to(dev).float()
        if dtype != "f32":
            sp = sp.to(torch.bfloat16 if dtype == "bf16" else torch.float16)
        n_age, n_Z, n_ls = sp.shape
        # templates are zero outside their range: one zero node on each side
        self.T = torch.zeros((n_age * n_Z, n_ls + 2), dtype=torch.float64, device=dev)
        self.T[:, 1:-1] = sp.double().reshape(n_age * n_Z, n_ls)
        self.n_Z = n_Z
        self.la = torch.from_numpy(ssp.log10_age_nodes).to(dev)
        self.lz = torch.from_numpy(ssp.log10_Z_nodes).to(dev)
        d = {k: v.detach().double() for k, v in p.items() if isinstance(v, torch.Tensor)}
        self.dvi = self.dva = None
        if p["preprojected"]:
            x, y, v = d["x"], d["y"], d["v_los"]
        else:
            R, Di, Da = _orientation(p["inclination"], p["azimuth"], p["position_angle"])
            x = (R[0] * d["x"] + R[1] * d["y"]) + R[2] * d["z"]
            y = (R[3] * d["x"] + R[4] * d["y"]) + R[5] * d["z"]
            v = (R[6] * d["vx"] + R[7] * d["vy"]) + R[8] * d["vz"]
            self.dvi = Di[0] * d["vx"] + Di[1] * d["vy"] + Di[2] * d["vz"]
            self.dva = Da[0] * d["vx"] + Da[1] * d["vy"]
        ix = torch.floor((x - (-0.5 * tel.nx) * tel.spaxel_size) * (1.0 / tel.spaxel_size)).long()
        iy = torch.floor((y - (-0.5 * tel.ny) * tel.spaxel_size) * (1.0 / tel.spaxel_size)).long()
        self.inside = torch.nonzero((ix >= 0) & (ix < tel.nx) & (iy >= 0) & (iy < tel.ny)).flatten()
        self.key = (iy * tel.nx + ix)[self.inside]
        self.q = [t[self.inside] for t in (d["mass"], d["age"], d["Z"], v)]
        self.n = x.numel()
        self.j = torch.arange(tel.n_lambda + 1, dtype=torch.float64, device=dev)

    @staticmethod
    def _cell(q, nodes):
        i = (torch.searchsorted(nodes, q.detach(), right=True) - 1).clamp_(0, nodes.numel() - 2)
        return i, ((q - nodes[i]) / (nodes[i + 1] - nodes[i])).clamp(0.0, 1.0)

    def spectra(self, mass, age, Z, v):
        tel, ssp, m = self.tel, self.ssp, self.T.shape[1]
        ia, ta = self._cell(torch.log10(age), self.la)
        iz, tz = self._cell(torch.log10(Z), self.lz)
        c = ia * self.n_Z + iz
        M = (mass * (1 - ta) * (1 - tz))[:, None] * self.T[c]
        M = M + (mass * ta * (1 - tz))[:, None] * self.T[c + self.n_Z]
        M = M + (mass * (1 - ta) * tz)[:, None] * self.T[c + 1]
        M = M + (mass * ta * tz)[:, None] * self.T[c + self.n_Z + 1]
        dop = ((1.0 + tel.z_cosmo) * (1.0 + v / C_KMS))[:, None]
        j = self.j[None, :] - 0.5 if tel.resample else self.j[None, :-1]
        t = ((tel.lambda0 + j * tel.dlambda) / dop - ssp.lambda0) / ssp.dlambda + 1.0
        k = torch.floor(t.detach()).long().clamp_(0, m - 2)
        f = t - k
        f = torch.where((f.detach() >= 0) & (f.detach() <= 1), f, f.detach().clamp(0.0, 1.0))
        a = M.gather(1, k)
        s = M.gather(1, k + 1) - a
        if not tel.resample:
            return a + f * s
        C = torch.cumsum(M, 1) - 0.5 * M  # C[k + 1] - C[k] = the trapezoid between nodes k and k + 1
        F = C.gather(1, k) + f * a + 0.5 * f * f * s
        return (F[:, 1:] - F[:, :-1]) / (t[:, 1:] - t[:, :-1])

    def cube(self):
        tel = self.tel
        out = torch.zeros((tel.ny * tel.nx, tel.n_lambda), dtype=torch.float64, device=self.dev)
        with torch.no_grad():
            for b in range(0, self.key.numel(), 8192):
                s = slice(b, b + 8192)
                out.index_add_(0, self.key[s], self.spectra(*(t[s] for t in self.q)))
            return _conv64(out.view(tel.ny, tel.nx, tel.n_lambda), tel)

    def gradients(self, G):
        tel = self.tel
        G0 = _conv64(G.double(), tel).view(tel.ny * tel.nx, tel.n_lambda)
        g = [torch.zeros(self.n, dtype=torch.float64, device=self.dev) for _ in range(4)]
        for b in range(0, self.key.numel(), 4096):
            s = slice(b, b + 4096)
            leaf = [t[s].clone().requires_grad_() for t in self.q]
            loss = (self.spectra(*leaf) * G0[self.key[s]]).sum()
            for full, part in zip(g, torch.autograd.grad(loss, leaf)):
                full[self.inside[s]] = part
        return g


def exact(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    tel, ssp = _telescope(case), _ssp(case["grid"])
    if case["kind"] == "convolve":
        return _conv64(_block(case, seed, dev).double(), tel)
    if case["s2n"] > 0.0:
        return None  # the noise is defined by its random stream
    if case["kind"] == "serve":
        got = []
        for rt, s, n, incl in _requests(case, seed):
            p = dict(_galaxy("disk3d", n, s, dev), inclination=incl, azimuth=0.0, position_angle=0.0)
            got.append(_Exact(rt, ssp, case["dtype"], p, dev).cube())
        return got
    p = _particles(case, seed, dev)
    E = _Exact(tel, ssp, case["dtype"], p, dev)
    if case["kind"] == "forward":
        return E.cube()
    g = E.gradients(_cotangent((tel.ny, tel.nx, tel.n_lambda), seed, dev))
    out = [E.cube(), *g]
    if case["galaxy"] == "disk3d":
        dv = g[3]
        out.append(torch.stack([dv.sum(), (p["mass"].double() * g[0]).sum(), (dv * E.dvi).sum(), (dv * E.dva).sum()]))
    return out
