"""The deposit's slabs and the fixed-point Doppler shifts on the host (no GPU):
csrc/slab_layout.h as the library uses it, and the setup's and the deposit's
arithmetic on it replayed (double-float FP32 sums, 32-bit fixed point, the high word
of a product). For bin steps of every kind, bin centres and means, up to 8192 bins
(where the shifts are taken at bin 4096) and speeds up to and past the slab's halo:
  - a particle on the fast rounds starts, in every tile, at the FP64 node position to
    the roundings of the fixed point and of the FP32 fraction;
  - every node its rounds read lies in the slab, and neither number saturates;
  - speeds the halo covers (800 km/s) are on the fast rounds, and particles that
    approach leave them no earlier than particles that recede."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2412_08265_gb300", "csrc")

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cmath>
#include <initializer_list>
#include <random>
#include "slab_layout.h"
using namespace rubix;
constexpr double C = 299792.458;
struct DF { float hi, lo; };
static DF norm(float h, float l) { volatile float s = h + l; volatile float d = s - h; return DF{s, l - d}; }
static DF of(double x) { float h = (float)x; return DF{h, (float)(x - (double)h)}; }
static DF add(DF a, DF b) {
    volatile float s = a.hi + b.hi, z = s - a.hi, u = s - z;
    volatile float p = a.hi - u, q = b.hi - z, e = p + q, r = a.lo + b.lo;
    return norm(s, e + r);
}
static DF neg(DF a) { return DF{-a.hi, -a.lo}; }
static DF mulf(DF a, float b) { float p = a.hi * b, e = fmaf(a.hi, b, -p); return norm(p, fmaf(a.lo, b, e)); }
static DF mul(DF a, DF b) { float p = a.hi * b.hi, e = fmaf(a.hi, b.hi, -p); return norm(p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e))); }
static bool saturated = false;
static int rn(float v) {  // __float2int_rn
    if (!(std::fabs(v) < 2147483648.f)) { saturated = true; return v > 0 ? INT32_MAX : INT32_MIN; }
    return (int)std::nearbyint(v);
}
static int fixed(DF x, float scale) {
    const float v = x.hi * scale;
    const int i = rn(v);
    return (int)((uint32_t)i + (uint32_t)rn((v - (float)i) + x.lo * scale));
}
static int32_t mulhi(int32_t a, int32_t b) { return (int32_t)(((int64_t)a * b) >> 32); }

struct Grid { const char* name; int n_age, n_Z, n_ls; double ls0, ls1; int n_lambda; double l0, dl, z; };
static int bad = 0;
static double worst = 0;
static bool on_rounds(const SlabLayout& L, const Grid& G, double dls, int m, float v, long long* tiles) {
    // k_setup
    const double alpha = 1.0 / ((1.0 + G.z) * dls);
    const DF Az = of(G.dl * alpha), Ls = of(G.l0 * alpha + ((double)L.jc - 0.5 * m) * (G.dl * alpha)), invc = of(1.0 / C);
    const DF b = mulf(invc, v), q = add(DF{1.f, 0.f}, b);
    const float g0 = b.hi / q.hi;
    const DF res = add(b, neg(mulf(q, g0)));
    const DF g = norm(g0, res.hi / q.hi);
    const DF A = add(Az, neg(mul(Az, g)));
    const float sc = std::ldexp(1.f, L.fb), scg = std::ldexp(1.f, L.fb + 13);
    const DF S = neg(mul(Ls, g)), D = neg(mul(Az, g));
    const float Af = A.hi + A.lo;
    const float s_a = fmaf(-(float)L.jc, D.hi, S.hi), s_b = fmaf((float)(G.n_lambda - L.jc), D.hi, S.hi);
    if (!(Af > 0.f && Af <= L.a_max && std::fabs(D.hi * scg) < 2147483000.f && std::fmin(s_a, s_b) >= L.s_min &&
          std::fmax(s_a, s_b) <= L.s_max))
        return false;
    saturated = false;
    const int s0 = fixed(S, sc), gi = fixed(D, scg);
    const double A64 = G.dl / ((1.0 + G.z) * (1.0 + (double)v / C) * dls);
    for (int t = 0; t < L.n_tiles; ++t) {
        // k_deposit
        const int j0 = t * L.tile_w;
        const int32_t jrel = (int32_t)((uint32_t)(j0 - L.jc) << 19);
        const uint32_t p = (uint32_t)mulhi(jrel, gi) + (uint32_t)s0 + L.tile_ref[(size_t)m * L.n_tiles + t];
        const uint32_t kw = p >> L.fb;
        const float f = (float)(p & ((1u << L.fb) - 1u)) * std::ldexp(1.f, -L.fb);
        const double t64 = ((G.l0 + (j0 - 0.5 * m) * G.dl) / ((1.0 + G.z) * (1.0 + (double)v / C)) - G.ls0) / dls - L.klo[t];
        const double err = std::fabs((double)kw + (double)f - t64);
        worst = std::fmax(worst, err);
        // s0 and tile_ref rounded (1/2 unit each), g rounded (2^-14 unit per bin, up to
        // 4096 bins), the product cut off (1); the fraction rounded to FP32
        const double bound = 2.25 * std::ldexp(1.0, -L.fb) + std::ldexp(1.0, -25) + 1e-9;
        const long long top = (long long)kw + (long long)std::floor((double)f + L.last * A64) + 1;
        if (err > bound || kw >= (uint32_t)(L.slab_w - L.need) || top >= L.slab_w || saturated) {
            if (bad++ < 5)
                std::printf("%s mean %d v %g tile %d: position off %g (bound %g), nodes %u .. %lld of %d, saturated %d\n", G.name, m, v,
                            t, err, bound, kw, top, L.slab_w, saturated);
        }
        ++*tiles;
    }
    return true;
}
int main() {
    const long long entries = (232448 - 1024) / 8;
    const Grid grids[] = {
        {"muse", 50, 10, 3721, 4700, 9450, 3721, 4750, 1.25, 0},
        {"muse z", 50, 10, 3721, 4700, 9450, 3501, 4900, 1.25, 0.03},
        {"survey", 12, 6, 2000, 3600, 7400, 1000, 4001.5, 3.0, 0},
        {"4096", 20, 5, 4400, 4500, 9999, 4096, 4600, 1.25, 0},
        {"4097", 20, 5, 4400, 4500, 9999, 4097, 4600, 1.25, 0},
        {"8192 near 1", 20, 5, 8600, 4500, 9999, 8192, 4600, 0.635, 0},
        {"8192 above 1", 20, 5, 8600, 4500, 9999, 8192, 4600, 0.6397, 0},
        {"8192 below 1", 12, 4, 8600, 4500, 9999, 8192, 4600, 0.5, 0.1},
        {"8192 coarse", 12, 4, 16384, 4500, 21000, 8192, 4600, 1.9, 0},
        {"8192 fine", 1, 1, 1000, 4500, 9999, 8192, 4600, 0.6, 0},
        {"coarse", 9, 5, 1801, 4500, 6750, 700, 4550.3, 2.4, 0},
    };
    std::mt19937 rng(1);
    std::uniform_real_distribution<float> U(-2500.f, 2500.f);
    long long tiles = 0;
    for (const Grid& G : grids) {
        const double dls = (G.ls1 - G.ls0) / (G.n_ls - 1);
        const SlabLayout L = slab_layout(G.n_age, G.n_Z, G.ls0, dls, G.n_lambda, G.l0, G.dl, G.z, entries, 800.0 / C, 0);
        if (L.slab_w == 0 || L.jc != (G.n_lambda > 4096 ? 4096 : 0)) { std::printf("%s: no slab\n", G.name); return 2; }
        for (int m = 0; m < 2; ++m) {
            for (int i = 0; i < 4000; ++i) on_rounds(L, G, dls, m, U(rng), &tiles);
            for (float v : {0.f, 1e-3f, -1e-3f, 799.9f, -799.9f})
                if (!on_rounds(L, G, dls, m, v, &tiles)) { std::printf("%s mean %d: %g km/s off the rounds\n", G.name, m, v); return 3; }
            // the first speeds off the rounds, on both sides
            int up = 800, down = 800;
            while (up < 5000 && on_rounds(L, G, dls, m, (float)up, &tiles)) up += 5;
            while (down < 5000 && on_rounds(L, G, dls, m, (float)-down, &tiles)) down += 5;
            if (down < 0.97 * up) { std::printf("%s mean %d: receding to %d km/s, approaching to %d\n", G.name, m, up, down); bad++; }
        }
    }
    std::printf("%lld tiles, worst position error %g\n", tiles, worst);
    return bad ? 1 : 0;
}
"""


def test_fixed_point_shifts_and_slabs(tmp_path):
    src, exe = tmp_path / "slab.cpp", tmp_path / "slab"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
