"""Grids of the passes after the deposit (csrc/conv_layout.h, host arithmetic;
compiled and run on the host, no GPU). The row split of the fused PSF/LSF kernel is
the best of all splits of the rows into equal parts, and it is found in a number of
steps that stays small however many rows there are (every launch asks for it). The
row pass has a warp for every unit of work up to its eight blocks per SM, also
where few spaxels hold many particles."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2412_08265_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "conv_layout.h"
using namespace rubix;
// every split into k parts, in order
static int every_split(int ny, int rp, long long columns, long long slots, int max_ty) {
    int best = ny;
    double cost = 1e300;
    for (int k = 1; k <= ny; ++k) {
        const int ty = (ny + k - 1) / k;
        if (ty > max_ty) continue;
        if (ty < 2 * rp && best <= max_ty) break;
        const long long ctas = columns * ((ny + ty - 1) / ty);
        const double c = (double)((ctas + slots - 1) / slots) * (ty + 2 * rp + 4);
        if (c < cost * 0.999) { cost = c; best = ty; }
    }
    return best;
}
int main() {
    for (int ny : {1, 2, 3, 7, 25, 81, 150, 300, 599, 600, 601, 1200, 1201, 4096, 65535, 1 << 20})
        for (int rp : {0, 2, 3, 4})
            for (long long columns : {1ll, 2ll, 36ll, 627ll, 1292ll, 40000ll, 1ll << 21})
                for (long long slots : {4ll, 592ll, 608ll}) {
                    int tried = 0;
                    const int ty = rows_per_cta(ny, rp, columns, slots, 600, &tried);
                    const int want = every_split(ny, rp, columns, slots, 600);
                    if (ty != want) { std::printf("ny %d rp %d: %d, best %d\n", ny, rp, ty, want); return 1; }
                    // the distinct heights up to 600 rows
                    if (tried > 600) { std::printf("ny %d rp %d: %d splits tried\n", ny, rp, tried); return 2; }
                }
    return 0;
}
"""


ROWS = r"""
#include <cstdio>
#include <initializer_list>
#include "conv_layout.h"
using namespace rubix;
int main() {
    for (long long n_s : {1ll, 5ll, 64ll, 625ll, 1600ll, 22500ll, 1ll << 24})
        for (long long max_split : {0ll, 1ll, 3ll, 100ll, 4000ll, 80000ll, 1ll << 22})
            for (int n_lambda : {1, 128, 129, 1000, 3721, 8192})
                for (int n_sm : {1, 152}) {
                    const long long blocks = row_blocks(n_s, max_split, n_lambda, n_sm), full = 8ll * n_sm;
                    const long long split = max_split < n_s ? max_split : n_s;
                    const long long units = split * ((n_lambda + kCombineBins - 1) / kCombineBins);
                    const long long warps = blocks * (kRowThreads / 32);
                    if (blocks < 1 || blocks > full) return 1;
                    if (blocks < full && (warps < n_s || warps < units)) {
                        std::printf("%lld spaxels, %lld split, %d bins: %lld blocks\n", n_s, max_split, n_lambda, blocks);
                        return 2;
                    }
                }
    return 0;
}
"""


def _run(tmp_path, program):
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(program)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_row_pass_has_a_warp_per_unit(tmp_path):
    _run(tmp_path, ROWS)


def test_row_split_is_the_best_and_cheap_to_find(tmp_path):
    _run(tmp_path, PROGRAM)
