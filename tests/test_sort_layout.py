"""The radix sort's scratch (csrc/sort_layout.h, host arithmetic): a plan is
sized once for its capacity and then sorts any number of particles up to it, in
tiles whose size changes with the number of particles, with keys of any width.
The scratch of a capacity must hold the layout of every smaller call. Compiled
and run on the host; no GPU."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2412_08265_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "sort_layout.h"
using namespace rubix;
int main() {
    long long checked = 0;
    for (int n_sm : {1, 20, 132, 148, 152, 160}) {
        const long long s = short_tile_keys(n_sm);
        const long long caps[] = {1, 65536, s - 1, s, s + 1, s + s / 16, 2 * s, 3 * s, 4 * s, 5 * s, 40 * s, 1ll << 30,
                                  2000000, 4000000, 1200000 + 1200000 / 8};
        for (long long cap : caps) {
            if (cap < 1 || cap > (1ll << 30)) continue;
            std::vector<long long> ns = {0, 1, 255, 1024, 4096, 65536, s / 2, s - 1023, s - 1, s, s + 1, s + 4096, cap / 2,
                                         cap - 1, cap, 1000000, 1200000};
            for (int i = 1; i < 200; ++i) ns.push_back(cap / 200 * i);
            for (long long n : ns) {
                if (n < 0 || n > cap) continue;
                for (int n_keys : {2, 257, 513, 22501, 40000, 62501, 157501, 202501, 1 << 18, 1 << 20, 0x7fffffff})
                    for (int longt = 0; longt < 2; ++longt) {
                        const SortLayout L = sort_layout(n, n_keys, n_sm, longt);
                        const size_t held = sort_scratch_ints(cap, n_sm, longt);
                        ++checked;
                        if (L.ints > held) {
                            std::printf("sms %d capacity %lld call %lld keys %d long %d: needs %zu, held %zu\n", n_sm, cap, n,
                                        n_keys, longt, L.ints, held);
                            return 1;
                        }
                        // the tiles hold every key, the passes every bit
                        if ((long long)L.n_tiles * kSortThreads * L.rounds < n || L.passes * 9 < L.bits ||
                            (1ll << L.bits) < n_keys)
                            return 2;
                    }
            }
        }
    }
    std::printf("%lld layouts\n", checked);
    return 0;
}
"""


def test_scratch_of_a_capacity_holds_every_smaller_call(tmp_path):
    src, exe = tmp_path / "layout.cpp", tmp_path / "layout"
    src.write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
