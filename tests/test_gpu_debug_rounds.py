"""The bounds-checking build (RUBIX_DEBUG=1) on the rounds of every bin step
(tests/_debug_rounds.py): its kernels check every slab read, each round's node
included, and set a bit in the device error word instead of reading out of range. It
must report nothing and give the release build's cubes and gradients bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def _run(kind, tmp_path):
    out = str(tmp_path / f"{kind}.npz")
    r = subprocess.run([sys.executable, os.path.join(HERE, "_debug_rounds.py"), kind, out], capture_output=True, text=True,
                       timeout=1200)
    assert r.returncode == 0, r.stderr[-3000:]
    return np.load(out)


def test_debug_build_on_every_kind_of_rounds(tmp_path):
    dbg = _run("debug", tmp_path)
    rel = _run("release", tmp_path)
    assert sorted(dbg.files) == sorted(rel.files)
    for k in dbg.files:
        if k.endswith("/err"):
            assert int(dbg[k][0]) == 0 and int(rel[k][0]) == 0, (k, int(dbg[k][0]))
        else:
            assert np.array_equal(dbg[k], rel[k]), k
    # shifts past the halo reached the global path, the others stayed in the slabs
    for k in dbg.files:
        if k.endswith("/slow"):
            assert (int(dbg[k][0]) > 0) == k.startswith("fast"), (k, int(dbg[k][0]))
