"""The first half-space build of a process runs its launch classes side by side like the later ones:
a kernel's first use loads it and waits for what is running, so the classes' kernels are loaded
before the first of them is launched.  The first build may take half as long again as the
second (loading; classes one after the other take twice as long)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))

SCRIPT = r'''
import sys, time
sys.path.insert(0, ROOT)
import numpy as np, torch
import paper_2110_12165_gb300 as hbi
from synthetic import meshes
small, m = meshes.scaled_thrust_mesh(9, 5, seed=6), meshes.scaled_thrust_mesh(47, 43, seed=6)
def build(m, half):
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    h = hbi.hbi_build(m.verts, 32e9, 0.25, 3, 1e-4, 64, 0, "mixed", rake=np.full(m.n_elem, 0.3), half_space=half)
    torch.cuda.synchronize()
    return time.perf_counter() - t0
build(small, False)   # the context, the packing kernels
print(build(m, True), build(m, True))
'''


def test_first_half_space_build_takes_no_longer():
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % os.path.dirname(HERE) + SCRIPT], capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    first, second = (float(v) for v in r.stdout.split()[-2:])
    assert first < 1.5 * second, (first, second)
