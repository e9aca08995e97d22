"""Leaf row units cut into pieces for the UY phase: the cutter on the host (CPU; needs nvcc), and
the product of small and ragged operators, whose pieces take one, two and four rows per pass and
end in partial row blocks, against the oracle on its own factors (FP64 storage: the sums differ
from the oracle's in order only, 1e-12 as in the other product tests)."""
import os
import subprocess

import numpy as np
import pytest

from test_host_tables import ROOT, _nvcc


def test_pieces_tile_their_units(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_pieces")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(ROOT, "tests", "host_pieces.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert out[:2] == ["violations", "0"]
    assert int(out[3]) > int(out[5])   # some units are cut


@pytest.mark.gpu
@pytest.mark.parametrize("cells,leaf,op", [((5, 3), 8, 3), ((9, 7), 16, 0), ((23, 11), 64, 2), ((40, 25), 32, 3),
                                           ((61, 43), 64, 1)])
def test_cut_units_against_the_oracle(cells, leaf, op):
    import oracle
    import paper_2110_12165_gb300 as hbi
    from gpu_util import dev, host, import_oracle, rel_l2
    from synthetic import meshes, rng
    import torch
    m = meshes.scaled_thrust_mesh(*cells, seed=9)
    H = oracle.HMatrix(m, op, 1e-4, leaf, 1, 32e9, 0.25, rake=np.full(m.n_elem, 0.7))
    x = rng.normal(31, oracle.OP_NIN[op] * m.n_elem)
    h = import_oracle(H, "fp64")
    assert h.stats()["n_tasks_uy"] >= h.stats()["n_leaves"]
    y = torch.zeros(oracle.OP_NOUT[op] * m.n_elem, dtype=torch.float64, device="cuda")
    hbi.hbi_matvec(h, dev(x), y)
    assert rel_l2(host(y), H.matvec(x)) < 1e-12
