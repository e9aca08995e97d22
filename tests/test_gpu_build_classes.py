"""The build's launch classes (blocks evaluated whole before their ACA, CTAs of 64, 128 and 256
threads, recompression by rank): operators whose blocks fall into each of them against the dense
operator of the same elements (eta so small that no block is admissible), 10 eps as for the
other built operators; full and half space, one and several components, ragged leaves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2110_12165_gb300 as hbi
from synthetic import meshes, rng
from gpu_util import dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mesh,op,leaf,storage,recompress,half", [
    ("thrust", 3, 64, "fp64", 0.0, False),      # sides of 20 to 600 elements
    ("thrust", 3, 16, "mixed", 1e-4, False),
    ("planar", 0, 32, "fp64", 1e-5, False),
    ("planar", 1, 7, "fp64", 0.0, False),
    ("thrust", 2, 24, "fp64", 0.0, True)])
def test_built_operator_equals_its_dense_entries(mesh, op, leaf, storage, recompress, half):
    if mesh == "thrust":
        m = meshes.scaled_thrust_mesh(*((20, 11) if half else (47, 23)), seed=6)
    else:
        m = meshes.planar_vertical_rect(53, 41, 250.0, origin=(0.0, 0.0, -500.0))
    eps, rake = 1e-4, np.full(m.n_elem, 0.3)
    args = (m.verts, 32e9, 0.25, op)
    h = hbi.hbi_build(*args, eps, leaf, 1, storage, rake=rake, recompress_eps=recompress, half_space=half)
    d = hbi.hbi_build(*args, eps, 128, 0, "fp64", rake=rake, eta=1e-9, half_space=half)
    assert h.stats()["n_lowrank"] > 20 and d.stats()["n_lowrank"] == 0
    x = dev(rng.normal(17, h.nin * m.n_elem))
    y, ref = (torch.zeros(h.nout * m.n_elem, dtype=torch.float64, device="cuda") for _ in range(2))
    hbi.hbi_matvec(h, x, y)
    hbi.hbi_matvec(d, x, ref)
    assert rel_l2(host(y), host(ref)) < 10 * eps
