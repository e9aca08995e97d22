"""The multi-RHS product's row split and gather at the edges of its row lengths: k at and beside 16,
32 and 64, alternating on one handle (the split rows' length, the row of zeros and the buffers
change with k), with inputs that hold zeros, an all-zero right-hand side and magnitudes 30
decades apart.  Each right-hand side against the single-vector product (2e-5 relative L2 as in
the other multi-RHS tests: the 22-bit input split and FP32 order)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2110_12165_gb300 as hbi
from synthetic import meshes, rng
from gpu_util import dev, host, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cells,leaf,op,storage", [((9, 5), 8, 3, "mixed"), ((31, 17), 64, 3, "fp16"), ((45, 23), 32, 1, "mixed")])
def test_row_lengths_alternate(cells, leaf, op, storage):
    m = meshes.scaled_thrust_mesh(*cells, seed=8)
    h = hbi.hbi_build(m.verts, 32e9, 0.25, op, 1e-4, leaf, 1, storage, rake=np.full(m.n_elem, 0.2), recompress_eps=1e-4,
                      multi_rhs=True)
    nx, ny = h.nin * m.n_elem, h.nout * m.n_elem
    X = rng.normal(41, 64 * nx).reshape(64, nx)
    X[:, ::5] = 0.0
    X[3] = 0.0
    X *= 10.0 ** np.linspace(-15, 15, 64)[:, None]
    ref = np.empty((64, ny))
    y = torch.zeros(ny, dtype=torch.float64, device="cuda")
    for r in range(64):
        hbi.hbi_matvec(h, dev(X[r]), y)
        ref[r] = host(y)
    for k in (16, 64, 17, 1, 33, 32, 48, 15, 64):
        Y = torch.full((k * ny,), float("nan"), dtype=torch.float64, device="cuda")
        hbi.hbi_matvec_multi(h, k, dev(X[:k].reshape(-1)), Y)
        got = host(Y).reshape(k, ny)
        for r in range(k):
            if r == 3:
                assert not got[r].any()
            else:
                assert rel_l2(got[r], ref[r]) < 2e-5, (k, r)
