"""The build's launch class of a block, from its shape (CPU; needs nvcc): only blocks of short sides are
evaluated whole by one small CTA, never a small leaf against a cluster of any size, which a
small fault beside a large one gives.  On the GPU: such meshes against the dense operator of the same
elements, and blocks evaluated whole that meet a singular pair, which are taken up again row by row
and column by column and fail only if that reaches the pair."""
import os
import subprocess

import numpy as np
import pytest

from test_host_tables import ROOT, _nvcc


def test_blocks_evaluated_whole_have_short_sides(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_aca_classes")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(ROOT, "tests", "host_aca_classes.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = [tuple(int(v) for v in line.split()) for line in out if line.strip()]
    assert len(rows) == 256
    by = {(t, s): c for t, s, c, _ in rows}
    for t, s, c, step in rows:
        side = max(t, s)
        assert step == (0 if side > 128 else 1 if side > 64 else 2)
        assert c in (step, 3) and c == by[s, t]
        if c == 3:   # no more pair evaluations than 20 rows and columns of it, each of a few warps
            assert side <= 128 and (t * s + 31) // 32 <= 20 * ((t + 31) // 32 + (s + 31) // 32)
    assert by[40, 40] == 3 and by[16, 128] == 3 and by[128, 128] == 1 and by[16, 4000] == 0


def _build(verts, eps=1e-4, leaf=32, **kw):
    import paper_2110_12165_gb300 as hbi
    return hbi.hbi_build(verts, 32e9, 0.25, 3, eps, leaf, 0, "fp64", rake=np.full(len(verts), 0.3), **kw)


def _product(h, x):
    import paper_2110_12165_gb300 as hbi
    import torch
    from gpu_util import dev, host
    y = torch.zeros(h.nout * h.n, dtype=torch.float64, device="cuda")
    hbi.hbi_matvec(h, dev(x), y)
    return host(y)


@pytest.mark.gpu
@pytest.mark.parametrize("small", [(1, 1), (4, 4), (7, 3)])
def test_a_small_fault_beside_a_large_one(small):
    from gpu_util import rel_l2
    from synthetic import meshes, rng
    v = np.concatenate([meshes.planar_vertical_rect(40, 25, 250.0, origin=(0.0, 0.0, -500.0)).verts,
                        meshes.planar_vertical_rect(*small, 50.0, origin=(30e3, 3e3, -700.0)).verts])
    x = rng.normal(19, 2 * len(v))
    assert rel_l2(_product(_build(v), x), _product(_build(v, eta=1e-9), x)) < 10 * 1e-4


@pytest.mark.gpu
def test_a_block_with_a_singular_pair():
    import paper_2110_12165_gb300 as hbi
    from gpu_util import rel_l2
    from synthetic import meshes, rng
    # receivers, and a sliver 40 km off whose long edge runs through one receiver's centre
    near = meshes.planar_vertical_rect(10, 10, 250.0, origin=(0.0, 0.0, -500.0)).verts
    x, z, w = 1375.0, -1875.0, 1e-4
    sliver = np.array([[[x, -80e3, z], [x, 200.0, z], [x, 200.0, z - w], [x, -80e3, z - w]]])
    # among ordinary elements, whose columns are far larger: neither its column nor that receiver's row is
    # among the five pivots, so the operator is built
    far = meshes.planar_vertical_rect(4, 2, 1000.0, origin=(-2e3, -40e3, -400.0)).verts
    eps = 1e-2
    h = _build(np.concatenate([near, far, sliver]), eps=eps, leaf=100)
    n = len(near) + len(far)
    u = rng.normal(23, 2 * n).reshape(2, n)
    y = _product(h, np.pad(u, ((0, 0), (0, 1))).reshape(-1)).reshape(3, n + 1)[:, :n]
    ref = _product(_build(np.concatenate([near, far]), eta=1e-9), u.reshape(-1)).reshape(3, n)
    assert h.stats()["n_lowrank"] == 2 and h.stats()["max_rank"] == 5
    assert rel_l2(y, ref) < 10 * eps
    # alone: its column is the first pivot's
    with pytest.raises(hbi.HbiError, match="SINGULAR"):
        _build(np.concatenate([near, sliver]), eps=eps, leaf=100)
