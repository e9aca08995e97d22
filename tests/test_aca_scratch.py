"""The scratch of the build's ACA stays within its share of the free memory, whatever the largest block:
the plan on the host (CPU; needs nvcc), and an operator built on the GPU where little memory is left,
so that the larger blocks keep no components and, with less, the scratch they would take does not
exist: the same operator bit for bit."""
import os
import subprocess

import numpy as np
import pytest

from test_host_tables import ROOT, _nvcc


def test_scratch_stays_within_its_share(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_aca_scratch")
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-o", exe,
                        os.path.join(ROOT, "tests", "host_aca_scratch.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    rows = [tuple(int(v) for v in line.split()) for line in out if line.strip()]
    assert len(rows) == 5 * 5 * 4
    for q in range(0, len(rows), 4):
        total = 0
        for free, side, c, jobs, resident, want, grid, slot in rows[q:q + 4]:
            assert 1 <= grid <= min(jobs, resident) and 0 <= slot <= want
            assert slot == want if c == 3 else grid == min(jobs, resident)
            total += grid * slot
        assert total <= max(free // 16, 6 * 40 * 40)   # at the least one block of the whole class
        if free * 8 >= 270 << 30 and side <= 10000:
            assert all(row[6:] == (min(row[3], row[4]), row[5]) for row in rows[q:q + 4])   # all of it fits


@pytest.mark.gpu
@pytest.mark.parametrize("free", [3 << 30, 700 << 20])
def test_an_operator_built_where_little_memory_is_left(free):
    import gc

    import paper_2110_12165_gb300 as hbi
    import torch
    from gpu_util import dev, host
    from synthetic import meshes, rng
    m = meshes.planar_vertical_rect(100, 50, 250.0, origin=(0.0, 0.0, -500.0))   # factors 277 MB, scratch up to 479 MB
    x = dev(rng.normal(29, 2 * m.n_elem))

    def product():
        h = hbi.hbi_build(m.verts, 32e9, 0.25, 3, 1e-4, 32, 0, "fp64", rake=np.full(m.n_elem, 0.3))
        y = torch.zeros(3 * m.n_elem, dtype=torch.float64, device="cuda")
        hbi.hbi_matvec(h, x, y)
        return host(y)

    ref = product()
    gc.collect()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")
    try:
        y = product()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert np.array_equal(y, ref)
