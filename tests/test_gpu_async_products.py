"""hbi_matvec_async inside the caller's own CUDA graph and on the caller's streams: its kernels are
launched with programmatic dependencies and write the caller's array directly, so a captured
product replayed on new inputs, and products of two handles interleaved on two streams, must give
the bits of the plain calls."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2110_12165_gb300 as hbi
from synthetic import meshes, rng
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


def _handle(cells, op, storage):
    m = meshes.scaled_thrust_mesh(*cells, seed=5)
    return hbi.hbi_build(m.verts, 32e9, 0.25, op, 1e-4, 32, 1, storage, rake=np.full(m.n_elem, 0.4),
                         recompress_eps=1e-4 if storage == "mixed" else 0.0)


@pytest.mark.parametrize("cells,op,storage", [((9, 5), 3, "fp64"), ((31, 17), 0, "fp32"), ((40, 25), 3, "mixed")])
def test_captured_product_replays(cells, op, storage):
    h = _handle(cells, op, storage)
    x = dev(rng.normal(7, h.nin * h.n))
    y, ref = (torch.zeros(h.nout * h.n, dtype=torch.float64, device="cuda") for _ in range(2))
    hbi.hbi_matvec(h, x, ref)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        hbi.hbi_matvec_async(h, x, y)
    for seed in (7, 8):
        x.copy_(dev(rng.normal(seed, h.nin * h.n)))
        g.replay()
        torch.cuda.synchronize()
        got = host(y).copy()
        hbi.hbi_matvec(h, x, ref)
        assert np.array_equal(got, host(ref))


def test_two_handles_on_two_streams():
    hs = [_handle((40, 25), 3, "mixed"), _handle((31, 17), 2, "fp32")]
    xs = [dev(rng.normal(11 + k, h.nin * h.n)) for k, h in enumerate(hs)]
    refs = [torch.zeros(h.nout * h.n, dtype=torch.float64, device="cuda") for h in hs]
    for h, x, r in zip(hs, xs, refs):
        hbi.hbi_matvec(h, x, r)
    ys = [torch.zeros_like(r) for r in refs]
    streams = [torch.cuda.Stream() for _ in hs]
    torch.cuda.synchronize()
    for _ in range(20):
        for h, x, y, s in zip(hs, xs, ys, streams):
            hbi.hbi_matvec_async(h, x, y, stream=s)
    torch.cuda.synchronize()
    for y, r in zip(ys, refs):
        assert np.array_equal(host(y), host(r))
