"""A multi-RHS product refused under stream capture (it synchronises) leaves the handle as it was: the
next call computes what it would have without the refused one, although the split rows hold NaN
from an earlier call with longer rows where the shorter rows end.  Against the single-vector
product (2e-5 relative L2 as in the other multi-RHS tests)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2110_12165_gb300 as hbi
from synthetic import meshes, rng
from gpu_util import dev, host, rel_l2

pytestmark = pytest.mark.gpu


def _cudart():
    """The CUDA runtime this process has loaded."""
    with open("/proc/self/maps") as f:
        path = next(line.split()[-1] for line in f if "libcudart" in line)
    return ctypes.CDLL(path)


@pytest.mark.parametrize("k", [7, 20])
def test_call_after_a_refused_one(k):
    m = meshes.scaled_thrust_mesh(31, 17, seed=8)
    h = hbi.hbi_build(m.verts, 32e9, 0.25, 3, 1e-4, 32, 1, "mixed", rake=np.full(m.n_elem, 0.2), recompress_eps=1e-4,
                      multi_rhs=True)
    nx, ny = h.nin * m.n_elem, h.nout * m.n_elem
    X = rng.normal(43, k * nx).reshape(k, nx)
    x, Y = dev(X.reshape(-1)), torch.zeros(64 * ny, dtype=torch.float64, device="cuda")
    hbi.hbi_matvec_multi(h, 64, torch.full((64 * nx,), float("nan"), dtype=torch.float64, device="cuda"), Y)
    rt, s, graph = _cudart(), torch.cuda.Stream(), ctypes.c_void_p()
    torch.cuda.synchronize()
    assert rt.cudaStreamBeginCapture(ctypes.c_void_p(s.cuda_stream), 2) == 0   # relaxed
    with pytest.raises(hbi.HbiError):
        hbi.hbi_matvec_multi(h, k, x, Y, stream=s)
    assert rt.cudaStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) != 0   # invalidated
    rt.cudaGetLastError()
    hbi.hbi_matvec_multi(h, k, x, Y)
    y = torch.zeros(ny, dtype=torch.float64, device="cuda")
    for r in range(k):
        hbi.hbi_matvec(h, dev(X[r]), y)
        assert rel_l2(host(Y)[r * ny:(r + 1) * ny], host(y)) < 2e-5, r
