"""The first part of a Cash-Karp stage (what needs no product) runs ahead inside the UY launch for
pieces of 16 to 64 elements.  An ensemble of many one-leaf members keeps its leaf rows whole (one
piece a member, of 12 to 72 elements); the same fault stepped alone is cut into short pieces, whose
stages run in one go.  Both must give the same trajectory to the last bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2110_12165_gb300 as hbi
from synthetic import friction, meshes
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n1,n2", [(4, 3), (4, 4), (10, 4), (8, 8), (17, 4), (9, 8)])
def test_pieces_run_ahead_equal_a_single_run(n1, n2):
    nm, eps, steps = 1000, 1e-6, 12
    m = meshes.dipping_rect(n1, n2, 250.0, 30.0)
    n, rk = m.n_elem, np.full(m.n_elem, np.pi / 2)
    Fs = [friction.ensemble_friction(m, seed=60 + k) for k in range(3)]
    mine = [Fs[k % 3] for k in range(nm)]
    hE, starts = hbi.hbi_build_ensemble([m.verts] * nm, 32e9, 0.25, oracle.OP_RAKE_SHEAR, eps, 128, 1, "fp32",
                                        rakes=[rk] * nm)
    assert hE.stats()["n_tasks_uy"] == nm                     # every member one piece
    fric = lambda fs: hbi.friction(*(dev(np.concatenate([getattr(F, f) for F in fs])) for f in ("a", "b", "dc", "rake")),
                                   Fs[0].f0, Fs[0].V0, Fs[0].Vpl, Fs[0].mu, Fs[0].cs)

    def state(fs):
        st = [oracle.steady_state(F.V_init, F.a, F.b, F.sigma0, F.f0, F.V0) for F in fs]
        return np.concatenate([np.concatenate(c) for c in ([p for p, _ in st], [t for _, t in st],
                                                           [F.sigma0 for F in fs], [np.zeros(n)] * len(fs))])

    sE, tE, dtE = dev(state(mine)), dev(np.zeros(nm)), dev(np.full(nm, 3e9))   # starts with rejected attempts
    st, done, _ = hbi.hbi_step_ensemble(hE, fric(mine), sE, tE, dtE, 1e-4, steps)
    assert st == 0 and list(done) == [steps] * nm
    got = host(sE).reshape(4, nm, n)
    h1 = hbi.hbi_build(m.verts, 32e9, 0.25, oracle.OP_RAKE_SHEAR, eps, 128, 1, "fp32", rake=rk)
    for k, F in enumerate(Fs):
        s1, t1, dt1 = dev(state([F])), dev([0.0]), dev([3e9])
        assert hbi.hbi_step(h1, fric([F]), s1, t1, dt1, 1e-4, steps)[:2] == (0, steps)
        for q in (k, 3 * 160 + k, 3 * 332 + k):
            assert np.array_equal(got[:, q].ravel(), host(s1)), f"member {q} differs"
            assert host(tE)[q] == host(t1)[0] and host(dtE)[q] == host(dt1)[0]
