"""The work a user of this library has it do, as timed cases through its public entry points.

A simulation builds the lattice H-matrix of a fault once (hbi_build), then spends its time in
the adaptive Runge-Kutta steps of the rate-and-state ODE (hbi_step and its rake-free and
ensemble forms), six products y = H x per attempt.  Beside that stand the product alone, the
product with many right-hand sides, and the adjoint gradient of a run of fixed steps.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  fault, operator, friction and inputs of one user, on the GPU
    run(state)           one pass through the public entry points
    work(case)           bytes and operations the path cannot do without
    exact(case, seed)    the same outputs from the dense operator in plain 64-bit torch

The seed makes the fault (the jitter of its mesh), its friction and its state.
"""
import math

import numpy as np
import torch

import paper_2110_12165_gb300 as hbi

KM = 1000.0
MU, NU, CS = 32e9, 0.25, 3460.0          # rigidity, Poisson's ratio, shear-wave speed
F0, V0, VPL = 0.6, 1e-6, 1e-9            # reference friction and slip rate, plate rate
SIGMA0, EPS_RK = 50e6, 1e-4
ELEM_BYTES = {"fp64": (8, 8), "fp32": (4, 4), "mixed": (2, 4), "adaptive": (2, 4), "fp16": (2, 2)}


def listed():
    return [
        # the paper's plain method at its smallest: one strike-slip product of a planar fault in
        # FP64 (64 x 32 squares, leaf 32, eps 1e-6); 20 MB of factors, so latency and launches
        dict(name="product-planar-2048-fp64", kind="product", mesh="planar", n1=64, n2=32, op=0, storage="fp64",
             leaf=32, depth=0, aca_eps=1e-6),
        # the 0.7 km thrust fault with FP32 factors, strike and dip slip to all three tractions
        dict(name="product-thrust-20022-fp32", kind="product", mesh="thrust", n1=141, n2=71, op=3, storage="fp32",
             leaf=64, depth=2, aca_eps=1e-4),
        # the 0.25 km thrust fault in the storage the large runs use (FP16 far field, FP32 near)
        dict(name="product-thrust-160000-mixed", kind="product", mesh="thrust", n1=400, n2=200, op=3, storage="mixed",
             leaf=64, depth=2, aca_eps=1e-4),
        # a handful of slip-rate vectors at once on a small ragged fault
        dict(name="multi-thrust-5246-k7", kind="multi", mesh="thrust", n1=61, n2=43, op=3, storage="mixed", leaf=64,
             depth=2, aca_eps=1e-4, k=7),
        # a full block of right-hand sides on a 0.5 km fault
        dict(name="multi-thrust-40000-k64", kind="multi", mesh="thrust", n1=200, n2=100, op=3, storage="mixed",
             leaf=64, depth=2, aca_eps=1e-4, k=64),
        # adaptive steps of the small FP64 fault in mid-cycle: launch-bound
        dict(name="step-planar-2048-fp64", kind="step", mesh="planar", n1=64, n2=32, op=0, storage="fp64", leaf=32,
             depth=0, aca_eps=1e-6, steps=50),
        # adaptive steps of the 0.7 km fault
        dict(name="step-thrust-20022-mixed", kind="step", mesh="thrust", n1=141, n2=71, op=3, storage="mixed",
             leaf=64, depth=2, aca_eps=1e-4, steps=20),
        # adaptive steps of the 0.25 km fault, the production run
        dict(name="step-thrust-160000-mixed", kind="step", mesh="thrust", n1=400, n2=200, op=3, storage="mixed",
             leaf=64, depth=2, aca_eps=1e-4, steps=4),
        # rake-free friction on a ragged mid-size fault with FP64 factors
        dict(name="vector-thrust-10010-fp64", kind="vector", mesh="thrust", n1=91, n2=55, op=3, storage="fp64",
             leaf=64, depth=2, aca_eps=1e-4, steps=10),
        # an ensemble of independent dipping faults of uneven size, FP32 factors
        dict(name="ensemble-12-faults-fp32", kind="ensemble", mesh="rect", n1=12, n2=9000, op=0, storage="fp32",
             leaf=64, depth=2, aca_eps=1e-4, steps=10),
        # the gradient of a slip-rate misfit with respect to a - b and d_c
        dict(name="gradient-thrust-20022-fp32", kind="gradient", mesh="thrust", n1=141, n2=71, op=3, storage="fp32",
             leaf=64, depth=2, aca_eps=1e-4, steps=10),
        # a new fault geometry: build the operator and take its first product
        dict(name="build-thrust-20022-mixed", kind="build", mesh="thrust", n1=141, n2=71, op=3, storage="mixed",
             leaf=64, depth=2, aca_eps=1e-4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["product", "product", "transpose", "multi", "step", "step", "vector", "ensemble", "gradient",
                       "build"])
    # elements: the whole range for products and steps, up to the listed sizes for the others
    top = {"product": 140000, "transpose": 70000, "multi": 38000, "step": 110000, "vector": 40000, "gradient": 20000,
           "build": 40000}.get(kind, 0)
    c = dict(kind=kind)
    if kind == "ensemble":
        c.update(mesh="rect", n1=rng.randint(2, 12), n2=_log(rng, 600, 9000), op=0, storage="fp32")
    else:
        planar = kind != "vector" and rng.random() < 0.3
        n = _log(rng, 300, min(top, 20000) if planar else top)
        aspect = rng.uniform(1.3, 2.6)
        cells = n if planar else n / 2
        n2 = max(3, int(round(math.sqrt(cells / aspect))))
        n1 = max(5, int(round(cells / n2)))
        c.update(mesh="planar" if planar else "thrust", n1=n1, n2=n2)
        c["op"] = 3 if kind == "vector" or not planar else rng.choice([0, 1, 2])
        if kind == "multi":
            c["storage"] = rng.choice(["mixed", "fp16"])
            c["k"] = rng.randint(2, 64)
        else:
            small = n < 25000
            c["storage"] = rng.choice(["fp64", "fp32", "mixed", "adaptive"] if small else ["fp32", "mixed", "adaptive"])
    c["leaf"] = rng.choice([32, 64])
    c["depth"] = rng.choice([0, 1, 2])
    c["aca_eps"] = rng.choice([1e-4, 1e-4, 1e-5])
    if kind in ("step", "vector", "ensemble", "gradient"):
        c["steps"] = rng.randint(3, 10)
    return c


# ------------------------------------------------------------------ faults and friction
def _rng(case, seed, what):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, what, case["n1"], case["n2"]])


def _rect(n1, n2, h, dip):
    """n1 x n2 squares of side h, dipping at `dip` radians: vertices (n, 4, 3), centres (n, 2)."""
    i, s = np.meshgrid(np.arange(n1), np.arange(n2))
    i, s = i.ravel(), s.ravel()
    x = np.stack([i, i + 1, i + 1, i], 1) * h
    d = np.stack([s, s, s + 1, s + 1], 1) * h
    v = np.stack([x, d * np.cos(dip), -d * np.sin(dip)], -1)
    return np.ascontiguousarray(v), np.stack([(i + 0.5) * h, (s + 0.5) * h], 1)


def _thrust(n1, n2, rng):
    """A 100 x 50 km thrust surface (dip 10 to 30 degrees, undulating trace) of 2 n1 n2 triangles
    with jittered interior nodes: vertices (n, 3, 3), centres in (strike, down-dip) metres."""
    dx, ds = 100 * KM / n1, 50 * KM / n2
    X, S = np.meshgrid(np.arange(n1 + 1) * dx, np.arange(n2 + 1) * ds, indexing="ij")
    inner = (slice(1, -1), slice(1, -1))
    X[inner] += 0.15 * dx * rng.uniform(-1, 1, X[inner].shape)
    S[inner] += 0.15 * ds * rng.uniform(-1, 1, S[inner].shape)
    d0, k = np.deg2rad(10.0), np.deg2rad(20.0) / (50 * KM)
    Y = (np.sin(d0 + k * S) - np.sin(d0)) / k + 2 * KM * np.sin(2 * np.pi * X / (40 * KM))
    Z = -(1 * KM + (np.cos(d0) - np.cos(d0 + k * S)) / k)
    P, Q = np.stack([X, Y, Z], -1), np.stack([X, S], -1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(n1), np.arange(n2), indexing="ij"))
    even = ((i + j) % 2 == 0)[:, None]
    c00, c10 = np.stack([i, j], 1), np.stack([i + 1, j], 1)
    c11, c01 = np.stack([i + 1, j + 1], 1), np.stack([i, j + 1], 1)
    t = np.stack([np.stack([c00, c10, np.where(even, c11, c01)], 1),
                  np.stack([np.where(even, c00, c10), c11, c01], 1)], 1).reshape(-1, 3, 2)
    return np.ascontiguousarray(P[t[..., 0], t[..., 1]]), Q[t[..., 0], t[..., 1]].mean(1)


def _faults(case, seed):
    """[(vertices, centres)]: one fault, or the members of an ensemble."""
    rng = _rng(case, seed, 1)
    if case["mesh"] == "thrust":
        return [_thrust(case["n1"], case["n2"], rng)]
    if case["mesh"] == "planar":
        return [_rect(case["n1"], case["n2"], 250.0, 0.5 * np.pi)]
    out = []
    for m in range(case["n1"]):   # members of n2 / 5 to n2 elements, 2:1, dips of 15 to 60 degrees or vertical
        nd = max(2, 2 * int(round(math.sqrt(case["n2"] * (0.2 + 0.8 * (m + 1) / case["n1"]) / 2) / 2)))
        out.append(_rect(2 * nd, nd, 250.0, 0.5 * np.pi if m % 4 == 3 else np.deg2rad(rng.uniform(15, 60))))
    return out


def _smooth(centres, rng):
    """A smooth random field of about unit variance on one fault."""
    L = np.ptp(centres, axis=0) + 1.0
    f = np.zeros(len(centres))
    for _ in range(12):
        k = rng.uniform(-4, 4, 2) * np.pi / L
        f += math.sqrt(2 / 12) * np.cos(centres @ k + rng.uniform(0, 2 * np.pi))
    return f


def _friction(case, seed, faults):
    """Per element: a, b, d_c, rake and the slip rates of a fault in mid-cycle."""
    rng = _rng(case, seed, 2)
    cols = []
    for v, c in faults:
        n = len(c)
        size = np.ptp(c, axis=0)
        at = c.min(0) + size * rng.uniform(0.3, 0.7, 2)
        weak = (np.abs(c[:, 0] - at[0]) <= 0.15 * size[0]) & (np.abs(c[:, 1] - at[1]) <= 0.2 * size[1])
        b = np.full(n, 0.015)
        a = np.where(weak, 0.010, 0.019)
        rake = np.full(n, 0.0 if case["mesh"] == "planar" else 0.5 * np.pi)
        V = VPL * 10.0 ** (0.5 * _smooth(c, rng) - np.where(weak, 1.0, 0.0))
        dc = np.full(n, 0.005 if case["mesh"] != "rect" else rng.uniform(0.004, 0.02))
        phi = F0 - b * np.log(V / V0) + 0.002 * _smooth(c, rng)
        cols.append(np.stack([a, b, dc, rake, V, phi]))
    return np.concatenate(cols, axis=1)


def _T(a):
    return torch.tensor(np.ascontiguousarray(a, dtype=np.float64), device="cuda")


def _state0(case, fr):
    """phi, tau (or tau_s, tau_d), sigma and zero slip of that fault: tau from the friction law."""
    a, b, dc, rake, V, phi = fr
    n = len(a)
    sigma = np.full(n, SIGMA0)
    tau = a * sigma * np.arcsinh(V / (2 * V0) * np.exp(phi / a))
    if case["kind"] == "vector":   # the traction a little off the loading direction
        ang = rake + 0.1 * np.sin(np.arange(n))
        return np.concatenate([phi, tau * np.cos(ang), tau * np.sin(ang), sigma, np.zeros(2 * n)])
    return np.concatenate([phi, tau, sigma, np.zeros(n)])


def _input(case, seed, faults, rows, comps):
    """`rows` vectors of slip-rate deficits V - V_pl along `comps` components, in the caller's order."""
    rng = _rng(case, seed, 3)
    out = []
    for _ in range(rows):
        for _ in range(comps):
            f = np.concatenate([_smooth(c, rng) + 0.05 * rng.standard_normal(len(c)) for _, c in faults])
            out.append(VPL * (10.0 ** f - 1.0))
    return np.concatenate(out)


def _steps_of(case):
    return np.full(case["steps"], 2e5)   # fixed steps of a gradient run (s), stable for this friction


def _build(case, faults, rake):
    two = ELEM_BYTES[case["storage"]][0] == 2
    keys = dict(recompress_eps=1e-4 if two else 0.0, transpose=case["kind"] in ("transpose", "gradient"),
                multi_rhs=case["kind"] == "multi")
    args = (MU, NU, case["op"], case["aca_eps"], case["leaf"], case["depth"], case["storage"])
    if case["kind"] == "ensemble":
        return hbi.hbi_build_ensemble([v for v, _ in faults], *args, rakes=rake, **keys)[0]
    return hbi.hbi_build(faults[0][0], *args, rake=rake[0], **keys)


def prepare(case, seed):
    faults = _faults(case, seed)
    fr = _friction(case, seed, faults)
    at = np.cumsum([len(c) for _, c in faults])[:-1]
    s = dict(case=case, faults=faults, rake=np.split(fr[3], at))
    n, kind = fr.shape[1], case["kind"]
    nin, nout = hbi.OP_NIN[case["op"]], hbi.OP_NOUT[case["op"]]
    if kind == "build":
        s["x"] = _T(_input(case, seed, faults, 1, nin))
        s["y"] = torch.zeros(nout * n, dtype=torch.float64, device="cuda")
        return s
    s["h"] = _build(case, faults, s["rake"])
    if kind in ("product", "transpose", "multi"):
        k = case.get("k", 1)
        ni, no = (nout, nin) if kind == "transpose" else (nin, nout)
        s["x"] = _T(_input(case, seed, faults, k, ni))
        s["y"] = torch.zeros(k * no * n, dtype=torch.float64, device="cuda")
        return s
    s["abdr"] = [_T(v) for v in fr[:4]]
    s["fric"] = hbi.friction(*s["abdr"], F0, V0, VPL, MU, CS)
    s["state0"] = _T(_state0(case, fr))
    if kind == "gradient":
        s["target"] = _T(np.log(fr[4]) + 0.1 * _rng(case, seed, 4).standard_normal(n))
        s["ga"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        s["gd"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        s["final"] = torch.zeros(4 * n, dtype=torch.float64, device="cuda")
        s["dts"] = _steps_of(case)
    else:
        m = len(faults)
        s["t0"], s["dt0"] = _T(np.zeros(m)), _T(np.full(m, 2e4))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "product":
        hbi.hbi_matvec(s["h"], s["x"], s["y"])
        return s["y"]
    if kind == "transpose":
        hbi.hbi_matvec_transpose(s["h"], s["x"], s["y"])
        return s["y"]
    if kind == "multi":
        hbi.hbi_matvec_multi(s["h"], case["k"], s["x"], s["y"])
        return s["y"]
    if kind == "build":
        h = _build(case, s["faults"], s["rake"])
        hbi.hbi_matvec(h, s["x"], s["y"])
        return s["y"]
    if kind == "gradient":
        loss = hbi.hbi_adjoint(s["h"], s["fric"], s["state0"], s["dts"], s["target"], s["ga"], s["gd"],
                               checkpoint_every=max(2, case["steps"] // 2), state_final=s["final"])
        return dict(loss=loss, grad_amb=s["ga"], grad_dc=s["gd"], state=s["final"])
    # adaptive steps from the state at hand, with their step records
    state, t, dt = s["state0"].clone(), s["t0"].clone(), s["dt0"].clone()
    step = {"step": hbi.hbi_step, "vector": hbi.hbi_step_vector, "ensemble": hbi.hbi_step_ensemble}[kind]
    status, done, rec = step(s["h"], s["fric"], state, t, dt, EPS_RK, case["steps"])
    if status != 0:
        raise RuntimeError("%s: %s" % (kind, hbi.status_string(status)))
    return dict(state=state, t=t, dt=dt, done=done, records=rec)


def work(case):
    """One product reads every stored entry of the operator once, its input, and writes its output;
    an attempt is six products, a gradient's step six forward and six transposed ones.  A step
    reads and writes its FP64 state once.  A build evaluates the entries it stores (about 250
    operations each).  The stored entries are those of the operator that is built."""
    faults = _faults(case, 1)
    n, kind = sum(len(c) for _, c in faults), case["kind"]
    nin, nout = hbi.OP_NIN[case["op"]], hbi.OP_NOUT[case["op"]]
    fr = _friction(case, 1, faults)
    st = hbi.hbi_stats(_build(case, faults, np.split(fr[3], np.cumsum([len(c) for _, c in faults])[:-1])))
    lr, de = ELEM_BYTES[case["storage"]]
    entries = st["entries_lowrank"] + st["entries_dense"]
    product = st["entries_lowrank"] * lr + st["entries_dense"] * de
    if kind == "build":
        return dict(bytes=product + 8 * (nin + nout) * n, flops=252.0 * entries)
    if kind in ("product", "transpose", "multi"):
        k = case.get("k", 1)
        return dict(bytes=product + 8 * k * (nin + nout) * n, flops=2.0 * entries * k)
    per_step = 12 if kind == "gradient" else 6
    words = 4 if kind != "vector" else 6
    return dict(bytes=case["steps"] * (per_step * product + 16 * words * n), flops=2.0 * per_step * case["steps"] * entries)


# ------------------------------------------------------------------ the same in 64 bits, densely
def _entries(v, rake, op, rows):
    """Rows of the dense stress operator of one fault's elements (uniform slip, collocated at the
    centres) for the receivers `rows`: (n_out, rows, n_in, n).  Each straight edge of an element
    contributes the Peach-Koehler line integral of a dislocation segment in closed form."""
    v = _T(v)
    nv = v.shape[1]
    c = v.mean(1)
    nrm = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    up = torch.zeros_like(nrm)
    up[:, 2] = 1.0
    st = torch.linalg.cross(up, nrm)
    st = st / st.norm(dim=1, keepdim=True)
    dp = torch.linalg.cross(nrm, st)
    dot = lambda a, b: a @ b.T          # receivers x sources
    xr, recv = c[rows], [st[rows], dp[rows], nrm[rows]]
    out = torch.zeros(3, len(rows), 2, len(v), dtype=torch.float64, device="cuda")
    for e in range(nv):
        p0, p1 = v[:, e], v[:, (e + 1) % nv]
        t = p1 - p0
        length = t.norm(dim=1)
        t = t / length[:, None]
        w = [p0[None, :, k] - xr[:, None, k] for k in range(3)]      # first end minus receiver
        s0 = sum(w[k] * t[None, :, k] for k in range(3))
        p = [w[k] - s0 * t[None, :, k] for k in range(3)]            # the perpendicular to the line
        p2 = sum(q * q for q in p)
        s1 = s0 + length[None, :]
        R0, R1 = (p2 + s0 * s0).sqrt(), (p2 + s1 * s1).sqrt()
        i30 = (s1 / R1 - s0 / R0) / p2
        i31 = 1 / R0 - 1 / R1
        i50 = (s1 / R1 ** 3 - s0 / R0 ** 3) / (3 * p2) + 2 / (3 * p2) * i30
        i51 = (1 / R0 ** 3 - 1 / R1 ** 3) / 3
        i52 = ((s1 / R1) ** 3 - (s0 / R0) ** 3) / (3 * p2)
        A = [p[k] * i30 + t[None, :, k] * i31 for k in range(3)]     # integral of rho / R^3
        pv = [sum(p[k] * r[:, None, k] for k in range(3)) for r in recv]
        tv = [dot(r, t) for r in recv]
        Av = [sum(A[k] * r[:, None, k] for k in range(3)) for r in recv]
        for q, b in enumerate((st, dp)):
            cb = torch.linalg.cross(b, t)
            Axb = [A[1] * b[None, :, 2] - A[2] * b[None, :, 1], A[2] * b[None, :, 0] - A[0] * b[None, :, 2],
                   A[0] * b[None, :, 1] - A[1] * b[None, :, 0]]
            gv = [-2 * sum(Axb[k] * r[:, None, k] for k in range(3)) for r in recv]
            pc = sum(p[k] * cb[None, :, k] for k in range(3))
            cA = sum(A[k] * cb[None, :, k] for k in range(3))
            cv = [dot(r, cb) for r in recv]
            for o, u in enumerate((0, 1, 2)):                        # traction component u of the normal's plane
                same = 1.0 if u == 2 else 0.0                        # n . u
                term = 3 * pc * (pv[2] * pv[u] * i50 + (pv[2] * tv[u] + pv[u] * tv[2]) * i51 + tv[2] * tv[u] * i52)
                term = term - (cv[2] * Av[u] + cv[u] * Av[2] + same * cA) + 2 * same * cA
                sig = MU / (8 * math.pi) * (gv[2] * tv[u] + gv[u] * tv[2]) + MU / (4 * math.pi * (1 - NU)) * term
                out[o, :, q] += sig if u < 2 else -sig
    if op in (2, 3):
        return out[:op]
    r = _T(rake)
    col = out[:, :, 0] * r.cos() + out[:, :, 1] * r.sin()
    rr = r[rows][:, None]
    shear = col[0] * rr.cos() + col[1] * rr.sin()
    return (shear[None] if op == 0 else torch.stack([shear, col[2]]))[:, :, None]


def _dense(case, faults, rakes):
    """Each fault's dense operator, (n_out n) x (n_in n)."""
    out = []
    for (v, c), rake in zip(faults, rakes):
        n = len(c)
        nin, nout = hbi.OP_NIN[case["op"]], hbi.OP_NOUT[case["op"]]
        A = torch.empty(nout, n, nin, n, dtype=torch.float64, device="cuda")
        for r in torch.arange(n, device="cuda").split(max(1, 12_000_000 // n)):
            A[:, r] = _entries(v, rake, case["op"], r)
        out.append(A.reshape(nout * n, nin * n))
    return out


def _rhs(case, S, y, fr):
    """dy/dt and V of one fault (y: components x n) with the stress-rate operator S."""
    a, b, dc, rake = fr
    eta = MU / (2 * CS)
    n = a.shape[0]
    nin, nout = hbi.OP_NIN[case["op"]], hbi.OP_NOUT[case["op"]]
    rate = lambda f: (V0 * (torch.exp((f - y[0]) / a) - torch.exp((-f - y[0]) / a)),
                      V0 * (torch.exp((f - y[0]) / a) + torch.exp((-f - y[0]) / a)) / (a * y[-1]))
    if case["kind"] == "vector":
        tn = (y[1] ** 2 + y[2] ** 2).sqrt()
        u = torch.stack([y[1] / tn, y[2] / tn])
        g, g1 = rate(tn / y[3])
        V = g * u
        s = (S @ (V - VPL * torch.stack([rake.cos(), rake.sin()])).reshape(-1)).reshape(nout, n)
        dphi = b / dc * (V0 * torch.exp((F0 - y[0]) / b) - g)
        dsig = s[2] if nout == 3 else torch.zeros_like(g)
        r = s[:2] - eta * (-g / a * dphi - tn / y[3] * g1 * dsig) * u
        par = (r * u).sum(0)
        dt = par / (1 + eta * g1) * u + (r - par * u) / (1 + eta * g / tn)
        return torch.stack([dphi, dt[0], dt[1], dsig]), V
    q = y[1] / y[2]
    V, g1 = rate(q)
    x = V - VPL
    s = (S @ (x if nin == 1 else torch.cat([x * rake.cos(), x * rake.sin()]))).reshape(nout, n)
    shear = s[0] if nin == 1 else rake.cos() * s[0] + rake.sin() * s[1]
    dsig = s[-1] if nout in (2, 3) and not (nin == 2 and nout == 2) else torch.zeros_like(V)
    dphi = b / dc * (V0 * torch.exp((F0 - y[0]) / b) - V)
    dtau = (shear - eta * (-q * g1 * dsig - V / a * dphi)) / (1 + eta * g1)
    return torch.stack([dphi, dtau, dsig]), V


CK_A = [[], [1 / 5], [3 / 40, 9 / 40], [3 / 10, -9 / 10, 6 / 5], [-11 / 54, 5 / 2, -70 / 27, 35 / 27],
        [1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096]]
CK_5 = [37 / 378, 0, 250 / 621, 125 / 594, 0, 512 / 1771]
CK_4 = [2825 / 27648, 0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4]


def _cash_karp(case, S, y, fr, dt):
    k = []
    for row in CK_A:
        k.append(_rhs(case, S, y + dt * sum(c * q for c, q in zip(row, k)) if row else y, fr)[0])
    return [y + dt * sum(c * q for c, q in zip(w, k)) for w in (CK_5, CK_4)]


def _adaptive(case, S, y, D, fr, dt):
    """`steps` accepted Cash-Karp steps: state, time, next step size and step records."""
    t, rejects, rec, vec = 0.0, 0, [], case["kind"] == "vector"
    V = _rhs(case, S, y, fr)[1]
    while len(rec) < case["steps"]:
        y5, y4 = _cash_karp(case, S, y, fr, dt)
        d, m = (y5 - y4).abs(), y5.abs()
        if vec:
            d = torch.stack([d[0], (d[1] ** 2 + d[2] ** 2).sqrt(), d[3]])
            m = torch.stack([m[0], (m[1] ** 2 + m[2] ** 2).sqrt(), m[3]])
        err = float((d / m.clamp_min(1e-30)).max())
        if not err <= EPS_RK:
            rejects += 1
            dt = max(dt / 2, 0.9 * dt * (err / EPS_RK) ** -0.25)
            continue
        V5 = _rhs(case, S, y5, fr)[1]
        y, D, t = y5, D + 0.5 * dt * (V + V5), t + dt
        V = V5
        speed = V.norm(dim=0) if vec else V.abs()
        shear = y[1:3].norm(dim=0) if vec else y[1]
        rec.append([t, dt, float(speed.max()), rejects, float((shear / y[-1]).mean())])
        rejects, dt = 0, min(2 * dt, 0.9 * dt * (err / EPS_RK) ** -0.2)
    return y, D, t, dt, np.array(rec)


def exact(case, seed):
    faults = _faults(case, seed)
    kind, n = case["kind"], sum(len(c) for _, c in faults)
    if n > 45000 or (n > 21000 and kind not in ("product", "multi", "build")):
        return None   # the dense operator takes too long, or too much memory to keep
    fr = _friction(case, seed, faults)
    at = np.cumsum([len(c) for _, c in faults])[:-1]
    rakes = np.split(fr[3], at)
    nin, nout = hbi.OP_NIN[case["op"]], hbi.OP_NOUT[case["op"]]
    if kind in ("product", "multi", "build"):
        k = case.get("k", 1)
        X = _T(_input(case, seed, faults, k, nin)).reshape(k, nin * n).T.contiguous()
        Y = torch.empty(nout, n, k, dtype=torch.float64, device="cuda")
        for r in torch.arange(n, device="cuda").split(max(1, 12_000_000 // n)):
            E = _entries(faults[0][0], rakes[0], case["op"], r)
            Y[:, r] = (E.reshape(-1, nin * n) @ X).reshape(nout, len(r), k)
        return Y.reshape(nout * n, k).T.contiguous().reshape(-1)
    S = _dense(case, faults, rakes)
    if kind == "transpose":
        return S[0].T @ _T(_input(case, seed, faults, 1, nout))
    if kind == "gradient":
        amb, dc = _T(fr[0] - fr[1]).requires_grad_(), _T(fr[2]).requires_grad_()
        b, rake = _T(fr[1]), _T(fr[3])
        y0 = _T(_state0(case, fr)).reshape(4, n)
        y, D = y0[:3], y0[3]
        f = (b + amb, b, dc, rake)
        V = _rhs(case, S[0], y, f)[1]
        for dt in _steps_of(case):
            y = _cash_karp(case, S[0], y, f, float(dt))[0]
            V1 = _rhs(case, S[0], y, f)[1]
            D, V = D + 0.5 * float(dt) * (V + V1), V1
        target = _T(np.log(fr[4]) + 0.1 * _rng(case, seed, 4).standard_normal(n))
        loss = 0.5 * ((V.log() - target) ** 2).sum()
        ga, gd = torch.autograd.grad(loss, (amb, dc))
        return dict(loss=float(loss), grad_amb=ga, grad_dc=gd, state=torch.cat([y.detach().reshape(-1), D.detach()]))
    words = 6 if kind == "vector" else 4
    ny, nd = (4, 2) if kind == "vector" else (3, 1)
    s0 = _T(_state0(case, fr)).reshape(words, n)
    f = [_T(v) for v in fr[:4]]
    parts, at = [], [0, *at, n]
    for m, Sm in enumerate(S):
        w = slice(int(at[m]), int(at[m + 1]))
        D0 = s0[ny:, w] if kind == "vector" else s0[ny, w]
        parts.append(_adaptive(case, Sm, s0[:ny, w], D0, [v[w] for v in f], 2e4))
    state = torch.cat([torch.cat([p[0] for p in parts], 1), torch.cat([p[1].reshape(nd, -1) for p in parts], 1)])
    rec = [p[4] for p in parts]
    return dict(state=state.reshape(-1), t=_T([p[2] for p in parts]), dt=_T([p[3] for p in parts]), done=None,
                records=rec[0] if kind == "step" else rec)
