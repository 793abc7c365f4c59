"""Cases that say what the framework is used for, each timed through its public entry points.

A case is one problem (mesh, degree, precision, flux, integrator, options) and a
number of steps; `run` advances it as a user's program does.  Sizes follow the
repository's own workloads (`workloads/`, `bench.py`, the tests): Kuhn grids of
4^3 to 40^3 cubes, degrees 1 to 5, FP32 and FP64 fields, one column or several.
States are random modal fields whose coefficients fall off with the degree, as
those of a resolved field in the middle of a run do.

`exact` is an independent FP64 evaluation of the same problems with plain torch
operations: dense reference operators by quadrature, fluxes from physical traces,
gradients by torch's own automatic differentiation.
"""
import math

import numpy as np
import torch

import workloads as W

AXES = range(3)


# -- the cases ---------------------------------------------------------------------------

def _case(name, kind, n, p, precision="fp32", flux="upwind", integrator="lsrk4", S=1, pml=False,
          jitter=0.0, steps=1, tune=False, option="", receivers=0, cavities=0):
    c = dict(kind=kind, n=n, p=p, precision=precision, flux=flux, integrator=integrator, S=S,
             pml=pml, jitter=jitter, steps=steps, tune=tune, option=option, receivers=receivers,
             cavities=cavities)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest calls: the 4^3 PEC cavity that validates a set-up, FP64 leapfrog,
        # 20 of its steps.  Launch latency and the serial chain of a step decide.
        _case("cavity_leapfrog_fp64", "advance", 4, 2, "fp64", "central", "leapfrog", steps=20),
        # A small scattering problem with a plane wave entering through one side, on an odd,
        # jittered grid with a ragged last tile: what an interactive study steps through.
        _case("incident_fp32", "advance", 9, 2, jitter=0.15, steps=10, option="incident"),
        # The headline workload: 32^3 jittered sphere, p = 3, FP32, tuned once, then stepped.
        _case("sphere_fp32", "advance", 32, 3, jitter=0.15, steps=5, tune=True),
        # The same problem in the plain FP64 method.
        _case("sphere_fp64", "advance", 32, 3, "fp64", jitter=0.15, steps=1),
        # The largest mesh: 40^3, p = 4, a dipole in an unbounded domain (PML), FP32, tuned.
        _case("dipole_pml_fp32", "advance", 40, 4, pml=True, steps=2, tune=True),
        # The paper's integrator with a PML, receivers sampled after every step.
        _case("dipole_leapfrog_fp32", "advance", 24, 4, "fp32", "central", "leapfrog", pml=True,
              steps=4, receivers=32),
        # Many sources on one PML mesh and uneven cavities, advanced together by one graph.
        _case("batch_fp32", "batch", 24, 3, S=16, pml=True, steps=2, cavities=6),
        # One window of the inverse problem: receiver records forward, then the adjoint's
        # gradient with respect to every element's eps and mu.
        _case("inverse_fp32", "inverse", 24, 3, S=8, pml=True, steps=4, receivers=32),
        # One right-hand side for a caller's own integrator: highest degree, three columns
        # (rows that start on no 16-byte boundary), element-wise materials.
        _case("rhs_p5_fp32", "rhs", 11, 5, S=3, jitter=0.1),
        # One step from host memory to host memory.
        _case("host_step_fp32", "host", 32, 3, jitter=0.15),
        # The paper's mixed orders: E of degree 3, H of degree 2.
        _case("mixed_fp32", "advance", 24, 2, jitter=0.15, steps=2, option="mixed"),
        # Central flux with the interior penalty's facet field.
        _case("penalty_fp32", "advance", 24, 3, flux="central", jitter=0.15, steps=3, option="sip"),
    ]


def draw(rng):
    """One more problem of the same ranges; sizes spread over their logarithm."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["advance", "advance", "advance", "rhs", "host", "batch", "inverse"])
    prec = rng.choice(["fp32", "fp32", "fp64"])
    p = rng.randint(1, 4 if prec == "fp64" else 5)
    hi = {1: 40, 2: 36, 3: 32, 4: 26, 5: 20}[p]
    if prec == "fp64":
        hi = {1: 24, 2: 20, 3: 16, 4: 12}[p]
    jit = rng.choice([0.0, 0.1, 0.15])
    if kind == "advance":
        option = rng.choice(["", "", "", "mixed", "sip", "incident"])
        integ = rng.choice(["lsrk4", "lsrk4", "leapfrog"]) if not option else "lsrk4"
        flux = "central" if integ == "leapfrog" or option == "sip" else rng.choice(["upwind", "upwind", "central"])
        if option == "mixed":
            p = min(p, 3)
            hi = 20 if prec == "fp32" else 10
        n = size(3, hi)
        S = rng.choice([1, 1, 2, 3]) if n < 16 else 1
        return _case("", "advance", n, p, prec, flux, integ, S, (not option) and rng.random() < 0.5, jit,
                     rng.randint(1, 6), n >= 10 and rng.random() < 0.5, option,
                     rng.choice([0, 0, 8]) if not option else 0)
    if kind in ("rhs", "host"):
        n = size(3, hi)
        return _case("", kind, n, p, prec, rng.choice(["upwind", "central"]), "lsrk4",
                     rng.choice([1, 2, 3]) if n < 16 else 1, kind == "rhs" and rng.random() < 0.5, jit)
    if kind == "batch":
        return _case("", "batch", size(4, 14), rng.randint(2, 4), "fp32", "upwind", "lsrk4",
                     rng.randint(2, 16), True, 0.0, rng.randint(1, 4), False, "", 0, rng.randint(1, 6))
    return _case("", "inverse", size(4, 12 if prec == "fp32" else 6), min(p, 3), prec, "upwind", "lsrk4",
                 rng.randint(1, 8), rng.random() < 0.7, jit, rng.randint(2, 6), False, "", rng.choice([8, 32]))


# -- the problems ------------------------------------------------------------------------

def _seeded(*ids):
    return np.random.default_rng([int(i) & 0x7FFFFFFF for i in ids])


def _device():
    return torch.device("cuda", torch.cuda.current_device()) if torch.cuda.is_available() else torch.device("cpu")


def _problem(c, seed):
    """Mesh, materials, sources, receivers and time step of a case (host data)."""
    box = c["pml"] or c["kind"] in ("batch", "inverse")
    lo, hi = ((-1.0,) * 3, (1.0,) * 3) if box else ((0.0,) * 3, (1.0,) * 3)
    n, p = c["n"], c["p"]
    pE = p + 1 if c["option"] == "mixed" else p
    xyz, tets = W.kuhn_mesh(n, lo, hi, c["jitter"], seed + 1)
    K = len(tets)
    rng = _seeded(seed, 2)
    if c["kind"] == "inverse" or c["kind"] == "rhs":
        eps = W.lognormal_material(K, 2.0, 0.3, seed + 3)
    elif box or c["integrator"] == "leapfrog":
        eps = np.full(K, 1.0 + rng.uniform())
    else:
        eps = W.sphere_material(xyz, tets, (0.5, 0.5, 0.5), 0.25, 2.0 + 4.0 * rng.uniform(), 1.0)
    mu = W.lognormal_material(K, 1.0, 0.1, seed + 4) if c["kind"] in ("inverse", "rhs") else np.ones(K)
    pml = dict(lo=(-0.75,) * 3, hi=(0.75,) * 3, thickness=0.25, sigma_max=40.0, order=2) if c["pml"] else None
    sources = None
    if box:   # one z dipole per column, in the middle of its pulse
        sources = [W.dipole(rng.uniform(-0.6, 0.6, size=3), rng.uniform(1.0, 4.0), 1.0) for _ in range(c["S"])]
    rec = rng.uniform(-0.6, 0.6, size=(c["receivers"], 3)) if box else rng.uniform(0.1, 0.9, size=(c["receivers"], 3))
    wave = None
    if c["option"] == "incident":
        wave = dict(faces=W.box_faces(n, tets, 2, 0), E0=(1.0, 0.3, 0.0), direction=(0.0, 0.0, 1.0), speed=1.0,
                    f0=1.0 + rng.uniform(), bw=0.5, t0=0.6)
    return dict(xyz=xyz, tets=tets, K=K, eps=eps, mu=mu, pml=pml, sources=sources, rec=rec, wave=wave, pE=pE,
                dt=W.stable_dt((hi[0] - lo[0]) / n, pE), t=0.5)


def _fields(shape, degrees, seed, dev, dtype):
    """Random coefficients, mode of total degree d scaled by 2^-d, on the device."""
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    u = torch.randn(shape, generator=g, device=dev, dtype=torch.float32)
    s = torch.tensor([2.0 ** -d for d in degrees], device=dev, dtype=torch.float32)
    return u.mul_(s.view((-1, 1, 1) if len(shape) == 3 else (1, -1, 1, 1))).to(dtype)


def _degrees(p):
    return [d for d in range(p + 1) for _ in range((d + 1) * (d + 2) // 2)]


def _start(c, K, seed, dev, dtype):
    """The initial state in the fields' layout: [6][N][K][S], or rows of a mixed-order plan."""
    if c["option"] == "mixed":
        dE, dH = _degrees(c["p"] + 1), _degrees(c["p"])
        return _fields((3 * (len(dE) + len(dH)), K, c["S"]), dE * 3 + dH * 3, seed + 5, dev, dtype)
    d = _degrees(c["p"])
    return _fields((6, len(d), K, c["S"]), d, seed + 5, dev, dtype)


ALPHA = 10.0   # the interior penalty's parameter


def _solver(c, q, dev):
    from paper_2002_08733_gb300 import dgmax as D
    D.load_library()
    g = D.Solver(q["xyz"], q["tets"], q["eps"], q["mu"], c["p"], c["precision"], c["flux"], c["integrator"],
                 q["dt"], S=c["S"], pml=q["pml"], max_receivers=len(q["rec"]), device=dev,
                 mixed=c["option"] == "mixed", sip=ALPHA if c["option"] == "sip" else None)
    if q["sources"]:
        g.set_sources(q["sources"])
    if len(q["rec"]):
        g.set_receivers(q["rec"])
    if q["wave"]:
        w = dict(q["wave"])
        g.set_incident(w.pop("faces"), **w)
    return g


def _cavities(c, seed):
    """The batch's uneven cavities: n in 6..20, p in 2..5, the sizes part of the case."""
    return [_case("", "advance", 6 + (5 * i + c["n"]) % 15, 2 + (3 * i + c["p"]) % 4) for i in range(c["cavities"])]


def prepare(case, seed):
    c, dev = case, _device()
    q = _problem(c, seed)
    g = _solver(c, q, dev)
    u = _start(c, q["K"], seed, dev, g.dtype)
    s = dict(case=c, g=g, t=q["t"])
    if c["kind"] == "host":
        s["host_in"] = u.cpu().pin_memory()
        s["host_out"] = torch.empty_like(s["host_in"]).pin_memory()
        return s
    if c["kind"] == "rhs":
        s["u"] = u
        s["aux"] = _fields(tuple(g.aux[0].shape), _degrees(c["p"]), seed + 6, dev, g.dtype) if g.npml else None
        return s
    g.fields[g.current()].copy_(u)
    if g.npml:
        g.aux[g.current()].copy_(_fields(tuple(g.aux[0].shape), _degrees(c["p"]), seed + 6, dev, g.dtype))
    if c["option"] == "sip":
        d = [k for k in range(c["p"] + 1) for _ in range(k + 1)]
        g.hs[g.current()].copy_(_fields(tuple(g.hs[0].shape), d, seed + 7, dev, g.dtype) * 0.1)
    torch.cuda.synchronize(dev)
    if c["kind"] == "inverse":
        s["u"], s["a"] = u, g.aux[g.current()].clone() if g.npml else None
        s["eps"], s["mu"] = q["eps"], q["mu"]
        s["ws"] = g.adjoint_workspace(c["steps"])
        s["target"] = _target(c, seed, dev)
        return s
    if c["integrator"] == "leapfrog":
        g.leapfrog_start(q["t"])
    if c["tune"] and c["integrator"] == "lsrk4" and c["option"] != "mixed":
        g.autotune()
    if c["kind"] == "batch":
        from paper_2002_08733_gb300 import dgmax as D
        s["members"] = [g]
        for i, cc in enumerate(_cavities(c, seed)):
            m = _solver(cc, _problem(cc, seed + 100 * (i + 1)), dev)
            m.fields[m.current()].copy_(_start(cc, m.K, seed + 100 * (i + 1), dev, m.dtype))
            s["members"].append(m)
        torch.cuda.synchronize(dev)
        s["batch"] = D.Batch(s["members"])
        s["batch"].t[:] = q["t"]
    return s


def _target(c, seed, dev):
    """Observed records of the inverse problem [step][column][receiver][component]."""
    g = torch.Generator(device=dev)
    g.manual_seed((int(seed) + 8) & 0x7FFFFFFFFFFF)
    return torch.randn((c["steps"], c["S"], c["receivers"], 3), generator=g, device=dev, dtype=torch.float64)


def run(state):
    c, g = state["case"], state["g"]
    if c["kind"] == "rhs":
        out = g.rhs(state["u"], state["aux"], state["t"])
        return {"du": out[0], "daux": out[1]} if g.npml else {"du": out}
    if c["kind"] == "host":
        g.advance_host(state["host_in"], state["host_out"], 1, state["t"])
        return {"fields": state["host_out"]}
    if c["kind"] == "inverse":
        # one gradient of the misfit 1/2 sum |E - E*|^2 over the window
        g.fields[g.current()].copy_(state["u"])
        if g.npml:
            g.aux[g.current()].copy_(state["a"])
        g.set_materials(state["eps"], state["mu"])
        rec = g.forward_record(c["steps"], state["t"], state["ws"])
        deps, dmu = g.adjoint(c["steps"], state["t"], rec - state["target"], state["ws"])
        return {"records": rec, "deps": deps, "dmu": dmu}
    if c["kind"] == "batch":
        state["batch"].advance(c["steps"])
        return {"fields%d" % i: m.fields[m.current()] for i, m in enumerate(state["members"])}
    out = {}
    if c["receivers"]:
        rec = []
        for k in range(c["steps"]):
            g.advance(1, state["t"])
            rec.append(g.sample_receivers())
            state["t"] += g.dt
        out["records"] = torch.stack(rec)
    else:
        g.advance(c["steps"], state["t"])
        state["t"] += c["steps"] * g.dt
    out["fields"] = g.fields[g.current()]
    if g.npml:
        out["aux"] = g.aux[g.current()]
    if c["option"] == "sip":
        out["facets"] = g.hs[g.current()]
    return out


# -- what a pass cannot do without -------------------------------------------------------

def _launches(c):
    """(state buffers read or written per unknown, stages) of one pass."""
    if c["kind"] == "rhs":
        return 2, 1
    if c["integrator"] == "leapfrog":
        return 3 * c["steps"], 2 * c["steps"]   # per step: one field read and written, the other read, twice half
    n = 1 if c["kind"] == "host" else c["steps"]
    return 19 * n, 5 * n                        # u read, u and the residual written, the residual read in four stages


def _nonzeros(p):
    S, R = _operators(p)
    return int((np.abs(S) > 1e-12).sum()), int((np.abs(R) > 1e-12).sum())


def _one(c, scale_bytes=1.0, scale_flops=1.0):
    pE = c["p"] + 1 if c["option"] == "mixed" else c["p"]
    rows = 3 * (W.n_modes(pE) + W.n_modes(c["p"]))
    nS, nR = _nonzeros(pE)
    K, rs = 6 * c["n"] ** 3, 8 if c["precision"] == "fp64" else 4
    cols = K * c["S"]
    moves, stages = _launches(c)
    if c["pml"]:   # the layer outside [-0.75, 0.75]^3 holds auxiliaries
        rows *= 1.0 + (1.0 - 0.75 ** 3)
    geo = 5 * 9 * rs + 16                       # metric, flux coefficients and neighbours per element
    # curl, tangential traces (once per element) and their lift, 3x3 mass block, update
    flops = 2.0 * (4 * nS + 8 * nR) + 16.0 * W.n_face_modes(pE) * 4 + 10.0 * rows
    if c["integrator"] == "leapfrog":
        flops /= 2
    b = moves * rows * rs * cols + stages * geo * K
    if c["option"] == "sip":
        b += (5 * stages - stages // 5) * 3 * W.n_face_modes(pE) * rs * 2 * K   # two facets an element
    return scale_bytes * b, scale_flops * flops * cols * stages


def work(case):
    b, f = _one(case)
    for cc in _cavities(case, 0) if case["kind"] == "batch" else []:
        x = _one(dict(cc, steps=case["steps"]))
        b, f = b + x[0], f + x[1]
    if case["kind"] == "inverse":   # forward, recomputed forward, adjoint sweep
        b, f = 3 * b, 3 * f
    return {"bytes": b, "flops": f}


# -- the same in 64 bits, plain torch ----------------------------------------------------

def _jacobi(n, a, x):
    """P_n^(a,0) by the three-term recurrence."""
    p0, p1 = np.ones_like(x), 0.5 * ((a + 2.0) * x + a)
    if n == 0:
        return p0
    for m in range(2, n + 1):
        c1 = 2.0 * m * (m + a) * (2.0 * m + a - 2.0)
        c3 = (2.0 * m + a - 2.0) * (2.0 * m + a - 1.0) * (2.0 * m + a)
        c4 = 2.0 * (m + a - 1.0) * (m - 1.0) * (2.0 * m + a)
        p0, p1 = p1, (((2.0 * m + a - 1.0) * a * a + c3 * x) * p1 - c4 * p0) / c1
    return p1


def _basis(p, X):
    """Orthonormal modes (graded by degree, then i, then j) at reference points X [n, 3]."""
    x, y, z = (X[:, a].astype(np.complex128 if np.iscomplexobj(X) else np.float64) for a in AXES)
    out = []
    for d in range(p + 1):
        for i in range(d + 1):
            for j in range(d - i + 1):
                k = d - i - j
                f = _jacobi(i, 0.0, 2 * z / (1 - x - y) - 1) * (1 - x - y) ** i
                f = f * _jacobi(j, 2 * i + 1.0, 2 * y / (1 - x) - 1) * (1 - x) ** j
                f = f * _jacobi(k, 2 * i + 2 * j + 2.0, 2 * x - 1)
                out.append(f * math.sqrt(2.0 * (2 * i + 1) * (i + j + 1) * (2 * d + 3)))
    return np.stack(out, axis=1)


def _face_basis(p, X):
    s, t = X[:, 0], X[:, 1]
    out = []
    for d in range(p + 1):
        for i in range(d + 1):
            f = _jacobi(i, 0.0, 2 * t / (1 - s) - 1) * (1 - s) ** i * _jacobi(d - i, 2 * i + 1.0, 2 * s - 1)
            out.append(f * math.sqrt(2.0 * (2 * i + 1) * (d + 1)))
    return np.stack(out, axis=1)


def _tri(q):
    g, w = np.polynomial.legendre.leggauss(q)
    s = 0.5 * (1 + g)[None, :] + 0 * g[:, None]
    t = 0.5 * (1 + g)[:, None] * (1 - s)
    return np.stack([s.ravel(), t.ravel()], 1), (w[:, None] * w[None, :] * (1 - s) / 4).ravel()


def _tet(q):
    g, w = np.polynomial.legendre.leggauss(q)
    u = 0.5 * (1 + g)
    A, B, C = np.meshgrid(u, u, u, indexing="ij")
    WW = np.einsum("a,b,c->abc", w, w, w) / 8
    x, y = C, B * (1 - C)
    return np.stack([x.ravel(), y.ravel(), (A * (1 - x - y)).ravel()], 1), (WW * (1 - x) * (1 - x - y)).ravel()


_OPS = {}


def _operators(p):
    """S[a, l, m] = int phi_l d_a phi_m and R[f, m, l] = int_face psi_m phi_l."""
    if p not in _OPS:
        X, w = _tet(p + 3)
        v = _basis(p, X)
        S = []
        for a in AXES:
            Z = X.astype(np.complex128)
            Z[:, a] += 1e-30j
            S.append(np.einsum("q,ql,qm->lm", w, v, _basis(p, Z).imag / 1e-30))
        P, wf = _tri(p + 3)
        ref = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1.0]])
        R = []
        for f in range(4):
            a, b, c = ref[[i for i in range(4) if i != f]]
            Y = a + P[:, :1] * (b - a) + P[:, 1:] * (c - a)
            R.append(np.einsum("q,qm,ql->ml", wf, _face_basis(p, P), _basis(p, Y)))
        _OPS[p] = np.stack(S), np.stack(R)
    return _OPS[p]


LSRK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
          -1275806237668 / 842570457699)
LSRK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
          3134564353537 / 4481467310338, 2277821191437 / 14882151754819)
LSRK_C = (0.0, 1432997174477 / 9575080441755, 2526269341429 / 6820363962896, 2006345519317 / 3224310063776,
          2802321613138 / 2924317926251)


class _Exact:
    """The semi-discrete problem of one plan; fields [6][N][K][S] in FP64."""

    def __init__(self, c, q, dev):
        self.c, self.q, self.dev = c, q, dev
        self.p = q["pE"]
        self.upwind, self.sip = c["flux"] == "upwind", ALPHA if c["option"] == "sip" else 0.0
        tets = np.sort(np.asarray(q["tets"]), axis=1)
        V = np.asarray(q["xyz"])[tets]
        K = self.K = len(tets)
        A = np.transpose(V[:, 1:] - V[:, :1], (0, 2, 1))
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        M = np.transpose(np.linalg.inv(A), (0, 2, 1))
        det = np.linalg.det(A)
        self.A, self.M, self.det, self.V, self.Anp = T(A), T(M), T(det), V, A
        self.sgn = torch.sign(self.det)
        S, R = _operators(self.p)
        self.S, self.R = T(S), T(R)
        self.N, self.NF = S.shape[1], R.shape[1]
        self.NH = W.n_modes(c["p"])
        # neighbours: faces by their sorted vertices
        loc = [[i for i in range(4) if i != f] for f in range(4)]
        F = np.concatenate([tets[:, l] for l in loc])          # face id f K + e
        o = np.lexsort((F[:, 2], F[:, 1], F[:, 0]))
        same = np.all(F[o[1:]] == F[o[:-1]], axis=1)
        nb = np.full(4 * K, -1, dtype=np.int64)
        nb[o[1:][same]], nb[o[:-1][same]] = o[:-1][same], o[1:][same]
        self.nb = torch.as_tensor(nb, device=dev).view(4, K)
        m = np.array([[1, 1, 1], [-1, 0, 0], [0, -1, 0], [0, 0, -1.0]])
        vn = np.einsum("erc,fc->fer", M, m)
        ln = np.linalg.norm(vn, axis=2)
        self.n, self.twoF = T(vn / ln[..., None]), T(np.abs(det)[None] * ln)
        self.inc = torch.zeros(4, K, dtype=torch.bool, device=dev)
        if q["wave"]:
            want = {tuple(sorted(v)) for v in q["wave"]["faces"].tolist()}
            b = np.nonzero(nb < 0)[0]
            hit = [i for i in b if tuple(F[i].tolist()) in want]
            self.inc.view(-1)[torch.as_tensor(hit, device=dev)] = True
        cen = V.mean(axis=1)
        sig = np.zeros((K, 3))
        if q["pml"]:
            d = np.maximum(0, np.maximum(np.array(q["pml"]["lo"]) - cen, cen - np.array(q["pml"]["hi"])))
            sig = q["pml"]["sigma_max"] * (d / q["pml"]["thickness"]) ** q["pml"]["order"]
        el = np.nonzero(np.any(sig > 0, axis=1))[0]
        self.el = torch.as_tensor(el, device=dev)
        s = T(sig[el])
        self.sig = s
        self.eta = torch.stack([s[:, 1] + s[:, 2] - s[:, 0], s[:, 2] + s[:, 0] - s[:, 1], s[:, 0] + s[:, 1] - s[:, 2]], 1)
        self.xi = torch.stack([(s[:, 0] - s[:, 1]) * (s[:, 0] - s[:, 2]), (s[:, 1] - s[:, 2]) * (s[:, 1] - s[:, 0]),
                               (s[:, 2] - s[:, 0]) * (s[:, 2] - s[:, 1])], 1)
        self.eps, self.mu = T(q["eps"]), T(q["mu"])
        self.src = [self._point(r["pos"], r) for r in q["sources"]] if q["sources"] else []
        self.rec = [self._point(r, None) for r in q["rec"]]
        if self.sip:   # facets by (lower element, its local face)
            e = torch.arange(K, device=dev)
            own = (self.nb >= 0) & (self.nb % K > e[None])
            num = torch.cumsum(own.t().reshape(-1).long(), 0).view(K, 4).t() - 1
            self.own = own
            self.facet = torch.where(own, num, torch.where(self.nb >= 0, num.reshape(-1)[self.nb.clamp(min=0)], -1))
            self.nfacets = int(own.sum())

    def _point(self, pos, rec):
        pos = np.asarray(pos, dtype=np.float64)
        lam = np.linalg.solve(self.Anp, (pos - self.V[:, 0])[:, :, None])[:, :, 0]
        e = int(np.nonzero((lam >= -1e-12).all(1) & (lam.sum(1) <= 1 + 1e-12))[0][0])
        phi = torch.as_tensor(_basis(self.p, lam[e:e + 1])[0], dtype=torch.float64, device=self.dev)
        return e, phi, rec

    def _mul(self, mats, v, el=None):
        """mats [K, 3, 3] times the components of v [3][N][K][S]."""
        return torch.einsum("kij,jnks->inks", mats, v)

    def physical(self, D, el):
        """A^T diag(D) A^-T of the elements el."""
        return torch.einsum("kai,ka,kaj->kij", self.A[el], D, self.M[el])

    def rates(self, u, t, hs=None, eps=None, mu=None):
        """Curl, flux and source terms through the mass inverse: du [6][N][K][S] (and dh_s)."""
        eps, mu = self.eps if eps is None else eps, self.mu if mu is None else mu
        K, S = self.K, u.shape[3]
        d = lambda a, v: torch.einsum("lm,mks->lks", self.S[a], v)  # noqa: E731
        curl = lambda v: torch.stack([d(1, v[2]) - d(2, v[1]), d(2, v[0]) - d(0, v[2]), d(0, v[1]) - d(1, v[0])])  # noqa: E731
        sg = self.sgn[None, None, :, None]
        rE, rH = sg * curl(u[3:6]), -sg * curl(u[0:3])
        tr = torch.einsum("fml,clks->cmfks", self.R, u).reshape(6, self.NF, 4 * K, S)   # traces by face id
        X = torch.cat([torch.einsum("kij,jmfks->imfks", self.M, tr[3 * b:3 * b + 3].view(3, self.NF, 4, K, S))
                       for b in (0, 1)]).view(6, self.NF, 4 * K, S)                     # physical
        del tr
        Z = torch.sqrt(mu / eps)
        dhs = torch.zeros_like(hs) if hs is not None else None
        for f in range(4):
            ids = torch.arange(f * K, (f + 1) * K, device=self.dev)
            nb = self.nb[f]
            has = (nb >= 0)
            own = X[:, :, f * K:(f + 1) * K]
            oth = X[:, :, torch.where(has, nb, ids)]
            h4 = has[None, None, :, None]
            i4 = self.inc[f][None, None, :, None]
            one = torch.ones((), dtype=torch.float64, device=self.dev)
            dE = torch.where(h4, oth[:3] - own[:3], torch.where(i4, 0 * one, -2 * one) * own[:3])
            dH = torch.where(h4, oth[3:] - own[3:], torch.where(i4, -2 * one, 0 * one) * own[3:])
            del oth
            if self.q["wave"]:
                dE = dE + self._incident(f, t)[..., None]
            Zp = torch.where(has, Z[torch.where(has, nb % K, torch.arange(K, device=self.dev))], Z)
            n = self.n[f]
            cr = lambda v: torch.stack([n[:, 1, None] * v[2] - n[:, 2, None] * v[1],  # noqa: E731
                                        n[:, 2, None] * v[0] - n[:, 0, None] * v[2],
                                        n[:, 0, None] * v[1] - n[:, 1, None] * v[0]])
            kk = lambda v: v[None, None, :, None]  # noqa: E731
            nE, nH = cr(dE), cr(dH)
            if self.upwind:
                fE = kk(Zp / (Z + Zp)) * nH - kk(1 / (Z + Zp)) * cr(nE)
                fH = kk(Z / (Z + Zp)) * nE + kk(Z * Zp / (Z + Zp)) * cr(nH)
            else:
                fE, fH = 0.5 * nH, 0.5 * nE
            if hs is not None:
                fac = self.facet[f]
                on = (fac >= 0)[None, None, :, None]
                fE = fE + torch.where(on, cr(hs[:, :, fac.clamp(min=0)]), 0 * one)
                o = self.own[f]
                muF = 0.5 * (mu + torch.where(has, mu[torch.where(has, nb % K, torch.arange(K, device=self.dev))], mu))
                dhs[:, :, fac[o]] = (-kk(self.sip / muF) * nE)[:, :, o]
            pull = lambda v: torch.einsum("kji,jmks->imks", self.M, v) * kk(self.twoF[f])  # noqa: E731
            rE = rE + torch.einsum("ml,cmks->clks", self.R[f], pull(fE))
            rH = rH - torch.einsum("ml,cmks->clks", self.R[f], pull(fH))
        for s, (e, phi, r) in enumerate(self.src):
            w = 1.0 / (2.0 * math.pi * r["bw"])
            gt = math.sin(2 * math.pi * r["f0"] * (t - r["t0"])) * math.exp(-(t - r["t0"]) ** 2 / (2 * w * w))
            z = torch.zeros_like(rE)
            z[:, :, e, s] = gt * (self.M[e].t() @ torch.tensor(r["dir"], dtype=torch.float64, device=self.dev))[:, None] * phi
            rE = rE - z
        G = torch.einsum("kai,kaj->kij", self.A, self.A) / self.det.abs()[:, None, None]
        du = torch.cat([self._mul(G / eps[:, None, None], rE), self._mul(G / mu[:, None, None], rH)])
        if self.NH < self.N:
            du[3:, self.NH:] = 0
        return du, dhs

    def _incident(self, f, t):
        """Face modes of 2 E_inc on face f: [3][NF][K]."""
        w = self.q["wave"]
        out = torch.zeros(3, self.NF, self.K, dtype=torch.float64, device=self.dev)
        el = torch.nonzero(self.inc[f]).flatten()
        if len(el) == 0:
            return out
        P, wq = _tri(16)
        a, b, c = (self.V[el.cpu().numpy()][:, i] for i in range(4) if i != f)
        r = a[:, None] + P[None, :, :1] * (b - a)[:, None] + P[None, :, 1:] * (c - a)[:, None]
        x = t - w["t0"] - r @ np.asarray(w["direction"]) / w["speed"]
        s = 1.0 / (2 * math.pi * w["bw"])
        g = np.cos(2 * math.pi * w["f0"] * x) * np.exp(-x ** 2 / (2 * s * s))
        v = 2.0 * np.einsum("q,qm,kq,c->cmk", wq, _face_basis(self.p, P), g, np.asarray(w["E0"]))
        out[:, :, el] = torch.as_tensor(v, device=self.dev)
        return out

    def rhs(self, u, a, t, hs=None, eps=None, mu=None):
        du, dhs = self.rates(u, t, hs, eps, mu)
        if a is None:
            return du, None, dhs
        el = self.el
        da = []
        full = torch.zeros_like(du)
        for b, mat in ((0, self.eps if eps is None else eps), (1, self.mu if mu is None else mu)):
            v, m = u[3 * b:3 * b + 3, :, el], mat[el][None, None, :, None]
            x = a[3 * b:3 * b + 3]
            full[3 * b:3 * b + 3, :, el] = -self._mul(self.physical(self.eta, el), v) - x / m
            da.append(-self._mul(self.physical(self.sig, el), x) + m * self._mul(self.physical(self.xi, el), v))
        return du + full, torch.cat(da), dhs

    def lsrk(self, u, a, t, dt, hs=None, eps=None, mu=None, stage=None):
        ru = ra = rh = 0.0
        stage = stage or self.rhs
        for k in range(5):
            du, da, dh = stage(u, a, t + LSRK_C[k] * dt, hs, eps, mu)
            ru = LSRK_A[k] * ru + dt * du
            u = u + LSRK_B[k] * ru
            if a is not None:
                ra = LSRK_A[k] * ra + dt * da
                a = a + LSRK_B[k] * ra
            if hs is not None:
                rh = LSRK_A[k] * rh + dt * dh
                hs = hs + LSRK_B[k] * rh
        return u, a, hs

    def half(self, u, a, b, t, h):
        """Leapfrog update of field b (0: E, 1: H) over h, then of the other field's auxiliary."""
        u = u.clone()
        o = 1 - b
        x, y = u[3 * b:3 * b + 3], u[3 * o:3 * o + 3]
        du = self.rates(u, t)[0][3 * b:3 * b + 3]
        new = x + h * du
        if a is not None:
            a = a.clone()
            el, mats = self.el, (self.eps, self.mu)
            m, mo = mats[b][el][None, None, :, None], mats[o][el][None, None, :, None]
            D = lambda v: v.t()[:, None, :, None]  # noqa: E731
            ph = lambda v: self._mul(self.M[el], v)  # noqa: E731
            back = lambda v: torch.einsum("kji,jnks->inks", self.A[el], v)  # noqa: E731
            hd = 0.5 * h * D(self.eta)
            X = ((1 - hd) * ph(x[:, :, el]) + h * (ph(du[:, :, el]) - ph(a[3 * b:3 * b + 3]) / m)) / (1 + hd)
            hs = 0.5 * h * D(self.sig)
            Zo = ((1 - hs) * ph(a[3 * o:3 * o + 3]) + h * mo * D(self.xi) * ph(y[:, :, el])) / (1 + hs)
            new[:, :, el] = back(X)
            a[3 * o:3 * o + 3] = back(Zo)
        u[3 * b:3 * b + 3] = new
        return u, a

    def sample(self, u):
        """E at the receivers: [S][R][3]."""
        return torch.stack([torch.einsum("ij,jns,n->si", self.M[e], u[:3, :, e], phi) for e, phi, _ in self.rec], 1)


def _unpack(c, x, u):
    """Rows of a mixed-order plan -> [6][N][K][S] with H's missing modes zero."""
    if c["option"] != "mixed":
        return u
    N, NH, K, S = x.N, x.NH, u.shape[1], u.shape[2]
    out = torch.zeros(6, N, K, S, dtype=u.dtype, device=u.device)
    out[:3] = u[:3 * N].view(3, N, K, S)
    out[3:, :NH] = u[3 * N:].view(3, NH, K, S)
    return out


def _pack(c, x, u):
    if c["option"] != "mixed":
        return u
    return torch.cat([u[:3].reshape(-1, *u.shape[2:]), u[3:, :x.NH].reshape(-1, *u.shape[2:])])


def exact(case, seed):
    c, dev = case, _device()
    if dev.type != "cuda" and 6 * c["n"] ** 3 * c["S"] > 20000:
        return None
    q = _problem(c, seed)
    x = _Exact(c, q, dev)
    dt64 = torch.float64
    real = torch.float64 if c["precision"] == "fp64" else torch.float32   # the inputs as the plan holds them
    u = _unpack(c, x, _start(c, q["K"], seed, dev, real).to(dt64))
    a = _fields((6, x.N, len(x.el), c["S"]), _degrees(c["p"]), seed + 6, dev, real).to(dt64) if c["pml"] and len(x.el) else None
    t, dt = q["t"], q["dt"]
    if c["kind"] == "rhs":
        du, da, _ = x.rhs(u, a, t)
        return {"du": du, "daux": da} if a is not None else {"du": du}
    if c["kind"] == "host":
        return {"fields": x.lsrk(u, a, t, dt)[0].cpu()}
    if c["kind"] == "inverse":
        return _exact_gradient(c, q, x, u, a, seed)
    if c["kind"] == "batch":
        out = {}
        for i, cc in enumerate([c] + _cavities(c, seed)):
            if i:
                qq = _problem(cc, seed + 100 * i)
                x = _Exact(cc, qq, dev)
                u, a, dt = _start(cc, qq["K"], seed + 100 * i, dev, torch.float32).to(dt64), None, qq["dt"]
            for k in range(c["steps"]):
                u, a, _ = x.lsrk(u, a, t + k * dt, dt)
            out["fields%d" % i] = u
        return out
    hs = None
    if c["option"] == "sip":
        d = [k for k in range(c["p"] + 1) for _ in range(k + 1)]
        hs = (_fields((3, x.NF, x.nfacets, c["S"]), d, seed + 7, dev, real) * 0.1).to(dt64)
    rec = []
    if c["integrator"] == "leapfrog":
        u, a = x.half(u, a, 1, t, 0.5 * dt)
    for k in range(c["steps"]):
        if c["integrator"] == "leapfrog":
            u, a = x.half(u, a, 0, t + 0.5 * dt, dt)
            u, a = x.half(u, a, 1, t + dt, dt)
        else:
            u, a, hs = x.lsrk(u, a, t, dt, hs)
        t += dt
        if c["receivers"]:
            rec.append(x.sample(u))
    out = {"records": torch.stack(rec)} if rec else {}
    out["fields"] = _pack(c, x, u)
    if a is not None:
        out["aux"] = a
    if hs is not None:
        out["facets"] = hs
    return out


def _exact_gradient(c, q, x, u, a, seed):
    """Records and the misfit's gradient by automatic differentiation, stage by stage."""
    from torch.utils.checkpoint import checkpoint
    eps, mu = (v.clone().requires_grad_(True) for v in (x.eps, x.mu))
    stage = lambda *args: checkpoint(x.rhs, *args, use_reentrant=False)  # noqa: E731
    rec = []
    for k in range(c["steps"]):
        u, a, _ = x.lsrk(u, a, q["t"] + k * q["dt"], q["dt"], None, eps, mu, stage)
        rec.append(x.sample(u))
    rec = torch.stack(rec)
    (0.5 * ((rec - _target(c, seed, x.dev)) ** 2).sum()).backward()
    return {"records": rec.detach(), "deps": eps.grad, "dmu": mu.grad}
