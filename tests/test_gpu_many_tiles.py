"""The shapes that a launch takes by its number of tiles (of 32 columns).

* On meshes that are small in elements but have many columns, so that they pass the lines of
  the dispatch, each shape gives the bits of the 64-bit-index kernel, which always has the
  ordinary shape: the arithmetic of a column does not depend on the shape.
* The shapes of many tiles against the oracle: the residuals of the first two LSRK4 stages
  (r = dt f(u), then r = a_1 r + dt f(u), at the GPU's own u) at sampled elements, to the
  tolerances of one right-hand side (1e-5 and 1e-12 of the max-norm; the second residual is
  a sum of two of them).
* A partition whose parts lie below a line that the whole mesh passes: the same bits.
"""
import numpy as np
import pytest

import workloads as W
from oracle.assemble import Assembly
from oracle.mesh import Mesh
from oracle.solver import LSRK4_A, LSRK4_C, Solver as OSolver
from oracle_ref import rel_err, sigma_of

pytestmark = pytest.mark.gpu

PML = dict(lo=(-0.4,) * 3, hi=(0.4,) * 3, thickness=0.6, sigma_max=15.0, order=2)


@pytest.fixture(scope="module")
def D():
    from paper_2002_08733_gb300 import build as B, dgmax
    B.build()
    dgmax.load_library()
    return dgmax


def _mesh(n):
    xyz, tets = W.kuhn_mesh(n, (-1, -1, -1), (1, 1, 1), jitter=0.1, seed=400 + n)
    K = len(tets)
    return xyz, tets, W.lognormal_material(K, 1.5, 0.2, 401), W.lognormal_material(K, 1.0, 0.1, 402)


def _plan(D, n, S, p, prec, integrator="lsrk4", flux="upwind", pml=False, sip=None):
    import torch
    xyz, tets, eps, mu = _mesh(n)
    g = D.Solver(xyz, tets, eps, mu, p, prec, flux, integrator, W.stable_dt(2.0 / n, p) / 2, S=S,
                 pml=PML if pml else None, sip=sip)
    g.set_sources([W.dipole((0.11, -0.07, 0.05), 2.0, 0.2)] + [None] * (S - 1))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(403)
    for t in [g.fields[0]] + ([g.aux[0]] if g.npml else []) + ([g.hs[0]] if sip else []):
        t.copy_(torch.randn(t.shape, generator=gen, device="cuda", dtype=torch.float32))
    torch.cuda.synchronize()
    return g


def _tiles(n, S):
    return -(-6 * n ** 3 * S // 32)


# columns on both sides of 38, 76, 152 and 304 tiles, and of one element
SIZES = [(1, 1), (6, 1), (5, 3), (6, 2), (6, 4), (6, 8)]
assert [_tiles(n, S) for n, S in SIZES] == [1, 41, 71, 81, 162, 324]


@pytest.mark.parametrize("n,S", SIZES)
@pytest.mark.parametrize("prec,p", [("fp32", 1), ("fp32", 3), ("fp32", 4), ("fp32", 5),
                                    ("fp64", 1), ("fp64", 3), ("fp64", 4)])
@pytest.mark.parametrize("form", ["lsrk", "lsrk_pml", "rhs", "rhs_pml", "lf", "lf_pml", "sip"])
def test_shapes_give_the_same_bits(D, form, prec, p, n, S):
    import torch
    lf, pml, sip = form.startswith("lf"), form.endswith("pml"), 4.0 if form == "sip" else None
    out = []
    for index64 in (False, True):
        g = _plan(D, n, S, p, prec, "leapfrog" if lf else "lsrk4", "central" if lf or sip else "upwind", pml, sip)
        g.set_index64(index64)
        if form.startswith("rhs"):
            r = g.rhs(g.fields[0].clone(), g.aux[0].clone() if g.npml else None, 0.2)   # a caller's buffers
            r = list(r) if g.npml else [r]
        else:
            if lf:
                g.leapfrog_start(0.1)
            g.advance(1, 0.1)
            torch.cuda.synchronize()
            c = g.current()
            r = [g.fields[c]] + ([g.aux[c]] if g.npml else []) + ([g.hs[c]] if sip else [])
            g.status()
        out.append(r)
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("pml", [False, True])
@pytest.mark.parametrize("prec,p,n,S", [("fp32", 1, 6, 4), ("fp32", 2, 6, 4), ("fp32", 3, 6, 4), ("fp32", 4, 6, 8),
                                        ("fp64", 1, 6, 1), ("fp64", 1, 6, 2), ("fp64", 3, 6, 1), ("fp64", 3, 6, 2)])
def test_stages_of_many_tiles_match_oracle(D, prec, p, n, S, pml):
    tol = 1e-5 if prec == "fp32" else 1e-12
    xyz, tets, eps, mu = _mesh(n)
    g = _plan(D, n, S, p, prec, pml=pml)
    mesh = Mesh(xyz, tets)
    src = mesh.locate(np.array([0.11, -0.07, 0.05]))
    rng = np.random.default_rng(404)
    rows = np.unique(np.concatenate([rng.choice(len(tets), 10, replace=False), [0, len(tets) - 1, src]]))
    o = OSolver(Assembly(mesh, p, eps, mu, "upwind", sigma=sigma_of(mesh, PML if pml else None), rows=rows),
                S=S, sources=[W.dipole((0.11, -0.07, 0.05), 2.0, 0.2)] + [None] * (S - 1))
    ref, refa = 0.0, 0.0
    for k in range(2):
        u = g.state()
        aux = np.zeros_like(u)
        if pml:
            aux[g.pml_elements()] = g.from_device(g.aux[g.current()])
        f, fa = o.unpack(o.rhs(o.pack(u, aux) if pml else o.pack(u), 0.1 + LSRK4_C[k] * g.dt))
        ref = LSRK4_A[k] * ref + g.dt * f
        g.stage(k, 0.1)
        g.torch.cuda.synchronize()
        assert rel_err(g.from_device(g.res)[rows], ref) < (1 + k) * tol
        if pml:
            refa = LSRK4_A[k] * refa + g.dt * fa
            at = {int(e): i for i, e in enumerate(g.pml_elements())}
            sel = [i for i, e in enumerate(rows) if int(e) in at]
            assert len(sel) > 2
            got = g.from_device(g.aux_res)[[at[int(rows[i])] for i in sel]]
            assert rel_err(got, refa[sel]) < (1 + k) * tol
    g.status()


@pytest.mark.parametrize("prec,p,n,S,nparts", [("fp32", 2, 5, 8, 2), ("fp32", 4, 6, 8, 2), ("fp64", 2, 6, 1, 2),
                                               ("fp64", 2, 6, 2, 2)])
def test_parts_below_a_line_give_the_bits_of_the_whole(D, prec, p, n, S, nparts):
    xyz, tets, eps, mu = _mesh(n)
    dt = W.stable_dt(2.0 / n, p) / 2
    glob = D.Solver(xyz, tets, eps, mu, p, prec, "upwind", "lsrk4", dt, S=S, pml=PML)
    part = D.partition_slabs(xyz, tets, nparts, axis=2)
    parts = [D.PartitionedSolver(xyz, tets, eps, mu, p, prec, "upwind", dt, part, nparts, r, pml=PML, S=S,
                                 exchange=None) for r in range(nparts)]
    u = W.random_state(len(tets), S, p, seed=405)
    glob.set_state(u)
    for pt in parts:
        pt.set_state(u)
    glob.advance(2, 0.0)
    D.advance_local(parts, 2, 0.0)
    want = glob.state()
    for pt in parts:
        ids, got = pt.owned_state()
        assert np.array_equal(got, want[ids])
