"""Bulk copies of the tiles against per-thread loads, for the kernels and layouts that
test_gpu_bulk.py does not reach: plans for receivers (the reference-frame kernels' element and
face constants arrive by bulk copy too) and several columns per element.  The same bits; one
trajectory of each kind against the oracle as well.
"""
import numpy as np
import pytest

import workloads as W
from oracle_ref import build, rel_err

pytestmark = pytest.mark.gpu

PML = dict(lo=(-0.5,) * 3, hi=(0.5,) * 3, thickness=0.5, sigma_max=20.0, order=2)


@pytest.fixture(scope="module")
def D():
    from paper_2002_08733_gb300 import build as B, dgmax
    B.build()
    dgmax.load_library()
    return dgmax


def _plan(D, n, p, prec, S, pml, receivers, integrator="lsrk4", flux="upwind", jitter=0.1):
    xyz, tets = W.kuhn_mesh(n, (-1, -1, -1), (1, 1, 1), jitter=jitter, seed=500 + n)
    K = len(tets)
    eps = W.lognormal_material(K, 2.0, 0.3, 501)
    g = D.Solver(xyz, tets, eps, 1.0, p, prec, flux, integrator, W.stable_dt(2.0 / n, p) / 2, S=S,
                 pml=PML if pml else None, max_receivers=1 if receivers else 0)
    return g, xyz, tets, eps


def _compare(D, make, steps=3):
    out = []
    for per_thread in (False, True):
        g = make()
        g.set_tile_loads(per_thread)
        assert g.bulk_tile_loads() == (not per_thread)
        if g.opt.integrator == D.LEAPFROG:
            g.leapfrog_start(0.0)
        g.advance(steps, 0.0)
        g.status()
        out.append((g.state(), g.from_device(g.aux[g.current()]) if g.npml else np.zeros(1)))
    assert all(np.array_equal(a, b) for a, b in zip(*out))


# 6 n^3 S columns, 32 per tile: 1296 and 5184 (a half-full last tile of 16, full tiles), 192 and
# 384 S = 4, 8; rows of K S values start on 16-byte boundaries
@pytest.mark.parametrize("prec,n,S", [("fp32", 6, 1), ("fp32", 2, 4), ("fp32", 3, 4), ("fp32", 3, 8), ("fp64", 3, 1),
                                      ("fp64", 3, 2), ("fp64", 2, 4)])
@pytest.mark.parametrize("pml", [False, True])
@pytest.mark.parametrize("receivers", [False, True])
@pytest.mark.parametrize("integrator,flux", [("lsrk4", "upwind"), ("leapfrog", "central")])
@pytest.mark.parametrize("p", [2, 4])
def test_bulk_equals_per_thread(D, p, integrator, flux, receivers, pml, prec, n, S):
    def make():
        g, xyz, tets, eps = _plan(D, n, p, prec, S, pml, receivers, integrator, flux)
        g.set_sources([W.dipole((0.11, -0.07, 0.05), 2.0, 1.0)] + [None] * (S - 1))
        g.set_state(W.random_state(len(tets), S, p, seed=502) * 1e-2)
        return g
    _compare(D, make, 2)


@pytest.mark.parametrize("variant", [0, 1, 2])
def test_tile_shapes_of_plans_for_receivers(D, variant):
    """32 x 384, 32 x 192, 16 x 192."""
    def make():
        g, xyz, tets, eps = _plan(D, 6, 3, "fp32", 1, False, True)
        g.set_variant(variant)
        g.set_state(W.random_state(len(tets), 1, 3, seed=503))
        return g
    _compare(D, make)


@pytest.mark.parametrize("receivers", [False, True])
def test_incident_faces_of_plans_for_receivers(D, receivers):
    n, p = 6, 2
    xyz, tets = W.kuhn_mesh(n, jitter=0.1, seed=504)
    faces = np.concatenate([W.box_faces(n, tets, 2, 0), W.box_faces(n, tets, 0, 1)])
    wave = dict(E0=(0.8, -0.3, 0.45), direction=(0.0, 0.0, 1.0), speed=1.0, f0=0.3, bw=0.25, t0=0.4)

    def make():
        g = D.Solver(xyz, tets, 1.0, 1.0, p, "fp32", "upwind", "lsrk4", W.stable_dt(1 / n, p) / 2, S=1,
                     max_receivers=1 if receivers else 0)
        g.set_incident(faces, **wave)
        return g
    _compare(D, make, 5)
    a, b = make(), D.Solver(xyz, tets, 1.0, 1.0, p, "fp64", "upwind", "lsrk4", W.stable_dt(1 / n, p) / 2, S=1)
    b.set_incident(faces, **wave)
    for g in (a, b):
        g.advance(5, 0.0)
    assert np.abs(b.state()).max() > 0
    assert rel_err(a.state(), b.state()) < 1e-5      # FP64 (itself compared with the oracle) is the reference


@pytest.mark.parametrize("prec,n,S,expect", [("fp32", 4, 2, False), ("fp32", 4, 3, False), ("fp32", 4, 4, True),
                                             ("fp32", 3, 8, True), ("fp64", 3, 2, True), ("fp64", 3, 3, False)])
def test_which_layouts_have_bulk_copies(D, prec, n, S, expect):
    """Rows on 16-byte boundaries and, with several columns, an element's columns in whole
    16-byte units."""
    g, *_ = _plan(D, n, 2, prec, S, False, False)
    assert g.bulk_tile_loads() == expect


@pytest.mark.parametrize("prec,S,tol", [("fp32", 4, 1e-5), ("fp64", 2, 1e-12)])
@pytest.mark.parametrize("receivers", [False, True])
def test_bulk_copies_of_several_columns_match_oracle(D, receivers, prec, S, tol):
    p, n = 2, 3
    g, xyz, tets, eps = _plan(D, n, p, prec, S, True, receivers)
    srcs = [W.dipole((0.11, -0.07, 0.05), 2.0, 1.0)] + [None] * (S - 1)
    u = W.random_state(len(tets), S, p, seed=505) * 1e-2
    g.set_sources(srcs)
    g.set_state(u)
    assert g.bulk_tile_loads()
    g.advance(3, 0.0)
    o = build(xyz, tets, p, eps, 1.0, "upwind", pml=PML, S=S, sources=srcs)
    ref, aux = o.unpack(o.lsrk4(o.pack(u, np.zeros_like(u)), 0.0, g.dt, 3))
    assert rel_err(g.state(), ref) < 10 * tol        # (the trajectory tolerance of test_gpu_bulk.py)
    assert rel_err(g.from_device(g.aux[g.current()]), aux[g.pml_elements()]) < 10 * tol
