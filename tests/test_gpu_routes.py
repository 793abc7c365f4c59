"""Which kernel a plan runs, and that the choice shows in nothing but time.

FP32 plans run the tangential-trace kernel; those with receivers run
reference-frame kernels that keep the rounding of the records, except with the
interior penalty, which the tangential-trace kernel alone has.
"""
import numpy as np
import pytest

import workloads as W
from oracle.assemble import Assembly
from oracle.mesh import Mesh
from oracle.sip import SipSolver
from oracle.solver import Solver as OSolver
from oracle_ref import rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    from paper_2002_08733_gb300 import build as B, dgmax
    B.build()
    dgmax.load_library()
    return dgmax


# -- interior penalty with receivers ---------------------------------------------------

REC = np.array([[0.31, 0.42, 0.23], [0.77, 0.15, 0.61]])


def _penalty(D, p, n, receivers):
    xyz, tets = W.kuhn_mesh(n, jitter=0.12, seed=301)
    K = len(tets)
    eps = W.lognormal_material(K, 2.0, 0.3, 302)
    mu = W.lognormal_material(K, 1.2, 0.2, 303)
    g = D.Solver(xyz, tets, eps, mu, p, "fp32", "central", "lsrk4", W.stable_dt(1.0 / n, p) / 2, S=2,
                 sip=4.0, max_receivers=len(REC) if receivers else 0)
    if receivers:
        g.set_receivers(REC)
    g.set_state(W.random_state(K, 2, p, seed=304))
    return g, (xyz, tets, eps, mu)


@pytest.mark.parametrize("p,n", [(1, 2), (2, 3), (3, 2), (4, 1), (5, 1)])
def test_penalty_plan_with_receivers_steps(D, p, n):
    """advance, stage and autotune accept the plan, and receivers change no bit of its fields."""
    g, _ = _penalty(D, p, n, True)
    s, _ = _penalty(D, p, n, True)
    r, _ = _penalty(D, p, n, False)
    assert s.autotune()[0] == 0
    g.advance(2, 0.0)
    r.advance(2, 0.0)
    for step in range(2):
        for k in range(5):
            s.stage(k, step * s.dt)
    for o in (r, s):
        assert np.array_equal(g.state(), o.state())
        assert np.array_equal(g.facet_state(), o.facet_state())
    g.status()


@pytest.mark.parametrize("p", [1, 2, 3])
def test_penalty_plan_with_receivers_matches_oracle(D, p):
    """Fields to the FP32 trajectory tolerance of the penalty tests (1e-4 of the max-norm);
    records to 1e-6 of the oracle's evaluation of the same coefficients, as without the penalty."""
    g, (xyz, tets, eps, mu) = _penalty(D, p, 2, True)
    u = g.state()
    g.advance(5, 0.0)
    got = g.state()
    rec = g.sample_receivers().cpu().numpy()
    o = SipSolver(OSolver(Assembly(Mesh(xyz, tets), p, eps, mu, "central"), S=2), 4.0)
    ref, _ = o.unpack(o.lsrk4(o.pack(u), 0.0, g.dt, 5))
    assert rel_err(got, ref) < 1e-4
    plain = OSolver(Assembly(Mesh(xyz, tets), p, eps, mu, "central"), S=2)
    want = np.zeros_like(rec)
    for r, x in enumerate(REC):
        T = plain.asm.mesh.locate(x)
        for s in range(2):
            want[s, r] = plain.evaluate(got[T, s, 0:3].reshape(-1), T, x[None, :])[0]
    assert rel_err(rec, want) < 1e-6


# -- the kernel is the plan's, not the receivers' ----------------------------------------

PML = dict(lo=(-0.4,) * 3, hi=(0.4,) * 3, thickness=0.6, sigma_max=15.0, order=2)


def _plan(D, n, p, integrator="lsrk4", flux="upwind", S=1, pml=True, max_receivers=1, prec="fp32", src=True,
          nseed=0):
    xyz, tets = W.kuhn_mesh(n, (-1, -1, -1), (1, 1, 1), jitter=0.1, seed=310 + n + nseed)
    K = len(tets)
    eps = W.lognormal_material(K, 1.5, 0.2, 311)
    mu = W.lognormal_material(K, 1.0, 0.1, 312)
    g = D.Solver(xyz, tets, eps, mu, p, prec, flux, integrator, W.stable_dt(2.0 / n, p) / 2, S=S,
                 pml=PML if pml else None, max_receivers=max_receivers)
    if src:
        g.set_sources([W.dipole((0.11, -0.07, 0.05), 2.0, 0.2)] + [None] * (S - 1))
    u = W.random_state(K, S, p, seed=313) * 1e-2
    if g.npml:
        g.set_state(u, (W.random_state(K, S, p, seed=314) * 1e-3)[g.pml_elements()])
    else:
        g.set_state(u)
    if integrator == "leapfrog":
        g.leapfrog_start(0.0)
    return g


def _result(g):
    return g.state(), g.from_device(g.aux[g.current()]) if g.npml else np.zeros(1)


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(_result(a), _result(b)))


POINT = np.array([[0.1, 0.2, -0.1]])


@pytest.mark.parametrize("integrator,flux", [("lsrk4", "upwind"), ("leapfrog", "central")])
@pytest.mark.parametrize("p", [2, 4])
def test_setting_receivers_changes_no_bit_of_the_fields(D, p, integrator, flux):
    a = _plan(D, 3, p, integrator, flux)
    b = _plan(D, 3, p, integrator, flux)
    b.set_receivers(POINT)
    a.advance(2, 0.0)
    b.advance(2, 0.0)
    assert _same(a, b)
    a.set_receivers(POINT)          # in the middle of a run
    for g in (a, b):
        g.advance(1, 2 * g.dt)
    assert _same(a, b)


@pytest.mark.parametrize("p", [2, 4])
def test_batch_captured_before_the_receivers_are_set(D, p):
    """The graph's two steps and the odd third step run the same kernel."""
    import torch
    a = _plan(D, 3, p, src=False)
    b = _plan(D, 3, p, src=False)
    batch = D.Batch([a])
    a.set_receivers(POINT)
    batch.advance(3)
    torch.cuda.synchronize()
    b.set_receivers(POINT)
    b.advance(3, 0.0)
    assert _same(a, b)


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n,S,pml", [(1, 1, False), (2, 2, True), (2, 3, False), (3, 1, True), (4, 1, False)])
@pytest.mark.parametrize("integrator,flux", [("leapfrog", "central"), ("lsrk4", "upwind")])
def test_plans_for_receivers_agree_with_plans_without(D, p, n, S, pml, integrator, flux):
    """The two kernels on one problem: to twice the FP32 tolerance of one of them against
    the oracle (1e-5 of the max-norm)."""
    r = []
    for cap in (0, 1):
        g = _plan(D, n, p, integrator, flux, S, pml, cap)
        g.advance(3, 0.0)
        g.status()
        r.append(_result(g))
    assert rel_err(r[0][0], r[1][0]) < 2e-5
    assert not pml or rel_err(r[0][1], r[1][1]) < 2e-5


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("integrator,flux", [("leapfrog", "central"), ("lsrk4", "upwind")])
def test_plans_without_receivers_64_bit_indices(D, p, integrator, flux):
    a, b = (_plan(D, 2, p, integrator, flux, 3, True, 0) for _ in range(2))
    b.set_index64()
    for g in (a, b):
        g.advance(2, 0.0)
    assert _same(a, b)


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n,S", [(1, 1), (2, 3), (3, 1)])
def test_plans_for_receivers_without_a_layer(D, p, n, S):
    """LSRK4 stages of plans without a PML have an instantiation of their own; the 64-bit one
    serves both: the same bits."""
    a, b = (_plan(D, n, p, "lsrk4", "upwind", S, False, 1) for _ in range(2))
    b.set_index64()
    for g in (a, b):
        g.advance(2, 0.0)
    assert _same(a, b)
