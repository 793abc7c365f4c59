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
