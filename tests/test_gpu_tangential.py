"""The two routes of FP32 plans against each other and against the oracle.

Plans without receivers run the tangential-trace kernel, plans with receivers
the reference-frame kernels that keep the rounding of the records.  Both
evaluate the same system, so after a few steps they agree to twice the FP32
tolerance of one right-hand side against the oracle (1e-5 of the max-norm each).

Sizes at the edges of the tiles: 6 elements (less than half a tile), 48 (one and
a half), 162 (five and two columns); one, two or three columns per element
(rows aligned for bulk copies or not), with and without a PML, a dipole, and
64-bit indices.
"""
import numpy as np
import pytest

import workloads as W
from oracle_ref import build, rel_err

pytestmark = pytest.mark.gpu

TOL = 2e-5
PML = dict(lo=(-0.4,) * 3, hi=(0.4,) * 3, thickness=0.6, sigma_max=15.0, order=2)


@pytest.fixture(scope="module")
def D():
    from paper_2002_08733_gb300 import build as B, dgmax
    B.build()
    dgmax.load_library()
    return dgmax


def _run(D, n, p, integrator, flux, S, pml, receivers, steps, index64=False, prec="fp32"):
    xyz, tets = W.kuhn_mesh(n, (-1, -1, -1), (1, 1, 1), jitter=0.1, seed=200 + n)
    K = len(tets)
    eps = W.lognormal_material(K, 1.5, 0.2, 201)
    mu = W.lognormal_material(K, 1.0, 0.1, 202)
    g = D.Solver(xyz, tets, eps, mu, p, prec, flux, integrator, W.stable_dt(2.0 / n, p) / 2, S=S,
                 pml=PML if pml else None, max_receivers=1)
    g.set_sources([W.dipole((0.11, -0.07, 0.05), 2.0, 0.2)] + [None] * (S - 1))
    if receivers:
        g.set_receivers(np.array([[0.1, 0.2, -0.1]]))
    if index64:
        g.set_index64()
    u = W.random_state(K, S, p, seed=203) * 1e-2
    if g.npml:
        aux = W.random_state(K, S, p, seed=204) * 1e-3
        g.set_state(u, aux[g.pml_elements()])
    else:
        g.set_state(u)
    if integrator == "leapfrog":
        g.leapfrog_start(0.0)
    g.advance(steps, 0.0)
    g.status()
    a = g.from_device(g.aux[g.current()]) if g.npml else np.zeros(1)
    return g.state(), a


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n,S,pml", [(1, 1, False), (2, 2, True), (2, 3, False), (3, 1, True)])
@pytest.mark.parametrize("integrator,flux", [("leapfrog", "central"), ("lsrk4", "upwind")])
def test_routes_with_and_without_receivers_agree(D, p, n, S, pml, integrator, flux):
    a, aa = _run(D, n, p, integrator, flux, S, pml, False, 3)
    b, ba = _run(D, n, p, integrator, flux, S, pml, True, 3)
    assert rel_err(a, b) < TOL
    assert not pml or rel_err(aa, ba) < TOL


@pytest.mark.parametrize("p", [1, 4])
@pytest.mark.parametrize("receivers", [False, True])
@pytest.mark.parametrize("integrator,flux", [("leapfrog", "central"), ("lsrk4", "upwind")])
def test_64_bit_indices_give_the_same_bits(D, p, receivers, integrator, flux):
    a, aa = _run(D, 2, p, integrator, flux, 3, True, receivers, 2)
    b, ba = _run(D, 2, p, integrator, flux, 3, True, receivers, 2, index64=True)
    assert np.array_equal(a, b) and np.array_equal(aa, ba)


@pytest.mark.parametrize("p", [1, 2, 4])
@pytest.mark.parametrize("n,S", [(1, 1), (2, 3), (3, 1)])
def test_leapfrog_with_receivers_matches_oracle(D, p, n, S):
    xyz, tets = W.kuhn_mesh(n, jitter=0.1, seed=210 + n)
    K = len(tets)
    eps = W.lognormal_material(K, 1.5, 0.2, 211)
    dt = W.stable_dt(1.0 / n, p) / 2
    u = W.random_state(K, S, p, seed=212) * 1e-2
    g = D.Solver(xyz, tets, eps, 1.0, p, "fp32", "central", "leapfrog", dt, S=S, max_receivers=1)
    g.set_receivers(np.array([[0.3, 0.4, 0.5]]))
    g.set_state(u)
    g.leapfrog_start(0.0)
    g.advance(3, 0.0)
    o = build(xyz, tets, p, eps, 1.0, "central", S=S)
    ref = o.unpack(o.leapfrog(o.pack(u), 0.0, dt, 3))[0]
    assert rel_err(g.state(), ref) < TOL


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("n,S,pml", [(1, 1, False), (2, 3, True), (5, 1, True), (6, 1, False)])
@pytest.mark.parametrize("integrator,flux", [("leapfrog", "central"), ("lsrk4", "upwind")])
def test_fp64_cluster_agrees_with_one_cta_per_tile(D, p, n, S, pml, integrator, flux):
    """FP64 plans of at most 38 tiles run a cluster of CTAs per tile (n = 1, 2, 5: 1, 5 and
    24 tiles; n = 6: 41, one CTA per tile); 64-bit indices always one CTA.  The same sums of
    a few hundred terms: 1e-13 of the max-norm covers their rounding over three steps."""
    a, aa = _run(D, n, p, integrator, flux, S, pml, False, 3, prec="fp64")
    b, ba = _run(D, n, p, integrator, flux, S, pml, False, 3, index64=True, prec="fp64")
    assert rel_err(a, b) < 1e-13
    assert not pml or rel_err(aa, ba) < 1e-13
