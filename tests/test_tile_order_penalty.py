"""The tile order of a new plan with the interior penalty: plain at p = 5, else as without it,
and never in place of an order that the caller has set (CPU only)."""
import ctypes

import pytest

import workloads as W
from paper_2002_08733_gb300 import build as B, dgmax as D


def _order(plan):
    g = ctypes.c_int32()
    assert D._lib.dgm_get_tile_groups(plan.handle, ctypes.byref(g)) == 0
    return g.value


def _plan(p, n, S):
    B.build()
    D.load_library()
    xyz, tets = W.kuhn_mesh(n)
    return D.Plan(xyz, tets, 1.0, 1.0, p, "fp32", "central", "lsrk4", 1e-3, S=S)


# fields of 129 and 80 MB
@pytest.mark.parametrize("p,n,S,want", [(5, 10, 16, 1), (3, 24, 2, 6)])
def test_order_with_the_penalty(p, n, S, want):
    g = _plan(p, n, S)
    assert _order(g) == 6
    assert D._lib.dgm_set_sip(g.handle, ctypes.c_double(4.0)) == 0
    assert _order(g) == want
    assert D._lib.dgm_set_sip(g.handle, ctypes.c_double(0.0)) == 0
    assert _order(g) == 6
    assert D._lib.dgm_set_tile_groups(g.handle, 3) == 0
    assert D._lib.dgm_set_sip(g.handle, ctypes.c_double(4.0)) == 0
    assert _order(g) == 3
