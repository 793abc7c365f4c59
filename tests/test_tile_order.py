"""The tile visiting order that a new plan chooses from its mesh: the plain order where
all tiles run at once, the fields are small against L2, the plan is FP64 or
neighbours are numbered together; an interleaved one where they are numbered in
blocks (a Kuhn grid numbered type by type)."""
import ctypes

import numpy as np
import pytest

import workloads as W
from paper_2002_08733_gb300 import build as B, dgmax as D


def _groups(n, S, cube_by_cube, precision):
    B.build()
    D.load_library()
    xyz, tets = W.kuhn_mesh(n)
    if cube_by_cube:   # the six tetrahedra of a cube one after the other
        tets = tets.reshape(6, n ** 3, 4).transpose(1, 0, 2).reshape(-1, 4)
    p = D.Plan(xyz, np.ascontiguousarray(tets), 1.0, 1.0, 3, precision, "upwind", "lsrk4", 1e-3, S=S)
    g = ctypes.c_int32()
    assert D._lib.dgm_get_tile_groups(p.handle, ctypes.byref(g)) == 0
    return g.value


# fields of 0.2, 5, 80, 99, 80 and 159 MB
@pytest.mark.parametrize("n,S,cube_by_cube,precision,want",
                         [(4, 1, False, "fp32", 1), (12, 1, False, "fp32", 1), (24, 2, False, "fp32", 6),
                          (19, 5, False, "fp32", 6), (24, 2, True, "fp32", 1), (24, 2, False, "fp64", 1)])
def test_chosen_order(n, S, cube_by_cube, precision, want):
    assert _groups(n, S, cube_by_cube, precision) == want
