"""Device memory that a plan asks for beyond its fields (CPU only)."""
import pytest

import workloads as W


@pytest.mark.parametrize("mixed,prec,limit", [(False, "fp32", 1384), (False, "fp64", 1906), (True, "fp32", 1014),
                                              (True, "fp64", 1174)])
def test_geometry_bytes_per_element(mixed, prec, limit):
    """Bytes per element of the geometry buffer at p = 3 (mixed orders 3 and 2): of them 66 rows
    of face constants (none in mixed orders) and 40 of the tangential kernel, in the plan's
    precision.  The penalty needs no rows of its own."""
    from paper_2002_08733_gb300 import build, dgmax as D
    build.build()
    D.load_library()

    def size(n, **kw):
        xyz, tets = W.kuhn_mesh(n)
        g = D.Plan(xyz, tets, 1.0, 1.0, 2 if mixed else 3, prec, kw.get("flux", "upwind"), "lsrk4", 1e-3,
                   mixed=mixed, sip=kw.get("sip"))
        return len(tets), g.info.bytes_geom

    (k0, b0), (k1, b1) = size(6), size(10)
    assert (b1 - b0) / (k1 - k0) < limit
    if not mixed:
        assert size(6, sip=4.0, flux="central")[1] == b0
