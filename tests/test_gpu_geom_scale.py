"""The launch set and the crossings of grids whose lengths come in other units:
a power of two scales every length exactly, whatever the unit the lists are the
serial rule's, and the covering walk stays on FP32."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt

pytestmark = pytest.mark.gpu

SPH, CYL = I.SPHERICAL, I.CYLINDRICAL


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


def _edges(coord, n, s):
    e = I.sph_edges(*n) if coord == SPH else I.cyl_edges(*n)
    return (e[0] * s, e[1], e[2]) if coord == SPH else (e[0] * s, e[1], e[2] * s)


@pytest.mark.parametrize("coord,n", [(SPH, (9, 6, 8)), (CYL, (8, 7, 6))])
@pytest.mark.parametrize("s", [2.0 ** 36, 2.0 ** -40, 7e10, 1.5e-13, 3e100])
def test_crossings(coord, n, s):
    d, w = I.angle_set(4, 4)
    bc = I.CORE_B if coord == SPH else I.TRANSPARENT
    g = rt.Grid(coord, _edges(coord, n, s), d, w, inner_bc=bc)
    o = O.OracleGrid(coord, _edges(coord, n, s), d, w, bc)
    g1 = rt.Grid(coord, _edges(coord, n, 1.0), d, w, inner_bc=bc)
    for a in range(0, len(w), 3):
        x, y, z = o.angle(a), g.crossings(a), g1.crossings(a)
        for k in y:
            assert np.array_equal(x[k], y[k]), (a, k)
        if np.frexp(s)[0] == 0.5:
            assert np.array_equal(y["vox"], z["vox"]) and np.array_equal(y["len"], s * z["len"])
    assert g.info()["lost_rays"] == 0
    for q in (g, g1, o):
        q.close()


@pytest.mark.parametrize("coord,n", [(SPH, (65, 33, 65)), (CYL, (65, 65, 65))])
def test_walk_stays_fast(coord, n):
    d, w = I.angle_set(4, 8)
    bc = I.CORE_B if coord == SPH else I.TRANSPARENT

    def trace_ms(s):
        ms = []
        for _ in range(3):
            with rt.Grid(coord, _edges(coord, n, s), d, w, inner_bc=bc) as g:
                ms.append(g.info()["geometry_trace_ms"])
        return min(ms)

    ms = trace_ms(1.0)
    for s in (2.0 ** 36, 2.0 ** -40):  # the same arithmetic (on exact steps alone 9 and 4 times as long)
        assert trace_ms(s) < 2.0 * ms
