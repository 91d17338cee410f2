"""Launch sets and crossing lists where the FP32 walk of the completion has to
hand over to the exact one (ties, grazing lines, lines along edges and cones)
and where its hit words do not fit in shared memory, bit for bit against the
oracle."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


def _check(coord, edges, dirs, bc, angles):
    dirs = np.asarray(dirs, dtype=np.float64)
    dirs = dirs / np.sqrt((dirs * dirs).sum(1))[:, None]
    w = np.full(len(dirs), 1.0 / len(dirs))
    g = rt.Grid(coord, edges, dirs, w, inner_bc=bc)
    o = O.OracleGrid(coord, edges, dirs, w, bc)
    for a in angles:
        x, y = o.angle(a), g.crossings(a)
        for k in y:
            assert np.array_equal(x[k], y[k]), (a, k)
    assert g.info()["lost_rays"] == 0
    g.close()
    o.close()


def _directions(n_theta, n_phi):
    """Along the axes, the theta edges (cones), the phi edges and the phi mid-points, and nearly so."""
    out = [(0, 0, 1), (0, 0, -1), (1, 0, 0), (0, -1, 0), (1, 1, 0), (1, 1, 1), (1, 1e-9, 0), (1e-6, 0, 1)]
    for t in range(1, n_theta):
        for p in (0.0, 0.5, 1.0):
            th, ph = math.pi * t / n_theta, 2 * math.pi * p / n_phi
            for e in (0.0, 3e-8):
                out.append((math.sin(th + e) * math.cos(ph), math.sin(th + e) * math.sin(ph), math.cos(th + e)))
    return out


@pytest.mark.parametrize("coord,n,bc", [
    (I.SPHERICAL, (6, 4, 8), I.CORE_B), (I.SPHERICAL, (5, 3, 5), I.TRANSPARENT), (I.SPHERICAL, (3, 1, 1), I.CORE_B),
    (I.SPHERICAL, (19, 12, 16), I.CORE_B), (I.CYLINDRICAL, (6, 8, 4), I.TRANSPARENT),
    (I.CYLINDRICAL, (5, 5, 6), I.CORE_B), (I.CYLINDRICAL, (1, 1, 1), I.TRANSPARENT), (I.CYLINDRICAL, (2, 7, 1), I.CORE_B)])
def test_degenerate_directions(coord, n, bc):
    edges = I.sph_edges(*n) if coord == I.SPHERICAL else I.cyl_edges(*n)
    d = _directions(max(n[1], 2) if coord == I.SPHERICAL else 6, n[2] if coord == I.SPHERICAL else n[1])
    _check(coord, edges, d, bc, range(len(d)))


def test_axis_grid():
    _check(I.CYLINDRICAL, I.cyl_edges(7, 6, 5, R_min=0.0), _directions(5, 6), I.TRANSPARENT, range(20))


def test_hit_words_past_shared_memory():
    n = (112, 109, 112)  # 1.37e6 voxels: 171 KB of hit words
    _check(I.CYLINDRICAL, I.cyl_edges(*n), I.angle_set(2, 1)[0], I.TRANSPARENT, (1,))
