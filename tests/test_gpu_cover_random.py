"""The FP32 covering walk on grids of uneven edges and in random directions, some
of them a rounding away from an axis, an edge's cone or an edge's half-plane:
launch sets and crossings are the oracle's, bit for bit."""
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


def _cuts(rng, n, lo, hi, spread):
    w = np.exp(rng.normal(0.0, spread, n))
    e = lo + (hi - lo) * np.concatenate([[0.0], np.cumsum(w) / w.sum()])
    e[-1] = hi
    return e


def _edges(rng, coord):
    n = [int(rng.integers(1, m)) for m in (14, 12, 14)]
    spread = float(rng.choice([0.05, 0.7, 1.5]))
    phi = _cuts(rng, n[2] if coord == I.SPHERICAL else n[1], 0.0, 2.0 * math.pi, spread)
    r0, ratio = 10.0 ** rng.uniform(-2, 2), 10.0 ** rng.uniform(0.05, 4)
    if coord == I.SPHERICAL:
        r = r0 * ratio ** _cuts(rng, n[0], 0.0, 1.0, spread)
        return (r, _cuts(rng, n[1], 0.0, math.pi, spread), phi)
    R = r0 * ratio ** _cuts(rng, n[0], 0.0, 1.0, spread)
    if rng.random() < 0.3:
        R[0] = 0.0
    z = 10.0 ** rng.uniform(-1, 1) * R[-1]
    return (R, phi, _cuts(rng, n[2], -z * rng.uniform(0.2, 1.0), z, spread))


def _directions(rng, coord, edges, count):
    d = rng.normal(size=(count, 3))
    th = edges[1] if coord == I.SPHERICAL else np.array([0.5 * math.pi])
    ph = edges[2] if coord == I.SPHERICAL else edges[1]
    for i in range(0, count, 3):  # near an edge's cone, half-plane or both, or an axis
        t, p = rng.choice(th), rng.choice(ph)
        t = t if rng.random() < 0.7 else rng.uniform(0, math.pi)
        p = p if rng.random() < 0.7 else rng.uniform(0, 2 * math.pi)
        e = rng.choice([0.0, 1e-12, 1e-8, 1e-5], 2) * rng.choice([-1, 1], 2)
        d[i] = (math.sin(t + e[0]) * math.cos(p + e[1]), math.sin(t + e[0]) * math.sin(p + e[1]), math.cos(t + e[0]))
    return d / np.sqrt((d * d).sum(1))[:, None]


@pytest.mark.parametrize("seed", range(24))
def test_random_grids(seed):
    rng = np.random.default_rng(900 + seed)
    coord = I.SPHERICAL if seed % 2 == 0 else I.CYLINDRICAL
    edges = _edges(rng, coord)
    bc = I.CORE_B if edges[0][0] > 0.0 and rng.random() < 0.5 else I.TRANSPARENT
    d = _directions(rng, coord, edges, 24)
    w = np.full(len(d), 1.0 / len(d))
    o = O.OracleGrid(coord, edges, d, w, bc)
    g = rt.Grid(coord, edges, d, w, inner_bc=bc)
    assert g.info()["lost_rays"] == 0
    for a in range(len(w)):
        x, y = o.angle(a), g.crossings(a)
        for k in y:
            assert np.array_equal(x[k], y[k]), (a, k)
    g.close()
    o.close()
