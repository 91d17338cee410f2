"""The FP64 march and its transpose with one characteristic per lane: groups of
32 characteristics sorted by length, at sizes where the last group is nearly
empty or nearly full, with holes and core starts, one and several angle blocks."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt
from tests.helpers import tiny_problem

pytestmark = pytest.mark.gpu

CASES = [  # coord, n, angles, inner boundary, angle_block
    (I.SPHERICAL, (1, 1, 1), (2, 1), I.CORE_B, 0),       # one voxel: fewer characteristics than lanes
    (I.SPHERICAL, (3, 2, 3), (2, 3), I.CORE_B, 1),
    (I.SPHERICAL, (11, 6, 10), (6, 5), I.CORE_B, 7),
    (I.SPHERICAL, (9, 5, 7), (4, 4), I.TRANSPARENT, 0),   # hole: runs restart
    (I.CYLINDRICAL, (9, 8, 7), (6, 6), I.TRANSPARENT, 5),
    (I.CYLINDRICAL, (5, 3, 33), (2, 9), I.CORE_B, 0),
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


@pytest.mark.parametrize("coord,n,ang,bc,blk", CASES)
def test_march_against_oracle(coord, n, ang, bc, blk):
    p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.1, seed=31)
    g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, ng=False, angle_block=blk, I_outer=0.25)
    o = O.OracleGrid(coord, p["edges"], p["dirs"], p["weights"], bc, I_outer=0.25)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    S = p["B"].copy()
    for _ in range(3):  # the second and third steps run the streamed march
        J, L, _, _ = o.formal_solution(S, p["chi"], p["B"])
        S, _ = O.ali_update(S, J, L, p["eps"], p["B"])
        g.ali_step()
    # a few hundred roundings of 1.1e-16 along a line and in a voxel's sum
    assert np.max(np.abs(g.S() - S) / np.abs(S)) < 1e-13
    g.close()
    o.close()


@pytest.mark.parametrize("coord,n,ang,bc,blk", CASES)
def test_adjoint_streamed_against_general(coord, n, ang, bc, blk):
    p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.2, seed=32)
    rng = np.random.default_rng(5)
    nv = p["nvox"]
    gS, gJ, gF = rng.standard_normal(nv), rng.standard_normal(nv), rng.standard_normal((nv, 3))
    res = []
    for knobs in ({rt.RT_TUNE_STREAMED_WEIGHTS: 0}, {}, {rt.RT_TUNE_SCATTER: 0}):
        g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, angle_block=blk)
        for k, v in knobs.items():
            g.tune(k, v)
        g.set_opacity(p["chi"], p["eps"], p["B"])
        g.set_S(p["B"] * 0.5)
        res.append(g.adjoint(gS, gJ, gF.reshape(-1), tol=1e-14)[:3])
        g.close()
    for other in res[1:]:
        for a, b in zip(res[0], other):
            # the iterations stop within 1e-14 max|lam|, amplified by at most 1/eps = 5, plus the sums' rounding
            assert np.max(np.abs(a - b)) < 1e-11 * np.max(np.abs(a))
    for a, b in zip(res[1], res[2]):  # only the place of the values differs
        assert np.array_equal(a, b)
