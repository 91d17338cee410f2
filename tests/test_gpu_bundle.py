"""The mixed-precision J-only march in bundles of neighbouring characteristics:
bundles that hold one characteristic or a few, shares that end inside a tile,
voxels with more values than one unit takes, and several parts of the solid
angles, against the march that takes the characteristics in launch order."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt
from tests.helpers import tiny_problem

pytestmark = pytest.mark.gpu

CASES = [  # coord, n, angles, inner boundary, interpolation, angle_block, against the oracle too
    (I.SPHERICAL, (1, 1, 1), (1, 1), I.CORE_B, rt.RT_PARABOLIC, 0, True),       # a few characteristics in all
    (I.SPHERICAL, (2, 1, 3), (2, 3), I.CORE_B, rt.RT_LINEAR, 1, True),
    (I.SPHERICAL, (9, 5, 7), (4, 4), I.TRANSPARENT, rt.RT_PARABOLIC, 3, True),  # hole: runs restart
    (I.CYLINDRICAL, (4, 3, 65), (3, 7), I.CORE_B, rt.RT_PARABOLIC, 0, True),
    (I.CYLINDRICAL, (33, 9, 5), (12, 12), I.TRANSPARENT, rt.RT_PARABOLIC, 0, True),
    (I.SPHERICAL, (17, 9, 33), (24, 24), I.CORE_B, rt.RT_PARABOLIC, 0, False),  # full bundles, long lists
    (I.SPHERICAL, (33, 17, 33), (24, 24), I.CORE_B, rt.RT_PARABOLIC, 0, False),  # several parts
    (I.SPHERICAL, (129, 64, 65), (1, 2), I.CORE_B, rt.RT_PARABOLIC, 0, False),  # 64-bit keys of the tables' sort
]


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


@pytest.mark.parametrize("coord,n,ang,bc,interp,blk,orc", CASES)
def test_bundles(coord, n, ang, bc, interp, blk, orc):
    p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.1, seed=41)
    res = []
    for knobs in ({}, {rt.RT_TUNE_MARCH_COARSEN: 2}, {rt.RT_TUNE_OVERLAP: 0}, {rt.RT_TUNE_GRAPH: 0}):
        g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, interp=interp, precision=rt.RT_MIXED,
                    ng=False, angle_block=blk, I_outer=0.25)
        for k, v in knobs.items():
            g.tune(k, v)
        g.set_opacity(p["chi"], p["eps"], p["B"])
        for _ in range(4):
            g.ali_step()
        res.append(g.S())
        g.close()
    # the same FP32 weights and another order of the additions: as between the other march configurations
    assert np.max(np.abs(res[0] - res[1]) / np.abs(res[1])) < 2e-6
    assert np.array_equal(res[0], res[2]) and np.array_equal(res[0], res[3])
    if orc:
        o = O.OracleGrid(coord, p["edges"], p["dirs"], p["weights"], bc, I_outer=0.25, interp=interp)
        S = p["B"].copy()
        for _ in range(4):
            J, L, _, _ = o.formal_solution(S, p["chi"], p["B"])
            S, _ = O.ali_update(S, J, L, p["eps"], p["B"])
        o.close()
        assert np.max(np.abs(res[0] - S) / np.abs(S)) < 1e-5  # the mixed-precision bar


def test_reset_and_switch():
    """A new opacity refreshes the weights; a knob changed in between takes the other march and back."""
    p = tiny_problem(I.SPHERICAL, (11, 6, 10), 6, 6, I.CORE_B, eps=0.1, seed=42)

    def grid():
        return rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=I.CORE_B, precision=rt.RT_MIXED, ng=False)

    def steps(g, chi):
        g.set_opacity(chi, p["eps"], p["B"])
        for _ in range(4):
            g.ali_step()
        return g.S()

    g, h = grid(), grid()
    steps(g, p["chi"])
    g.tune(rt.RT_TUNE_MARCH_CHUNK, 256)
    steps(g, p["chi"])
    g.tune(rt.RT_TUNE_MARCH_CHUNK, 512)
    assert np.array_equal(steps(g, 3.0 * p["chi"]), steps(h, 3.0 * p["chi"]))
    g.close()
    h.close()
