"""The full FP64 formal solution on streamed weights and by the march that
evaluates them: the two agree to the rounding of FP64 sums, and a grid keeps to
one of them."""
import numpy as np
import pytest

from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt
from tests.helpers import tiny_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


def _grid(p, bc, knobs):
    g = rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=bc, ng=False, I_outer=0.25)
    for k, v in knobs.items():
        g.tune(k, v)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    return g


def _fs(g, p):
    g.set_S(0.5 * p["B"])
    g.formal_solution()
    return g.J(), g.Lstar(), g.flux()


@pytest.mark.parametrize("coord,n,ang,bc", [
    (I.SPHERICAL, (1, 1, 1), (2, 1), I.CORE_B), (I.SPHERICAL, (11, 6, 10), (6, 5), I.CORE_B),
    (I.SPHERICAL, (17, 9, 17), (8, 8), I.TRANSPARENT), (I.CYLINDRICAL, (9, 8, 7), (6, 6), I.TRANSPARENT),
    (I.CYLINDRICAL, (5, 3, 33), (2, 9), I.CORE_B)])
def test_streamed_against_evaluated(coord, n, ang, bc):
    p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.1, seed=51)
    res = []
    for knobs in ({}, {rt.RT_TUNE_STREAMED_WEIGHTS: 0}):
        g = _grid(p, bc, knobs)
        res.append(_fs(g, p))
        g.close()
    (J, L, F), (Je, Le, Fe) = res
    # a few hundred roundings of 1.1e-16 along a line and in a voxel's sum
    assert np.max(np.abs(J - Je) / np.abs(Je)) < 1e-13
    assert np.max(np.abs(L - Le)) < 1e-13 * np.max(np.abs(Le))
    assert np.max(np.abs(F - Fe)) < 1e-13 * 4 * np.pi * np.max(np.abs(Je))


def test_a_grid_keeps_its_way():
    """Too little free memory at the first formal solution: the later ones do not change over when the
    iteration has set the streams up."""
    torch = pytest.importorskip("torch")
    p = tiny_problem(I.SPHERICAL, (17, 9, 17), 6, 6, I.CORE_B, eps=0.1, seed=52)
    g = _grid(p, I.CORE_B, {})
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (3 << 30), dtype=torch.uint8, device="cuda")
    first = _fs(g, p)
    g.ali_step()
    g.ali_step()
    again = _fs(g, p)
    g.close()
    del hold
    torch.cuda.empty_cache()
    for a, b in zip(first, again):
        assert np.array_equal(a, b)
