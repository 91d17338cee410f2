"""The OS step of the nearest-neighbour Lambda* at the sizes where its solver
changes form: fewer voxels than blocks, a block's rows of one and of several
warps, halos with and without the cylindrical grid's phi seam."""
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


def _apply(coord, n, L, x):
    """sum_q L[v, q] x[neighbour q of v] over the 27 slots, phi periodic."""
    X = x.reshape(n)
    phi = 2 if coord == I.SPHERICAL else 1
    out = np.zeros(n)
    for q in range(27):
        Y = X
        for ax, d in enumerate((q // 9 - 1, (q // 3) % 3 - 1, q % 3 - 1)):
            Z = np.roll(Y, -d, axis=ax)
            if ax != phi and d:
                edge = [slice(None)] * 3
                edge[ax] = -1 if d > 0 else 0
                Z = Z.copy()
                Z[tuple(edge)] = 0.0
            Y = Z
        out += L[:, q].reshape(n) * Y
    return out.reshape(-1)


@pytest.mark.parametrize("coord,n,bc", [
    (I.SPHERICAL, (3, 4, 5), I.CORE_B),
    (I.SPHERICAL, (21, 18, 23), I.CORE_B),
    (I.SPHERICAL, (65, 33, 40), I.CORE_B),
    (I.CYLINDRICAL, (9, 8, 7), I.TRANSPARENT),
    (I.CYLINDRICAL, (20, 31, 21), I.TRANSPARENT),
    (I.CYLINDRICAL, (33, 65, 65), I.TRANSPARENT),  # the seam is read past the halo
])
def test_os_step_solves_its_system(coord, n, bc):
    p = tiny_problem(coord, n, 2, 4, bc, eps=0.05, seed=41)
    g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, use_lstar=rt.RT_LSTAR_NN, ng=False)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    L = g.Lstar_nn()
    g.ali_step()
    x, J = g.S() - p["B"], g.J()
    y = (1.0 - p["eps"]) * J + p["eps"] * p["B"] - p["B"]
    r = y - (x - (1.0 - p["eps"]) * _apply(coord, n, L, x))
    g.close()
    # a Jacobi sweep changes x by at most 1e-14 max|x|; 27 products and S's own rounding (S = B + x) on top
    assert np.max(np.abs(r)) < 1e-13 * np.max(np.abs(x)) + 1e-14 * np.max(np.abs(p["B"]))
