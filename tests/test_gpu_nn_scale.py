"""The OS step of the nearest-neighbour Lambda* on source functions of any scale:
the system is linear, so a power of two in B goes through to S exactly, and the
solver takes the same steps as long as its scalars stay in range."""
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


def _steps(p, coord, bc, scale):
    g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, use_lstar=rt.RT_LSTAR_NN, ng=False)
    g.set_opacity(p["chi"], p["eps"], p["B"] * scale)
    for _ in range(3):
        g.ali_step()
    S, t = g.S() / scale, g.timing()
    g.close()
    return S, t["os_krylov_its"], t["os_sweeps"]


@pytest.mark.parametrize("coord,n,bc", [
    (I.SPHERICAL, (17, 9, 17), I.CORE_B),          # halos and rows in shared memory
    (I.CYLINDRICAL, (17, 16, 15), I.TRANSPARENT),
    (I.CYLINDRICAL, (33, 65, 65), I.TRANSPARENT),  # the seam is read past the halo
])
def test_small_sources(coord, n, bc):
    p = tiny_problem(coord, n, 2, 4, bc, eps=1e-2, seed=43)
    S0, _, _ = _steps(p, coord, bc, 1.0)
    # below FP32's range the corrections are solved in FP64, where these scales are exact
    S1, its1, sw1 = _steps(p, coord, bc, 2.0 ** -260)
    S2, its2, sw2 = _steps(p, coord, bc, 2.0 ** -400)
    assert (its1, sw1) == (its2, sw2) and np.array_equal(S1, S2)
    # three solves to 1e-14 max|x| each, amplified by at most 1/eps
    assert np.max(np.abs(S1 - S0)) < 3 * 2 * 1e-12 * np.max(np.abs(S0))
