"""The OS step of the nearest-neighbour line operator: it solves its system, and
it runs on the shared-memory form of the solver as the continuum's does."""
import time

import numpy as np
import pytest

from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt
from tests.helpers import tiny_problem
from tests.test_gpu_nn_os import _apply

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


@pytest.mark.parametrize("coord,n,bc", [
    (I.SPHERICAL, (3, 4, 5), I.CORE_B),
    (I.SPHERICAL, (21, 18, 23), I.CORE_B),
    (I.CYLINDRICAL, (20, 31, 21), I.TRANSPARENT),
    (I.CYLINDRICAL, (33, 65, 65), I.TRANSPARENT),  # the seam is read past the halo
])
def test_line_os_step_solves_its_system(coord, n, bc):
    p = tiny_problem(coord, n, 2, 4, bc, eps=0.05, seed=44)
    g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, precision=rt.RT_MIXED)
    phi, wq = I.line_profile(3)
    ln = rt.Line(g, phi, wq, use_lstar=rt.RT_LSTAR_NN)
    ln.set(1e-2 * p["chi"], p["chi"], p["eps"], p["B"])
    ln.step()
    x, J = ln.S_l() - p["B"], ln.Jbar()  # S_l begins as B
    y = (1.0 - p["eps"]) * J + p["eps"] * p["B"] - p["B"]
    r = y - (x - (1.0 - p["eps"]) * _apply(coord, n, ln.Lbar_nn(), x))
    ln.close()
    g.close()
    # a Jacobi sweep changes x by at most 1e-14 max|x|; 27 products and S's own rounding (S = B + x) on top
    assert np.max(np.abs(r)) < 1e-13 * np.max(np.abs(x)) + 1e-14 * np.max(np.abs(p["B"]))


def test_line_os_step_costs_a_continuum_one():
    """One frequency, phi = 1 and no continuum: the line's system is the continuum's.  Its solve takes three
    grid barriers an iteration against two, in the same form (five in the global-memory form, 1.9 times)."""
    n = (33, 17, 33)
    p = I.make_problem("sph65", n=n, n_mu=8, n_phi=8, tau=100.0, eps=1e-4, noise=0.2)
    g = rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=p["inner_bc"], precision=rt.RT_MIXED)
    step = {}
    for lstar in (rt.RT_LSTAR_DIAG, rt.RT_LSTAR_NN):
        ln = rt.Line(g, np.ones(1), np.ones(1), use_lstar=lstar)
        ln.set(np.zeros(p["chi"].size), p["chi"], p["eps"], p["B"])
        ln.step()
        t = []
        for _ in range(12):  # a step returns with its result
            t0 = time.perf_counter()
            ln.step()
            t.append(1e3 * (time.perf_counter() - t0))
        step[lstar] = float(np.median(t))
        ln.close()
    g.close()
    g = rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=p["inner_bc"], precision=rt.RT_MIXED,
                use_lstar=rt.RT_LSTAR_NN, ng=False)
    g.tune(rt.RT_TUNE_NN_JTOL, 14)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    g.ali_step()
    g.set_timing(True)
    for _ in range(12):
        g.ali_step()
    t = g.timing()
    g.close()
    line, cont = step[rt.RT_LSTAR_NN] - step[rt.RT_LSTAR_DIAG], t["os_ms"] / t["os_solves"]
    print("OS step: line %.3f ms, continuum %.3f ms" % (line, cont))
    assert line < 1.6 * cont, (line, cont)
