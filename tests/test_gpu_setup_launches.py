"""Kernels launched for set-up: only what the march in use reads, and all of them counted."""
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


def _grid(precision, blk=3):
    p = tiny_problem(I.SPHERICAL, (11, 6, 10), 6, 5, I.CORE_B, eps=0.1, seed=53)
    g = rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=I.CORE_B, precision=precision, ng=False,
                angle_block=blk)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    return g


def _launches(g):
    n0 = g.timing()["kernel_launches"]
    g.ali_step()
    return g.timing()["kernel_launches"] - n0


def test_fp64_march_has_no_bundle_bounds():
    """The bounds of the march in launch order belong to the FP32 march: a new bundle size costs the FP64
    iteration nothing."""
    g = _grid(rt.RT_FP64)
    g.ali_step()
    g.ali_step()
    n = _launches(g)
    g.tune(rt.RT_TUNE_MARCH_CHUNK, 256)
    assert _launches(g) == n
    g.close()
    g = _grid(rt.RT_MIXED)
    g.ali_step()
    g.ali_step()
    n = _launches(g)
    g.tune(rt.RT_TUNE_MARCH_CHUNK, 256)
    assert _launches(g) == n + g.info()["n_blocks"]
    g.close()
