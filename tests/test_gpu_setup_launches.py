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


def _scan(n):
    return 3 if n > 0 else 1


def _radix(n, bits):
    return 1 + -(-bits // 8) * (2 + 3) if n > 0 else 0


def test_set_up_launches_are_counted():
    """First streamed FP64 step: the set-up of its slots (sort keys; per block the counts, the offsets, the radix
    passes of as many bits as a length has, the order and the groups; the scan of the groups), positions, fill and
    weights per block, then march and gather of every block and the update."""
    g = _grid(rt.RT_FP64, blk=7)
    g.tune(rt.RT_TUNE_STREAMED_WEIGHTS, 0)
    g.ali_step()  # the full solution without streams
    g.tune(rt.RT_TUNE_STREAMED_WEIGHTS, 1)
    g.tune(rt.RT_TUNE_GRAPH, 0)
    nblk = g.info()["n_blocks"]
    first = _launches(g)
    steady = _launches(g)
    cap = 2 * (4 * (11 + 6 + 10) + 16) + 8
    set_up = 1 + _scan(1) + nblk * (2 + _scan(cap + 1) + _radix(1, (cap).bit_length()) + 2)
    assert first - steady == set_up + 3 * nblk  # positions, fill, weights
    assert steady == 2 * nblk + 1  # march and gather per block, and the update
    g.close()
