"""Which grids take the bundled mixed march, and both of its forms against each
other: bundles asked for on small grids, the folded march in launch order in all
its settings, and a grid whose characteristics are too long for a bundle."""
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_0903_1949_gb300 import build as Bd
from paper_0903_1949_gb300 import inputs as I
from paper_0903_1949_gb300 import rt
from tests.helpers import tiny_problem
from tests.test_gpu_bundle import CASES

pytestmark = pytest.mark.gpu

LAUNCH, FORCE = {rt.RT_TUNE_BUNDLES: 0}, {rt.RT_TUNE_BUNDLES: 2}


@pytest.fixture(scope="module", autouse=True)
def _built():
    Bd.build()
    rt.load()


def _run(p, bc, knobs, interp=rt.RT_PARABOLIC, blk=0, steps=4, timing=False):
    """S after some mixed iterations, and bytes a segment of the marches (with timing)."""
    g = rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=bc, interp=interp, precision=rt.RT_MIXED,
                ng=False, angle_block=blk, I_outer=0.25)
    for k, v in knobs.items():
        g.tune(k, v)
    g.set_opacity(p["chi"], p["eps"], p["B"])
    g.ali_step()
    if timing:
        g.set_timing(True)
    for _ in range(steps - 1):
        g.ali_step()
    t = g.timing()
    S = g.S()
    g.close()
    return (S, t["march_bytes"] / max(1, t["march_segments"])) if timing else S


def _err(a, b):
    return float(np.max(np.abs(a - b) / np.abs(b)))


@pytest.mark.parametrize("coord,n,ang,bc,interp,blk,orc", CASES)
def test_forced_bundles(coord, n, ang, bc, interp, blk, orc):
    p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.1, seed=41)
    S, per = _run(p, bc, FORCE, interp, blk, timing=True)
    L, per_l = _run(p, bc, LAUNCH, interp, blk, timing=True)
    assert per_l == 24 and (per != 24 or p["nvox"] < 50)  # the forms stream different bytes: both ran
    assert _err(S, L) < 2e-6  # the same FP32 weights, another order of the additions
    for more in ({rt.RT_TUNE_OVERLAP: 0}, {rt.RT_TUNE_GRAPH: 0}):
        assert np.array_equal(_run(p, bc, {**FORCE, **more}, interp, blk), S)
    if orc:
        o = O.OracleGrid(coord, p["edges"], p["dirs"], p["weights"], bc, I_outer=0.25, interp=interp)
        S_o = p["B"].copy()
        for _ in range(4):
            J, La, _, _ = o.formal_solution(S_o, p["chi"], p["B"])
            S_o, _ = O.ali_update(S_o, J, La, p["eps"], p["B"])
        o.close()
        assert _err(S, S_o) < 1e-5 and _err(L, S_o) < 1e-5  # the mixed-precision bar


@pytest.mark.parametrize("coord,n,bc,interp", [
    (I.SPHERICAL, (17, 9, 17), I.CORE_B, rt.RT_PARABOLIC),
    (I.CYLINDRICAL, (9, 8, 7), I.TRANSPARENT, rt.RT_PARABOLIC),
    (I.SPHERICAL, (11, 6, 10), I.CORE_B, rt.RT_LINEAR)])
def test_launch_order_settings(coord, n, bc, interp):
    """The folded march in launch order: the same arithmetic in the same order gives the same bits."""
    p = tiny_problem(coord, n, 6, 6, bc, eps=0.1, seed=45)
    S = _run(p, bc, LAUNCH, interp)
    for var in ({rt.RT_TUNE_SCATTER: 0}, {rt.RT_TUNE_OVERLAP: 0}, {rt.RT_TUNE_S_BLOCKED: 0}, {rt.RT_TUNE_GRAPH: 0},
                {rt.RT_TUNE_MARCH_STREAMS: 1}, {rt.RT_TUNE_MARCH_LOOKAHEAD: 0},
                {rt.RT_TUNE_SCATTER: 0, rt.RT_TUNE_S_BLOCKED: 0, rt.RT_TUNE_OVERLAP: 0}):
        assert np.array_equal(_run(p, bc, {**LAUNCH, **var}, interp), S), var
    assert np.array_equal(_run(p, bc, {**LAUNCH, rt.RT_TUNE_MARCH_CHUNK: 512}, interp), S)
    for chunk in (64, 4096):
        assert _err(_run(p, bc, {**LAUNCH, rt.RT_TUNE_MARCH_CHUNK: chunk}, interp), S) < 2e-6


def test_long_characteristics_keep_launch_order():
    """More than 4096 segments of a characteristic: no bundle holds a few of them."""
    p = tiny_problem(I.CYLINDRICAL, (1, 1, 4500), 2, 3, I.TRANSPARENT, eps=0.1, seed=46, R_min=0.5, R_max=500.0, z_max=2.0)
    S, per = _run(p, I.TRANSPARENT, FORCE, timing=True)
    L, _ = _run(p, I.TRANSPARENT, LAUNCH, timing=True)
    assert per == 24
    assert _err(S, L) < 2e-6


def test_small_and_cylindrical_grids_skip_the_tables():
    """Their first streamed iteration costs what the march in launch order needs (its own set-up, not 4 times)."""
    for coord, n, ang, bc in ((I.SPHERICAL, (17, 9, 17), (8, 8), I.CORE_B), (I.CYLINDRICAL, (33, 33, 33), (8, 8), I.TRANSPARENT)):
        p = tiny_problem(coord, n, ang[0], ang[1], bc, eps=0.1, seed=47)
        ms = {}
        for name, knobs in (("default", {}), ("launch", LAUNCH)):
            t = []
            for _ in range(5):
                g = rt.Grid(coord, p["edges"], p["dirs"], p["weights"], inner_bc=bc, precision=rt.RT_MIXED, ng=False)
                for k, v in knobs.items():
                    g.tune(k, v)
                g.set_opacity(p["chi"], p["eps"], p["B"])
                g.ali_step()
                t0 = time.perf_counter()
                g.ali_step()  # the first that streams weights; returns with its result
                t.append(time.perf_counter() - t0)
                g.close()
            ms[name] = 1e3 * min(t)
        assert ms["default"] < 2.0 * ms["launch"], (coord, ms)


def test_large_spherical_grid_takes_bundles():
    p = I.make_problem("sph65", n_mu=8, n_phi=8)
    _, per = _run(p, I.CORE_B, {}, timing=True)
    assert per != 24
    _, per = _run(p, I.CORE_B, LAUNCH, timing=True)
    assert per == 24


def test_unit_sums_keep_their_compensation():
    """One solid angle: most voxels' values make one unit, and a sum of four FP32 values or more is rarely an
    FP32 number itself (as in launch order, where the compensated sum is taken over the whole list)."""
    p = tiny_problem(I.SPHERICAL, (17, 9, 17), 1, 1, I.CORE_B, eps=0.1, seed=48)
    for knobs in (LAUNCH, FORCE):
        with rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=I.CORE_B, precision=rt.RT_MIXED, ng=False,
                     I_outer=0.25) as g:
            for k, v in knobs.items():
                g.tune(k, v)
            g.set_opacity(p["chi"], p["eps"], p["B"])
            g.ali_step()
            g.ali_step()
            J = g.J()
            many = np.bincount(g.crossings(0)["vox"], minlength=p["nvox"]) >= 4
        assert many.sum() > 100 and np.mean((J == J.astype(np.float32))[many]) < 0.5, knobs


def test_error_against_fp64():
    """Few solid angles: bundles are no further from FP64 than launch order (1 % for the other order of the scan)."""
    p = I.make_problem("sph65", n=(65, 33, 65), n_mu=2, n_phi=4, tau=1e3, noise=0.2)
    rng = np.random.default_rng(9)
    S = p["B"] * np.exp(0.5 * rng.standard_normal(p["B"].size))
    J = {}
    for name, prec, knobs in (("fp64", rt.RT_FP64, {}), ("launch", rt.RT_MIXED, LAUNCH), ("bundles", rt.RT_MIXED, FORCE)):
        with rt.Grid(p["coord"], p["edges"], p["dirs"], p["weights"], inner_bc=I.CORE_B, precision=prec, ng=False) as g:
            for k, v in knobs.items():
                g.tune(k, v)
            g.set_opacity(p["chi"], p["eps"], p["B"])
            g.ali_step()
            g.set_S(S)
            g.ali_step()
            J[name] = g.J()
    rms = {k: float(np.sqrt(np.mean((J[k] / J["fp64"] - 1.0) ** 2))) for k in ("launch", "bundles")}
    assert rms["bundles"] < 1.01 * rms["launch"], rms
