"""The FP64 interpolation weights (Coef64), their derivatives (Coef64D) and the
reciprocal they use (rcp64) against decimal arithmetic of many digits: from
optical depths far below rounding to far above 1, dense around the change of
form at x = 1, with the next segment's depth from x / 2 to much larger ones."""
import ctypes
import os
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

from paper_0903_1949_gb300 import build as Bd

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53  # half an ulp of a number in [1, 2), relative
NAMES = ("E", "alpha", "beta", "gamma", "E_x", "alpha_x", "beta_x", "gamma_x", "alpha_p", "beta_p", "gamma_p")


@pytest.fixture(scope="module")
def ev(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("coef") / "coef.so")
    subprocess.run([Bd.nvcc(), *Bd.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", Bd.CSRC,
                    os.path.join(ROOT, "tests", "coef_eval.cu"), "-o", so], check=True)
    f = ctypes.CDLL(so).coef_eval

    def call(form, x, p=None, para=None):
        x = np.ascontiguousarray(x, np.float64)
        p = np.zeros_like(x) if p is None else np.ascontiguousarray(p, np.float64)
        para = np.zeros(x.size, np.int32) if para is None else np.ascontiguousarray(para, np.int32)
        out = np.empty((x.size, 11))
        assert f(form, x.size, *(a.ctypes.data_as(ctypes.c_void_p) for a in (x, p, para, out))) == 0
        return out

    return call


def _functions(x):
    """e0, f1, f2, g1, g2 of a decimal x: f1 = (x - e0) / x, f2 = 2 f1 - e0, g1 = f1', g2 = f2', by their series below 1/8."""
    if x < Decimal("0.125"):
        f1 = f2 = g1 = g2 = Decimal(0)
        t = Decimal(1)  # x^(n - 2) / n! with alternating sign, n >= 2
        for n in range(2, 40):
            t = (Decimal(1) / 2) if n == 2 else -t * x / n
            f1 += t
            g1 += t * (n - 1)
            if n > 2:  # the coefficient of f2: 2 / (n + 1)! - 1 / n! shifted, sign of n
                f2 += -t * (n - 2)
                g2 += -t * (n - 2) * (n - 1)
        f1, f2, g2 = f1 * x, f2 * x, g2
        e0 = x - x * f1
        return e0, f1, f2, g1, g2
    e0 = 1 - (-x).exp()
    f1 = (x - e0) / x
    f2 = 2 * f1 - e0
    return e0, f1, f2, (e0 - f1) / x, e0 - f1 - f2 / x


def _exact(x, p, para):
    """The 11 values, and the size of the terms each is a sum of (what its rounding is relative to)."""
    x, p = Decimal(float(x)), Decimal(float(p))
    e0, f1, f2, g1, g2 = _functions(x)
    E = 1 - e0 if x < Decimal("0.125") else (-x).exp()
    if not para:
        v = [E, e0 - f1, f1, Decimal(0), -E, E - g1, g1] + [Decimal(0)] * 4
        s = [E, e0 + f1, f1, Decimal(1), E, E + g1, g1] + [Decimal(1)] * 4
        return v, s
    D = x + p
    v = [E, e0 - f1 - f2 / D, f1 + f2 / p, -x * f2 / (p * D), -E, E - g1 - g2 / D + f2 / D / D, g1 + g2 / p,
         -(f2 * p + x * g2 * D) / (p * D * D), f2 / D / D, -f2 / p / p, x * f2 * (x + 2 * p) / (p * p * D * D)]
    s = [E, e0 + f1 + f2 / D, f1 + f2 / p, x * f2 / (p * D), E, E + g1 + abs(g2) / D + f2 / D / D, g1 + abs(g2) / p,
         (f2 * p + x * abs(g2) * D) / (p * D * D), f2 / D / D, f2 / p / p, x * f2 * (x + 2 * p) / (p * p * D * D)]
    return v, s


def _points(lo, hi, n, seed):
    rng = np.random.default_rng(seed)
    x = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    p = x * np.exp(rng.uniform(np.log(0.5), np.log(1e3), n))
    p[: n // 8] = x[: n // 8] * np.exp(rng.uniform(0, np.log(1e30), n // 8))  # p >> x
    return x, p, (rng.random(n) < 0.7).astype(np.int32)


def _errors(out, x, p, para, k):
    """Errors in units of U times the size of the terms, (points, k)."""
    getcontext().prec = 60
    err = np.zeros((x.size, k))
    for i in range(x.size):
        v, s = _exact(x[i], p[i], para[i])
        for q in range(k):
            err[i, q] = float(abs(Decimal(float(out[i, q])) - v[q]) / max(s[q], Decimal("1e-290"))) / U
    return err


RANGES = [(1e-70, 1e-20), (1e-20, 1e-6), (1e-6, 0.5), (0.5, 1.0), (0.99, 1.01), (1.0, 4.0), (4.0, 700.0), (700.0, 1e8)]
# mean and largest error (in units of U, relative to the size of the terms) that a handful of roundings,
# each at most 1, give: E one exponential or two operations; alpha and beta three to five; gamma six.  f2 is the
# difference of terms 6 to 12 times its size just above x = 1.
MEAN, MOST = {"E": 0.55, "alpha": 0.65, "beta": 1.0, "gamma": 1.0}, {"E": 2.5, "alpha": 5.0, "beta": 13.0, "gamma": 8.0}


@pytest.mark.parametrize("lo,hi", RANGES)
def test_weights(ev, lo, hi):
    x, p, para = _points(lo, hi, 3000, 5)
    err = _errors(ev(0, x, p, para), x, p, para, 4)
    ser = _errors(ev(1, x, p, para), x, p, para, 4)
    wide = 4.0 if hi > 1.0 and lo < 4.0 else 1.0
    for q, name in enumerate(NAMES[:4]):
        m, top = float(err[:, q].mean()), float(err[:, q].max())
        f = wide if name == "gamma" else 1.0
        assert m < f * MEAN[name] and top < f * MOST[name], (name, m, top)
        # no worse than the series, expm1 and one division for each quotient
        assert name == "E" or m < 1.1 * float(ser[:, q].mean()) + 0.02, (name, m, float(ser[:, q].mean()))


@pytest.mark.parametrize("lo,hi", RANGES[:4])
def test_derivatives(ev, lo, hi):
    x, p, para = _points(lo, hi, 3000, 6)
    err = _errors(ev(2, x, p, para), x, p, para, 11).mean(axis=0)
    # series for g1 and g2: two to four roundings in what follows x, six to eight in the quotients
    for q, most in enumerate((0.55, 0.65, 1.0, 1.0, 0.55, 0.4, 0.7, 1.3, 1.3, 1.1, 1.6)):
        assert err[q] < most, (NAMES[q], err[q])


def test_reciprocal_and_quotient(ev):
    rng = np.random.default_rng(7)
    q = np.concatenate([np.exp2(rng.uniform(-1021, 1022, 40000)), np.exp2(rng.uniform(-902, -898, 4000)),
                        np.exp2(rng.uniform(898, 902, 4000)), rng.uniform(1.0, 2.0, 200000), 2.0 ** np.arange(-1021, 1022),
                        [np.inf, 5e-324, 2.0 ** -1022, 1.7976931348623157e308]])
    a = rng.uniform(0.5, 2.0, q.size)
    o = ev(3, q, a)
    for k in (0, 2):
        fin = np.isfinite(o[:, k + 1]) & (np.abs(o[:, k + 1]) > 2.0 ** -1000)
        ulps = np.abs(o[fin, k] - o[fin, k + 1]) / np.spacing(np.abs(o[fin, k + 1]))
        assert ulps.max() <= 1.0, (k, ulps.max())  # the estimate's error of 2^-20 cubed, and two roundings
        assert np.array_equal(o[~fin, k], o[~fin, k + 1], equal_nan=True)  # the division itself
        if k == 2:
            assert np.mean(ulps > 0) < 1e-3  # the residual settles all but near ties
