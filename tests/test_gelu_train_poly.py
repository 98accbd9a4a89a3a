"""CPU pins of the training kernels' GELU and its derivative.

With a = |v|, e = exp(-a^2 / 2) and Q = Phi(-a) = e S(a), S the polynomial in u = a / 3 - 1 of
csrc/gelu_train_poly.cuh (written by csrc/gelu_train_fit.py):
  v Phi(v) = max(v, 0) - a Q,   sigma'(v) = 1 - r for v >= 0, r else, r = e (S - a / sqrt(2 pi)).
Here: the committed header is what the generator writes; the formulas, evaluated step by step in
FP32 on the host, are within 2^-24 (1 + |v|) + 2e-8 of the 64-bit values (the rounding of the
result, of the polynomial and of the exponent on values of at most 1, and the fit, twice over);
infinities and NaN come out as from the erf form."""
import importlib.util
import io
import math
import pathlib
import re
from contextlib import redirect_stdout

import numpy as np
import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2604_27158_gb300" / "csrc"
F = np.float32


def _coefficients():
    text = (CSRC / "gelu_train_poly.cuh").read_text()
    deg = int(re.search(r"#define GELU_T_DEG (\d+)", text).group(1))
    body = re.search(r"#define GELU_T_COEFFS \{([^}]*)\}", text).group(1)
    c = [F(x.strip().rstrip("f")) for x in body.split(",")]
    assert len(c) == deg + 1
    return c


def _fma(a, b, c):
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(F)


def gelu_and_derivative(v):
    """The kernels' formula on an FP32 array (their ex2.approx: relative error below 2^-22)."""
    c = _coefficients()
    v = np.asarray(v, F)
    with np.errstate(all="ignore"):
        a = np.fmax(-v, np.fmin(v, F(64)))  # fmaxf / fminf: the other value for a NaN
        u = _fma(np.fmin(a, F(6)), F(1 / 3), F(-1))
        p = np.full_like(v, c[-1])
        for k in range(len(c) - 2, -1, -1):
            p = _fma(p, u, c[k])
        t = (a * a).astype(F) * F(-0.72134752044448170)
        e = np.exp2(t.astype(np.float64)).astype(F)
        g = _fma(-a, (e * p).astype(F), np.maximum(v, F(0)))  # max.NaN
        r = (e * _fma(-np.abs(v), F(0.39894228040143268), p)).astype(F)
        d = np.where(v >= 0, (F(1) - r).astype(F), np.where(v < 0, r, v))
    return g, d


def test_header_is_what_the_generator_writes():
    pytest.importorskip("scipy")
    spec = importlib.util.spec_from_file_location("gelu_train_fit", CSRC / "gelu_train_fit.py")
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    buf = io.StringIO()
    with redirect_stdout(buf):
        mod.main()
    assert buf.getvalue() == (CSRC / "gelu_train_poly.cuh").read_text()


def test_value_and_derivative_against_64_bits():
    v = np.concatenate([np.linspace(-12, 12, 60001), np.geomspace(1e-30, 30, 4001), -np.geomspace(1e-30, 30, 4001),
                        np.random.default_rng(0).standard_normal(40000)]).astype(F)
    g, d = gelu_and_derivative(v)
    x = v.astype(np.float64)
    cdf = np.array([0.5 * math.erfc(-s / math.sqrt(2)) for s in x])
    pdf = np.exp(-0.5 * x * x) / math.sqrt(2 * math.pi)
    bound = 2.0 ** -24 * (1 + np.abs(x)) + 2e-8
    assert np.all(np.abs(g - x * cdf) <= bound)
    assert np.all(np.abs(d - (cdf + x * pdf)) <= 2.0 ** -23 + 2e-8 + 2.0 ** -24 * np.abs(x) * pdf)


def test_infinities_and_nan_as_in_the_erf_form():
    g, d = gelu_and_derivative([np.inf, -np.inf, np.nan, 1e30, -1e30, 3e38, -3e38, 64.0, 65.0, -65.0, 0.0])
    assert g[0] == np.inf and np.isnan(g[1]) and np.isnan(g[2]) and np.isnan(d[:3]).all()
    assert list(g[3:]) == [F(1e30), 0, F(3e38), 0, 64, 65, 0, 0]
    assert list(d[3:]) == [1, 0, 1, 0, 1, 1, 0, 0.5]
