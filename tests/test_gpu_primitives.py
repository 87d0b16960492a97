"""The exponentials and reciprocal root of the pair arithmetics against extended precision (numpy's long double).

Bounds.  Float-float e^{-x}: rms of the relative error as the terms need it, 4.0e-15 for x < 0.04 (where 1 - E is
x itself) and 6.3e-15 below 8; low parts left unnormalised in its last factor give 4.2e-15 and 7.6e-15 there,
normalised ones 3.85e-15 and 5.24e-15 (the same operations in host arithmetic)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def evaluate():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import native_lib
    L = native_lib.load("primitives.cu")

    def f(which, x, kappa=1.0):
        x = np.ascontiguousarray(x, dtype=np.float64)
        out = np.empty_like(x)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert L.eval_primitive(which, ctypes.c_int64(x.size), p(x), ctypes.c_double(kappa), p(out)) == 0
        return out
    return f


def _rms(e):
    return float(np.sqrt(np.mean(np.square(e.astype(np.float64)))))


@pytest.mark.parametrize("hi,bound", [(0.04, 4.0e-15), (8.0, 6.3e-15)])
def test_float_float_exponential(evaluate, hi, bound):
    rng = np.random.Generator(np.random.PCG64(3))
    x = rng.uniform(0.0, hi, 400000)
    h = x.astype(np.float32)
    x = h.astype(np.float64) + (x - h.astype(np.float64)).astype(np.float32).astype(np.float64)   # as split
    ref = np.exp(-x.astype(np.longdouble))
    err = (evaluate(0, x).astype(np.longdouble) - ref) / ref
    assert _rms(err) < bound


U = 2.0 ** -53


def _log_uniform(lo, hi, n, seed):
    t = np.random.Generator(np.random.PCG64(seed)).random(n)
    return np.exp(np.log(lo) + (np.log(hi) - np.log(lo)) * t)


def test_fp64_reciprocal_root(evaluate):
    """Relative error at most 1.2 U: the last operation rounds by at most U, the series' next term is (5/16) e^3
    with |e| < 2^-18 (twice the seed's error of 2^-19 at most), the rest is below 2^-60.  rms below 0.5 U."""
    x = np.concatenate([_log_uniform(1e-6, 1e6, 200000, 1), _log_uniform(1e-297, 1e297, 100000, 2), 4.0 ** np.arange(-490, 490)])
    y = evaluate(2, x).astype(np.longdouble)
    ref = 1 / np.sqrt(x.astype(np.longdouble))
    err = ((y - ref) / ref).astype(np.float64)
    assert np.max(np.abs(err)) < 1.2 * U
    assert _rms(err[:200000]) < 0.5 * U


@pytest.mark.parametrize("kappa", [0.1257, 1.0, 30.0, 1e-3, 0.0])
def test_fp64_exponential(evaluate, kappa):
    """e^{-kappa r}: the result's rounding and the index's.  The index comes from r in 24 bits (truncated) and two
    roundings, so with y = kappa r log2(e) the remainder is off by up to d = y 2^-22 and reaches 2^-11 + d; only its
    third-order term is formed from the inexact remainder, which leaves ln(2)^4/24 (2^-11 + d)^3 d.  Below 2^-1000:
    0 (checked from 2^-1010 on)."""
    r = np.concatenate([_log_uniform(1e-3, 1e3, 300000, 3), _log_uniform(1e-30, 1e-3, 1000, 4), [0.0]])
    if kappa > 0:
        r = np.concatenate([r, np.arange(4096) / 1024.0 * np.log(2.0) / kappa, _log_uniform(600.0, 692.0, 20000, 5) / kappa])
    got = evaluate(1, r, kappa)
    kr = np.longdouble(kappa) * r.astype(np.longdouble)
    y = (kr / np.log(np.longdouble(2))).astype(np.float64)
    ok = y < 999.9
    ref = np.exp(-kr[ok])
    err = np.abs(((got[ok].astype(np.longdouble) - ref) / ref).astype(np.float64))
    d = y[ok] * 2.0 ** -22
    bound = 1.2 * U + 0.00962 * (2.0 ** -11 + d) ** 3 * d
    assert np.all(err < bound), np.max(err / bound)
    near = y[ok] < 43.0   # kappa r < 30
    assert _rms(err[near]) < 0.5 * U
    assert np.all(got[y > 1010.0] == 0.0)
    assert np.all(got[kr == 0] == 1.0)
