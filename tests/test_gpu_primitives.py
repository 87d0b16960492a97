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
