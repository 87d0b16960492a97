"""Single terms of the potential maps: a density of one node, so that a map's value is one pair's term.

Bound (float-float dipole term, relative to its uncancelled size a (1 + (eps_E/eps_I) E1) / r^2, rms over points 8
to 100 from the node, where (eps_E/eps_I) E1 passes through 1): 1.6e-14, the error of float-float arithmetic
normalised throughout; host arithmetic of the kernel's operations gives 1.0e-14."""
import math

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    return ctr


def _split(v):
    """The value a float-float pair holds."""
    h = np.asarray(v, dtype=np.float64).astype(np.float32).astype(np.float64)
    return h + (np.asarray(v) - h).astype(np.float32).astype(np.float64)


def test_float_float_dipole_term(ctr):
    prob = syn.ellipsoid_problem(h=0.2, kappa=0.1257)
    c1 = prob.eps_out / prob.eps_in
    rng = np.random.Generator(np.random.PCG64(7))
    errs = []
    with ctr.CtrIbim.from_problem(prob) as G:
        P, n, W = G.geometry()
        for j in rng.integers(0, G.M, size=16):
            u = rng.normal(size=(20000, 3))
            r = 8.0 * (100.0 / 8.0) ** rng.random((20000, 1))
            z = P[j] + r * u / np.linalg.norm(u, axis=1, keepdims=True)
            psi = np.zeros(G.M)
            psi[j] = 1.0
            got = G.potential_map(psi, np.zeros(G.M), z, ctr.DF64)
            a = _split(prob.grid.h ** 3 * W[j] / (4.0 * math.pi)).astype(np.longdouble)
            d = _split(z).astype(np.longdouble) - _split(P[j])
            r2 = np.sum(d * d, axis=1)
            kr = _split(prob.kappa).astype(np.longdouble) * np.sqrt(r2)
            E1 = np.exp(-kr) * (1 + kr)
            ref = a * (d @ _split(n[j]).astype(np.longdouble)) / (r2 * np.sqrt(r2)) * (c1 * E1 - 1)
            errs.append(((got - ref) * r2 / (a * (1 + c1 * E1))).astype(np.float64))
    assert math.sqrt(np.mean(np.square(np.concatenate(errs)))) < 1.6e-14
