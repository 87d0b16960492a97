"""Every point of long potential maps, and the two FP32 routes.

Points repeat with a period, so a skipped or misplaced range of points shows against the first period: float-float
and FP64 values are the same bits, FP32 ones within the maps' 2e-6 of scale (the number of splits may differ)."""
import numpy as np
import pytest

import synthetic as syn
from oracle import energy as oenergy
from oracle.system import OracleSystem

pytestmark = pytest.mark.gpu

PERIOD = 5001


@pytest.fixture(scope="module")
def ctr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    return ctr


def _points(n, seed):
    """n points 9 to 12 from the origin: outside both surfaces' tubes."""
    rng = np.random.Generator(np.random.PCG64(seed))
    u = rng.normal(size=(n, 3))
    return rng.uniform(9.0, 12.0, size=(n, 1)) * u / np.linalg.norm(u, axis=1, keepdims=True)


@pytest.mark.parametrize("which", ["sphere", "ellipsoid"])
def test_every_point_of_long_maps(ctr, oracle_tables, which):
    prob = syn.sphere_problem(h=0.25) if which == "sphere" else syn.ellipsoid_problem(h=0.2)
    S = OracleSystem.from_problem(prob, tables=oracle_tables)
    noise = syn.random_density(S.M, seed=1)
    psi, dpsi = 1.0 + 0.1 * noise[:S.M], 1.0 + 0.1 * noise[S.M:]
    base = _points(PERIOD, 9)
    # the FP64 maps of 11,203 nodes go in launches of 23,808 points
    edge = np.array([23806, 23807, 23808, 23809, 47615, 47616]) % PERIOD
    ref = oenergy.reaction_potential(S, psi, dpsi, base[edge])
    scale = np.max(np.abs(ref))
    for n in (PERIOD + 1, 50003):
        z = np.tile(base, (11, 1))[:n]
        with ctr.CtrIbim.from_problem(prob) as G:
            for prec, tol in ((ctr.FP32_REFINE, 2e-6), (ctr.DF64, 1e-12), (ctr.FP64, 1e-12)):
                got = G.potential_map(psi, dpsi, z, prec)
                again = got[np.arange(n) % PERIOD]
                if prec == ctr.FP32_REFINE:
                    assert np.max(np.abs(got - again)) / scale < tol
                else:
                    assert np.array_equal(got, again)
                assert np.max(np.abs(got[edge] - ref)) / scale < tol


def test_fp32_routes_give_the_same_bits(ctr):
    """11,203 nodes in ten splits either way: 11,000 points (484,000 unit sums) take the units, 13,000 the tiled
    kernel; a point's value has the same bits."""
    prob = syn.ellipsoid_problem(h=0.2)
    z = _points(13000, 4)
    with ctr.CtrIbim.from_problem(prob) as G:
        noise = syn.random_density(G.M, seed=2)
        psi, dpsi = noise[:G.M], noise[G.M:]
        tiled = G.potential_map(psi, dpsi, z, ctr.FP32_REFINE)
        units = G.potential_map(psi, dpsi, z[:11000], ctr.FP32_REFINE)
    assert np.array_equal(units, tiled[:11000])
