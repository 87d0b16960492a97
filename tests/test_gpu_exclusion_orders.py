"""Long and one-way exclusion lists in tree order, and systems within one target block.

Tolerances as for the operators elsewhere: FP64 1e-12, float-float 1e-12 (direct) and 1e-11 (treecode), FP32 2e-5."""
import numpy as np
import pytest

import synthetic as syn
from oracle import treecode as tc
from oracle.system import OracleSystem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    return ctr


def _rel(a, b):
    return float(np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("name", ["kreg_ellipsoid", "molecule"])
def test_treecode_with_kreg_rows(ctr, oracle_tables, name):
    """Mutual near blocks over tree positions with K-reg cylinders (alone, and beside plane rows)."""
    kreg = name == "kreg_ellipsoid"
    prob = syn.ellipsoid_problem(h=0.2) if kreg else syn.molecule_problem(n_atoms=60, seed=11, h=0.5)
    S = OracleSystem.from_problem(prob, tables=oracle_tables, method="kreg" if kreg else "hyb")
    sets = [set(S.excl_idx[S.excl_ptr[i]:S.excl_ptr[i + 1]].tolist()) for i in range(S.M)]
    assert sum(i not in sets[j] for i in range(S.M) for j in sets[i]) > 0   # one-way pairs exist
    tree = dict(degree=3, theta=0.61, leaf=16)
    opts = ctr.Options(tube_halfwidth=prob.tube, method=ctr.METHOD_KREG if kreg else ctr.METHOD_HYB,
                       farfield=ctr.FARFIELD_TREECODE, tree_degree=3, tree_theta=0.61, tree_leaf=16,
                       tree_degree_fp32=3, tree_theta_fp32=0.61)
    x = syn.random_density(S.M, seed=29, smooth_points=S.geo.P)
    with ctr.CtrIbim.from_problem(prob, options=opts) as G:
        for prec, tol, BS, div in ((ctr.FP64, 1e-12, 256, 1), (ctr.DF64, 1e-11, 256, 2), (ctr.FP32_REFINE, 2e-5, 1024, 1)):
            op = tc.TreeOperator(S, BS=BS, min_far=4 ** 3 // div, **tree)
            assert _rel(G.matvec(x, prec), op.matvec(x)) < tol, prec
            assert G.pair_schedule(prec)["symmetric_pairs"] > 0


@pytest.mark.parametrize("method", ["hyb", "kreg"])
@pytest.mark.parametrize("kappa", [0.0, 0.1257])
def test_system_within_one_block(ctr, oracle_tables, kappa, method):
    prob = syn.sphere_problem(h=0.25, R=0.5, half_box=1.25, kappa=kappa)
    S = OracleSystem.from_problem(prob, tables=oracle_tables, method=method)
    assert S.M < 256
    x = syn.random_density(S.M, seed=3)
    ref = S.matvec(x)
    opts = ctr.Options(tube_halfwidth=prob.tube, method=ctr.METHOD_KREG if method == "kreg" else ctr.METHOD_HYB)
    with ctr.CtrIbim.from_problem(prob, options=opts) as G:
        assert G.M == S.M
        for prec, tol in ((ctr.DF64, 1e-12), (ctr.FP64, 1e-12), (ctr.FP32_REFINE, 2e-5)):
            assert _rel(G.matvec(x, prec), ref) < tol, prec
