"""Pair kernels at the sizes where their loops can go wrong: ragged last tiles, steps and target blocks,
systems smaller than one block, strong and no screening; every arithmetic against the FP64 oracle.

Tolerances: float-float and FP64 operators 1e-12 (max norm, relative): a term carries 2^-44 or better and
the largest entries are sums of such terms; FP32 2e-5, as everywhere."""
import numpy as np
import pytest

import synthetic as syn
from oracle.system import OracleSystem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctr():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    return ctr


# node counts 862, 1404, 5014, 7290, 11203: remainders 2, 0, 2, 2, 3 by 4 and 94, 124, 22, 122, 67 by 128
PROBLEMS = {
    "sphere_862": lambda k: syn.sphere_problem(h=0.25, R=1.0, half_box=2.5, kappa=k),
    "sphere_1404": lambda k: syn.sphere_problem(h=0.25, R=1.3, half_box=2.8, kappa=k),
    "sphere_5014": lambda k: syn.sphere_problem(h=0.25, R=2.5, half_box=4.0, kappa=k),
    "sphere_7290": lambda k: syn.sphere_problem(h=0.25, R=3.0, half_box=4.5, kappa=k),
    "ellipsoid_11203": lambda k: syn.ellipsoid_problem(h=0.2, kappa=k),
}


@pytest.mark.parametrize("kappa", [0.0, 0.1257, 30.0])   # 30: kappa r up to 240, beyond the exponential's table
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_operator_at_ragged_sizes(ctr, oracle_tables, name, kappa):
    prob = PROBLEMS[name](kappa)
    S = OracleSystem.from_problem(prob, tables=oracle_tables)
    assert S.M == int(name.split("_")[1])
    x = syn.random_density(S.M, seed=S.M)
    ref = S.matvec(x)
    scale = np.max(np.abs(ref))
    with ctr.CtrIbim.from_problem(prob) as G:
        for precision, tol in ((ctr.DF64, 1e-12), (ctr.FP64, 1e-12), (ctr.FP32_REFINE, 2e-5)):
            assert np.max(np.abs(G.matvec(x, precision) - ref)) / scale < tol


@pytest.mark.parametrize("block", [512, 1024])
@pytest.mark.parametrize("name", ["kreg_sphere", "molecule"])
def test_excluded_pairs_of_symmetric_items(ctr, oracle_tables, name, block):
    """Rows with long and one-sided exclusion lists (K-reg cylinders; hybrid rows beside them): a pair that
    only one of its two rows leaves out is in the other's sum."""
    prob = syn.sphere_problem(h=0.25) if name == "kreg_sphere" else syn.molecule_problem(n_atoms=20, seed=1, h=0.5)
    kreg = name == "kreg_sphere"
    S = OracleSystem.from_problem(prob, tables=oracle_tables, method="kreg" if kreg else "hyb")
    sets = [set(S.excl_idx[S.excl_ptr[i]:S.excl_ptr[i + 1]].tolist()) for i in range(S.M)]
    assert sum(i not in sets[j] for i in range(S.M) for j in sets[i]) > 0   # one-way pairs exist
    x = syn.random_density(S.M, seed=5)
    ref = S.matvec(x)
    scale = np.max(np.abs(ref))
    opts = ctr.Options(tube_halfwidth=prob.tube, method=ctr.METHOD_KREG if kreg else ctr.METHOD_HYB, fp32_block=block)
    with ctr.CtrIbim.from_problem(prob, options=opts) as G:
        for precision, tol in ((ctr.DF64, 1e-12), (ctr.FP64, 1e-12), (ctr.FP32_REFINE, 2e-5)):
            assert np.max(np.abs(G.matvec(x, precision) - ref)) / scale < tol
