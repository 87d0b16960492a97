"""Charges at any finite position: one so far away that the square of its distance overflows adds nothing to the
right-hand side, as in the oracle (1/inf); neither does one at 1e140, whose contribution is below the sum's
rounding.  The values without them, bit for bit."""
import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


def test_far_charges_add_nothing():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    p = syn.sphere_problem(h=0.25)
    g = p.grid
    far = np.array([[1e160, 0.0, 0.0], [0.0, -3e200, 1e10], [1e140, 1e140, 0.0], [0.0, 0.0, 1.7e308]])
    q = np.array([1.0, -2.0, 0.5, 1.0])
    with ctr.CtrIbim.from_problem(p) as G:
        ref = G.rhs()
    with ctr.CtrIbim(g.n, g.origin, g.h, p.sdist, p.eps_in, p.eps_out, p.kappa,
                     np.concatenate([p.charge_xyz, far]), np.concatenate([p.charge_q, q])) as G:
        assert np.array_equal(G.rhs(), ref)
        _, _, info = G.solve()
        assert info.converged
