"""K-reg cylinders of tubes wider than the grid: the search covers the grid's part of its cube, whatever the cube's
size.  Whole numbers: the correction rows equal a search over all tube nodes."""
from dataclasses import replace

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width", [2, 13, 700, 1 << 20])   # half-width in grid spacings; (2 * 705 + 1)^3 > 2^31
def test_kreg_rows_at_any_tube_width(width):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    base = syn.sphere_problem(h=0.25, R=1.0, half_box=2.5)
    h = base.grid.h
    # the tube nodes are those within 2 h of the sphere at every width
    sd = np.where(np.abs(base.sdist) < 2 * h, base.sdist, np.copysign(4.0 * (1 << 20), base.sdist))
    prob = replace(base, sdist=sd, tube=width * h)
    with ctr.CtrIbim.from_problem(prob, options=ctr.Options(tube_halfwidth=prob.tube, method=ctr.METHOD_KREG)) as G:
        P, n, _ = G.geometry()
        lin = np.asarray(G.nodes())
        ptr, node, _ = G.corrections()
    nx, ny, _ = prob.grid.n
    ijk = np.stack([lin % nx, (lin // nx) % ny, lin // (nx * ny)], axis=1)
    y = np.asarray(prob.grid.origin) + h * ijk.astype(np.float64)
    tau = 2.0 * h
    K = int(np.ceil((prob.tube + tau) / h)) + 1
    total = 0
    for i in range(len(lin)):
        v = y - P[i]
        s = (v[:, 0] * n[i, 0] + v[:, 1] * n[i, 1]) + v[:, 2] * n[i, 2]
        t = v - s[:, None] * n[i]
        q2 = (t[:, 0] * t[:, 0] + t[:, 1] * t[:, 1]) + t[:, 2] * t[:, 2]
        want = np.nonzero((q2 < tau * tau) & (np.abs(ijk - ijk[i]).max(axis=1) <= K))[0]
        assert np.array_equal(node[ptr[i]:ptr[i + 1]], want)
        total += len(want)
    assert total > 10 * len(lin)
