"""The server's memory accounting holds the workspace of a request's energy: one sum per 64 nodes and charge."""
from dataclasses import replace

import numpy as np
import pytest

import synthetic as syn

pytestmark = pytest.mark.gpu


def test_energy_workspace_is_charged():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2210_03699_gb300 as ctr
    base = syn.sphere_problem(h=0.25)
    rng = np.random.Generator(np.random.PCG64(1))
    n = 80000
    z = rng.normal(size=(n, 3))
    z *= (0.8 * rng.random((n, 1)) ** (1 / 3)) / np.linalg.norm(z, axis=1, keepdims=True)
    many = replace(base, charge_xyz=z, charge_q=np.full(n, 1.0 / n))
    peak = {}
    for name, prob in (("one", base), ("many", many)):
        with ctr.Server(max_slots=1) as sv:
            t = sv.submit_problem(prob)
            r = sv.wait(t, 300)
            assert r.status == 0
            M = r.M
            sv.release(t)
            st = sv.stats()
            peak[name] = st["peak_used_bytes"]
            assert st["used_bytes"] == 0
    units = (M + 63) // 64
    charges = 4 * 8 * (n - len(base.charge_q))
    assert peak["many"] - peak["one"] >= charges + 8 * units * (n - len(base.charge_q))
