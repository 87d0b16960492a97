"""The pair schedules' planning (host): every interaction is in exactly one item, whichever way near block pairs
are evaluated, and systems whose closed exclusion lists do not fit in 32 bits have no item that needs them."""
import ctypes

import numpy as np
import pytest

import synthetic as syn
from oracle.system import OracleSystem

ctr = pytest.importorskip("paper_2210_03699_gb300")

ONE, SYM, NEAR = 0, 1, 2


@pytest.fixture(scope="module")
def planner():
    import native_lib
    L = native_lib.load("planner.cpp")
    L.plan_direct.restype = L.plan_tree.restype = L.cut_direct.restype = ctypes.c_int64
    L.estimated_seconds.restype = ctypes.c_double
    return L


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _coverage(items, M, BS):
    """How often each ordered pair (row, source) is evaluated."""
    c = np.zeros((M, M), dtype=np.int64)
    for I, j0, j1, kind in items:
        rows = slice(I * BS, min(M, (I + 1) * BS))
        c[rows, j0:j1] += 1
        if kind != ONE:
            c[j0:j1, rows] += 1
    return c


def test_closed_lists_fit_in_32_bits(planner):
    """Row starts over 2 E entries and entries 4 j + flags: both within an int32."""
    fit = lambda M, E: planner.closed_fit(ctypes.c_int64(M), ctypes.c_int64(E))
    assert fit(200000, 10**6) and fit(4300000, 2**30 - 1) and fit(2**29 - 1, 2**29)
    assert not fit(4300000, 2**30) and not fit(4300000, 2**31 - 1) and not fit(2**29, 2**29)


@pytest.mark.parametrize("closed", [0, 1])
@pytest.mark.parametrize("BS", [256, 512, 1024])
@pytest.mark.parametrize("M", [1, 256, 700, 1537, 2500])
def test_direct_runs_cover_every_interaction_once(planner, M, BS, closed):
    nb0 = (M + 255) // 256
    rng = np.random.Generator(np.random.PCG64(M))
    f = np.triu(rng.random((nb0, nb0)) < 0.4)
    flags = np.ascontiguousarray((f | f.T | np.eye(nb0, dtype=bool)).astype(np.uint8))
    out = np.zeros((4096, 4), dtype=np.int32)
    n = planner.plan_direct(ctypes.c_int64(M), BS, _p(flags), 256, nb0, closed, ctypes.c_int64(len(out)), _p(out))
    items = out[:n]
    assert 0 < n <= len(out)
    assert np.all(_coverage(items, M, BS) == 1)
    assert closed or not np.any(items[:, 3] == NEAR)
    near = np.kron(flags, np.ones((256, 256), dtype=np.uint8))[:M, :M]
    for I, j0, j1, kind in items:   # no correction pair in a plain symmetric item
        assert kind != SYM or not near[I * BS:(I + 1) * BS, j0:j1].any()


# 304 and 456 resident blocks: two and three on each of 152 SMs.  Without fine pieces these have 9.8, 12.4 and 12.3
# million items, with them 18.6, 23.5 and 23.4.
@pytest.mark.parametrize("pol,tile,slots,M", [(2, 128, 304, 1600000), (2, 128, 304, 1800001), (1, 128, 456, 3700000)])
def test_large_schedules_fit_the_engine(planner, pol, tile, slots, M):
    """The engine names items with 24 bits and refuses longer schedules."""
    BS = 256
    pairs = (ctypes.c_int64 * 2)()
    n = planner.cut_direct(pol, ctypes.c_int64(M), BS, tile, slots, pairs, ctypes.c_int64(0), None)
    assert 0 < n < 2 ** 24
    t = np.minimum(BS, M - BS * np.arange((M + BS - 1) // BS, dtype=np.int64))
    diag = int(np.sum(t * t))
    assert pairs[0] == diag and 2 * pairs[1] + diag == M * M


def test_runs_end_in_fine_pieces(planner):
    M, BS, tile = 178575, 256, 128
    pairs = (ctypes.c_int64 * 2)()
    out = np.zeros((1 << 20, 4), dtype=np.int32)
    n = planner.cut_direct(1, ctypes.c_int64(M), BS, tile, 456, pairs, ctypes.c_int64(len(out)), _p(out))
    items = out[:n]
    run = items[(items[:, 0] == 0) & (items[:, 3] == SYM)]
    lens = run[:, 2] - run[:, 1]
    assert np.array_equal(run[1:, 1], run[:-1, 2]) and run[-1, 2] == M
    assert lens[0] >= 4 * lens[-2] and np.all(np.diff(lens[:-1]) <= 0)


@pytest.mark.parametrize("closed", [0, 1])
@pytest.mark.parametrize("method", ["hyb", "kreg"])
def test_tree_runs_cover_the_near_field_once(planner, oracle_tables, method, closed):
    prob = syn.molecule_problem(n_atoms=20, seed=1, h=0.5) if method == "hyb" else syn.ellipsoid_problem(h=0.25)
    S = OracleSystem.from_problem(prob, tables=oracle_tables, method=method)
    M, BS = S.M, 256
    ptr, idx = np.asarray(S.excl_ptr, dtype=np.int64), np.asarray(S.excl_idx, dtype=np.int64)
    plan = ctr.farfield_plan(S.geo.ijk, ptr, idx, 2, 3, 0.61, 16, BS)
    perm, near_ptr = plan["perm"], np.ascontiguousarray(plan["near_ptr"], dtype=np.int64)
    near_rng = np.ascontiguousarray(plan["near_rng"], dtype=np.int32)
    pos = np.empty(M, dtype=np.int64)
    pos[perm] = np.arange(M)
    rows = [np.sort(pos[idx[ptr[i]:ptr[i + 1]]]) for i in perm]   # correction rows in tree positions
    tptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    texcl = np.concatenate(rows).astype(np.int32)
    out = np.zeros((1 << 16, 4), dtype=np.int32)
    n = planner.plan_tree(ctypes.c_int64(M), BS, _p(tptr), _p(texcl), ctypes.c_int64(len(near_ptr) - 1), _p(near_ptr),
                          _p(near_rng), closed, ctypes.c_int64(len(out)), _p(out))
    items = out[:n]
    assert 0 < n <= len(out)
    want = np.zeros((M, M), dtype=np.int64)
    for I in range(len(near_ptr) - 1):
        for b, e in near_rng[near_ptr[I]:near_ptr[I + 1]]:
            want[I * BS:(I + 1) * BS, b:e] = 1
    assert np.array_equal(_coverage(items, M, BS), want)
    kinds = set(items[:, 3].tolist())
    assert SYM in kinds and (NEAR in kinds) == bool(closed)
    pair = np.zeros((M, M), dtype=bool)
    for p in range(M):
        pair[p, texcl[tptr[p]:tptr[p + 1]]] = True
    for I, j0, j1, kind in items:
        if kind == SYM:
            r = slice(I * BS, (I + 1) * BS)
            assert not pair[r, j0:j1].any() and not pair[j0:j1, r].any()


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["kreg_sphere", "molecule"])
def test_near_block_pairs_one_sided(planner, oracle_tables, name):
    """A handle planned without closed lists: the operator's tolerances of the pair-edge tests."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    prob = syn.sphere_problem(h=0.25) if name == "kreg_sphere" else syn.molecule_problem(n_atoms=20, seed=1, h=0.5)
    kreg = name == "kreg_sphere"
    S = OracleSystem.from_problem(prob, tables=oracle_tables, method="kreg" if kreg else "hyb")
    x = syn.random_density(S.M, seed=5)
    ref = S.matvec(x)
    scale = np.max(np.abs(ref))
    opts = ctr.Options(tube_halfwidth=prob.tube, method=ctr.METHOD_KREG if kreg else ctr.METHOD_HYB)
    with ctr.CtrIbim.from_problem(prob, options=opts) as G:
        before = G.pair_schedule(ctr.FP64)["symmetric_pairs"]
        assert planner.replan_one_sided(G._h) == 0
        assert G.pair_schedule(ctr.FP64)["symmetric_pairs"] < before
        for precision, tol in ((ctr.DF64, 1e-12), (ctr.FP64, 1e-12), (ctr.FP32_REFINE, 2e-5)):
            assert np.max(np.abs(G.matvec(x, precision) - ref)) / scale < tol


@pytest.mark.gpu
def test_estimated_application_times(planner):
    """The engine's estimates, by which it splits applications, against the times: their ratios to the FP32 one
    (clocks cancel) within 8%."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with ctr.CtrIbim.from_problem(syn.ellipsoid_problem(h=0.05)) as G:
        t, e = [], []
        for pol, prec in enumerate((ctr.FP32_REFINE, ctr.DF64, ctr.FP64)):
            G.time_operator(prec, reps=1)
            t.append(min(G.time_operator(prec, reps=2)["pairs_ms"] for _ in range(2)))
            e.append(planner.estimated_seconds(G._h, pol))
    for pol in (1, 2):
        assert abs((e[pol] / e[0]) / (t[pol] / t[0]) - 1) < 0.08, (t, e)
