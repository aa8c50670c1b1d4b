"""The batch solver (a warp or a block per realisation) and the thresholds and
row tables of a scoring call at the sizes where they can go wrong, against the
oracle: more than 32 rows, tables longer than a block, tables past their limit
(the preparation's search), equal thresholds across rows and classes, floors,
capacities outside the fast quotient's range, thresholds far below 1. Every
comparison is bit for bit."""

import dataclasses
import time

import numpy as np
import pytest

from conftest import alloc_matches, load_model
from paper_2608_19659_gb300 import workloads
from test_gpu_floors import _floors
from test_gpu_solve import _as_dict, _realisations, _solve_batch

pytestmark = pytest.mark.gpu


def _scaled(w, cap=1.0, demand=1.0):
    f = np.float32
    return dataclasses.replace(w, cap_lo=w.cap_lo * f(cap), cap_hi=w.cap_hi * f(cap), demand=w.demand * f(demand))


# (1000 realisations: a warp each; 20: a block each)
@pytest.mark.parametrize("n", [1000, 20])
@pytest.mark.parametrize("K,B,G,floors,cap,demand", [
    (2, 8, 16, False, 1.0, 3.0), (1, 7, 2000, False, 1.0, 900.0), (3, 5, 1, False, 1.0, 1.0),
    (4, 16, 64, True, 1.0, 6.0), (8, 32, 256, False, 1.0, 20.0), (9, 3, 40, True, 1.0, 2.0),
    (64, 2, 120, False, 1.0, 1.0), (33, 4, 64, True, 1.0, 1.0), (2, 6, 32, False, 1e-25, 1.0),
    (3, 33, 24, False, 1.0, 1e6), (2, 5, 12, False, 1e-30, 1e-30)])
def test_batch_solver(fsb, cuda, oracle_lib, n, K, B, G, floors, cap, demand):
    rng = np.random.default_rng(K * 100 + B + G)
    w = _scaled(workloads.random_small(rng, K, B, G), cap, demand)
    if floors:
        w = dataclasses.replace(w, floor=_floors(rng, w, w.cap_hi, w.tail_lo))
    c, t = _realisations(rng, w, n)
    p = oracle_lib.Problem.of(w)
    with load_model(fsb, w) as m:
        recs = _solve_batch(fsb, cuda, m, c, t)
    for r in sorted(set(range(0, n, max(1, n // 12))) | {1, 2, 3, 4, 5, n - 1}):
        assert alloc_matches(_as_dict(recs[r], K), oracle_lib.solve(p, c[r], t[r], 1), K), r


@pytest.mark.parametrize("K,B,G,demand,ties,floors", [
    (2, 8, 16, 3.0, True, False),      # equal rows and classes: ranks ordered by row
    (9, 4, 60, 3.0, True, True),       # more than 32 rows
    (8, 8, 256, 30.0, False, False),   # a table longer than a block of the preparation
    (6, 5, 300, 40.0, True, False),
    (32, 2, 272, 400.0, False, False)  # past the table's limit: the preparation searches
])
def test_scoring_thresholds(fsb, cuda, oracle_lib, K, B, G, demand, ties, floors):
    rng = np.random.default_rng(7 * K + G)
    w = _scaled(workloads.random_small(rng, K, B, G, p_infeasible=0.1), demand=demand)
    if ties:  # the same capacities in every class, demands equal or in the ratio 1 : 2
        lo, hi = np.repeat(w.cap_lo[:1], K, 0), np.repeat(w.cap_hi[:1], K, 0)
        lam = np.where(np.arange(K) % 2, np.float32(2.0), np.float32(1.0)) * w.demand[0]
        w = dataclasses.replace(w, cap_lo=lo, cap_hi=hi, demand=lam.astype(np.float32))
    if floors:
        w = dataclasses.replace(w, floor=_floors(rng, w, w.cap_hi, w.tail_lo))
    cand = rng.permutation(w.cells)[:4].astype(np.int32)
    w = dataclasses.replace(w, candidates=cand, O=4, S=6)
    qn = oracle_lib.triangular_table(4096)
    ref = oracle_lib.score(w, qn)
    with load_model(fsb, w) as m:
        r = fsb.fs_score_candidates(m, w.candidates, w.O, w.S, w.seed)
        many = fsb.fs_score_candidates(m, np.tile(cand, 400), w.O, w.S, w.seed)  # small preparation blocks
    assert r.gamma_t == ref.gamma_t and np.array_equal(r.sum_eo, ref.sum_eo)
    assert np.array_equal(r.score, ref.score) and r.best == ref.best
    assert np.array_equal(many.sum_eo, np.tile(ref.sum_eo, (400, 1)))


def test_no_capacity_and_a_small_demand(fsb, cuda, oracle_lib):
    """Rows without capacity whose smallest threshold times the demand underflows
    (demand 0.25; not at 1.0) are dismissed at once, not after a walk over all
    replica counts, in the solver and in a scoring call's thresholds."""
    w = workloads.random_small(np.random.default_rng(1), 1, 2, 8700, p_infeasible=0.0)
    zero = np.zeros_like(w.cap_lo)
    us = {}
    for lam in (1.0, 0.25):
        x = dataclasses.replace(w, cap_lo=zero, cap_hi=zero, demand=np.array([lam], np.float32), O=4, S=6)
        with load_model(fsb, x) as m:
            t = []
            for _ in range(30):
                a = time.perf_counter()
                am, _, gt = fsb.fs_solve_bounds(m)
                r = fsb.fs_score_candidates(m, x.candidates[:4], x.O, x.S, 1)
                t.append(time.perf_counter() - a)
        assert am["t_star"] == 0.0 and gt == 0.0 and not r.sum_eo.any()
        us[lam] = 1e6 * sorted(t)[len(t) // 2]
    assert us[0.25] < 1.5 * us[1.0], us  # (51 us both; with the walk 622)
