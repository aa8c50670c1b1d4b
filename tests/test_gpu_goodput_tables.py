"""The goodput stage's shared tables (the other classes' best goodput per
realisation, class and threshold interval) at the ends of their range, against
the oracle bit for bit: a lone class (t* above every threshold), t* = 0 with
and without floors, floors that cannot be met, more than 32 rows, a pool that
takes the classes in several passes, the largest table of positions."""

import dataclasses

import numpy as np
import pytest

from conftest import load_model
from paper_2608_19659_gb300 import workloads
from test_gpu_floors import _floors

pytestmark = pytest.mark.gpu


def _check(fsb, oracle_lib, w):
    qn = oracle_lib.triangular_table(4096)
    ref = oracle_lib.score_goodput(w, qn)
    with load_model(fsb, w) as m:
        r = fsb.fs_score_goodput(m, w.candidates, w.O, w.S, w.seed)
    assert np.array_equal(r.sum_eo, ref.sum_eo), f"{int((r.sum_eo != ref.sum_eo).sum())} sums differ"
    assert r.gamma_gp == ref.gamma_gp and r.best == ref.best
    assert np.array_equal(r.gap, ref.gap) and np.array_equal(r.score, ref.score)


@pytest.mark.parametrize("K,B,G,demand,p_inf,floors,prior,O,S", [
    (1, 6, 24, 8.0, 0.2, False, 0, 4, 60), (1, 6, 24, 8.0, 0.2, False, 1, 4, 60),
    (3, 2, 20, 3.0, 0.8, False, 0, 4, 40),   # a class without an option: t* = 0
    (3, 2, 20, 3.0, 0.8, True, 1, 4, 40), (4, 3, 6, 4.0, 0.3, True, 0, 4, 40),
    (9, 2, 50, 3.0, 0.2, False, 0, 4, 10), (2, 4, 16, 3.0, 0.1, False, 0, 1, 200),
    (2, 4, 16, 3.0, 0.1, False, 1, 2, 200)])
def test_goodput_tables(fsb, cuda, oracle_lib, K, B, G, demand, p_inf, floors, prior, O, S):
    rng = np.random.default_rng(K * 10 + G + prior)
    w = workloads.random_small(rng, K, B, G, p_infeasible=p_inf)
    w = dataclasses.replace(w, demand=w.demand * np.float32(demand), O=O, S=S, prior=prior,
                            candidates=rng.permutation(w.cells)[:8].astype(np.int32))
    if floors:
        w = dataclasses.replace(w, floor=_floors(rng, w, w.cap_hi, w.tail_lo))
    _check(fsb, oracle_lib, w)


def test_goodput_pool_in_passes(fsb, cuda, oracle_lib):
    """Eight classes on 1024 GPUs at demands whose thresholds (over 4073 a
    realisation) need more rows than the pool's limit: the classes in two passes."""
    rng = np.random.default_rng(5)
    w = workloads.random_small(rng, 8, 2, 1024, p_infeasible=0.0)
    lam = rng.uniform(600.0, 900.0, 8).astype(np.float32)
    w = dataclasses.replace(w, demand=lam, O=4, S=3, candidates=np.array([0, 13, 37, 63], np.int32))
    _check(fsb, oracle_lib, w)


def test_new_bounds_allocate_nothing(fsb, cuda, oracle_lib):
    """A goodput call after one of the same plan takes no device memory, however
    many more thresholds its bounds have (some 90 a realisation, then 1200)."""
    torch = cuda
    w = workloads.random_small(np.random.default_rng(2), 8, 2, 256, p_infeasible=0.0)
    w = dataclasses.replace(w, candidates=w.candidates[:5].copy(), O=4, S=3, demand=np.full(8, 60.0, np.float32))
    many = dataclasses.replace(w, cap_lo=w.cap_lo * np.float32(200), cap_hi=w.cap_hi * np.float32(200))
    with load_model(fsb, many) as m:
        fsb.fs_score_goodput(m, w.candidates, w.O, w.S, w.seed)
        before = torch.cuda.mem_get_info()[0]
        fsb.fs_update_bounds(m, w.cap_lo, w.cap_hi, w.tail_lo, w.tail_hi)
        r = fsb.fs_score_goodput(m, w.candidates, w.O, w.S, w.seed)
        assert torch.cuda.mem_get_info()[0] == before
    assert np.array_equal(r.sum_eo, oracle_lib.score_goodput(w, oracle_lib.triangular_table(4096)).sum_eo)
