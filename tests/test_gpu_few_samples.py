"""The scorer's few-samples path (lanes per segment, no windows) on both sides of
its rule, against the oracle bit for bit: 1 to 128 calls a segment (group sizes
4 to 32, ragged last calls), many and few segments, floors, the monotone prior,
capacities outside the fast quotient's range, a caller's quantile table."""

import dataclasses

import numpy as np
import pytest

from conftest import load_model
from paper_2608_19659_gb300 import workloads
from test_gpu_floors import _floors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,B,G,n,O,S,prior,floors,cap", [
    (2, 8, 16, 16, 4, 1, 0, False, 1.0), (2, 8, 16, 16, 4, 17, 0, False, 1.0), (2, 8, 16, 64, 8, 62, 0, True, 1.0),
    (3, 5, 20, 31, 4, 127, 1, False, 1.0), (3, 5, 20, 31, 4, 129, 1, True, 1.0), (8, 6, 60, 40, 2, 33, 0, False, 1.0),
    (9, 4, 40, 33, 1, 30, 0, True, 1.0), (2, 4, 12, 9, 4, 50, 0, False, 1e-25)])
def test_few_samples(fsb, cuda, oracle_lib, K, B, G, n, O, S, prior, floors, cap):
    rng = np.random.default_rng(K * 100 + S)
    w = workloads.random_small(rng, K, B, G, p_infeasible=0.15)
    f = np.float32(cap)
    w = dataclasses.replace(w, cap_lo=w.cap_lo * f, cap_hi=w.cap_hi * f, demand=w.demand * np.float32(3.0), O=O, S=S,
                            prior=prior, candidates=rng.permutation(w.cells)[:n].astype(np.int32))
    if floors:
        w = dataclasses.replace(w, floor=_floors(rng, w, w.cap_hi, w.tail_lo))
    qn = oracle_lib.triangular_table(4096)
    ref = oracle_lib.score(w, qn)
    with load_model(fsb, w) as m:
        r = fsb.fs_score_candidates(m, w.candidates, O, S, w.seed)
        reps = -(-2048 // (n * O))  # enough segments for the rule's second half
        many = fsb.fs_score_candidates(m, np.tile(w.candidates, reps), O, S, w.seed)
    assert r.gamma_t == ref.gamma_t and r.best == ref.best and np.array_equal(r.sum_eo, ref.sum_eo)
    assert np.array_equal(many.sum_eo, np.tile(ref.sum_eo, (reps, 1)))


def test_few_samples_custom_quantiles(fsb, cuda, oracle_lib):
    rng = np.random.default_rng(3)
    w = workloads.random_small(rng, 2, 6, 16)
    qn = np.sort(rng.random(64)).astype(np.float32)
    w = dataclasses.replace(w, demand=w.demand * np.float32(3.0), O=4, S=21)
    ref = oracle_lib.score(w, qn)
    with load_model(fsb, w, qn) as m:
        r = fsb.fs_score_candidates(m, w.candidates, w.O, w.S, w.seed)
    assert np.array_equal(r.sum_eo, ref.sum_eo) and r.best == ref.best
