"""The tier-4 solver's batch and wide instances, with packed and two-word values
and with its cells in shared memory or in scratch, against the oracle bit for
bit (t* = 0, where every class's whole budget is free, among the realisations)."""

import dataclasses

import numpy as np
import pytest

from conftest import load_model
from paper_2608_19659_gb300 import workloads
from test_gpu_floors import _floors
from test_gpu_solve import _realisations, _solve_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K,B,G,scale,floors", [
    (1000, 2, 8, 16, 1.0, False), (700, 3, 5, 33, 1.0, True), (610, 1, 3, 1, 1.0, False),
    (620, 8, 4, 256, 1.0, False),            # one warp, cells in scratch
    (612, 3, 4, 40, 2.0**24, False),         # two-word values
    (9, 8, 32, 256, 1.0, True), (7, 12, 3, 64, 2.0**24, False),
    (6, 4, 2, 2000, 2.0**24, False)])        # wide, cells in scratch
def test_lexicographic_batch(fsb, cuda, oracle_lib, n, K, B, G, scale, floors):
    rng = np.random.default_rng(n + K + G)
    w = workloads.random_small(rng, K, B, G, p_infeasible=0.15)
    f = np.float32(scale)
    d = np.float32(max(1.0, G / (4.0 * K)))
    w = dataclasses.replace(w, cap_lo=w.cap_lo * f, cap_hi=w.cap_hi * f, demand=w.demand * f * d)
    if floors:
        w = dataclasses.replace(w, floor=_floors(rng, w, w.cap_hi, w.tail_lo))
    cap, tail = _realisations(rng, w, n)
    p = oracle_lib.Problem.of(w)
    with load_model(fsb, w) as m:
        fsb.fs_set_objective(m, fsb.FS_OBJECTIVE_LEXICOGRAPHIC)
        got = _solve_batch(fsb, cuda, m, cap, tail)
    for r in sorted(set(range(0, n, max(1, n // 6))) | {1, 2, 3, 4, 5, n - 1}):
        a, gp = oracle_lib.solve_lex(p, cap[r], tail[r])
        assert got[r]["t_star"] == np.float32(a.t_star) and got[r]["total_gpus"] == a.total_gpus, r
        assert got[r]["goodput"] == gp * 2.0**-20, r
        assert list(got[r]["replicas"][:K]) == a.replicas and list(got[r]["tp"][:K]) == a.tp, r
        assert list(got[r]["bin"][:K]) == a.bin, r
