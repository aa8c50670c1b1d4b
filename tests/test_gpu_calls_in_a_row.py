"""Asynchronous scoring calls queued without a wait between them: a call's
thresholds may be made while the previous call's scenarios still run, so calls
with other bounds, other candidate lists (none among them), few and many
samples, and dumps, whose scenarios read the rows, are queued in a mixed order
on the model's stream, and every call's outputs must be those of the same call
made alone."""

import dataclasses

import numpy as np
import pytest

from conftest import load_model
from paper_2608_19659_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side_stream", [False, True])
@pytest.mark.parametrize("K,B,G", [(2, 8, 16), (8, 6, 200)])
def test_calls_in_a_row(fsb, cuda, oracle_lib, K, B, G, side_stream):
    torch = cuda
    rng = np.random.default_rng(K + G)
    ws = [workloads.random_small(np.random.default_rng(s), K, B, G, p_infeasible=0.1) for s in (1, 2)]
    lam = (ws[0].demand * np.float32(G / (4.0 * K))).astype(np.float32)
    ws = [dataclasses.replace(w, demand=lam, slo=ws[0].slo) for w in ws]
    st = torch.cuda.Stream() if side_stream else None
    w = ws[0]
    plans = [(rng.permutation(w.cells)[:n].astype(np.int32), O, S, dump)
             for n, O, S, dump in ((16, 4, 2000, 0), (1, 8, 64, 0), (0, 4, 10, 0), (w.cells, 8, 1500, 0), (3, 4, 40, 1),
                                   (40, 2, 4096, 0))]

    def alone(m, plan, which):
        cand, O, S, _ = plan
        x = ws[which]
        fsb.fs_update_bounds(m, x.cap_lo, x.cap_hi, x.tail_lo, x.tail_hi)
        return fsb.fs_score_candidates(m, cand, O, S, 9)

    with load_model(fsb, w) as m:
        ref = {(k, b): alone(m, p, b) for k, p in enumerate(plans) for b in (0, 1)}
        stride = fsb.fs_dump_stride(m)
    m = fsb.fs_load_model(w.cap_lo, w.cap_hi, w.tail_lo, w.tail_hi, w.slo, w.demand, G, K, B, stream=st)
    dev = [torch.from_numpy(p[0]).cuda() for p in plans]
    torch.cuda.synchronize()
    calls = []
    with m:
        at = 0
        for _ in range(40):
            k = int(rng.integers(len(plans)))
            cand, O, S, dump = plans[k]
            if rng.random() < 0.3:
                at ^= 1
                x = ws[at]
                fsb.fs_update_bounds(m, x.cap_lo, x.cap_hi, x.tail_lo, x.tail_hi)
            n = len(cand)
            out = [torch.zeros(max(n, 1), dtype=torch.float64, device="cuda"), torch.zeros(1, device="cuda"),
                   torch.zeros(1, dtype=torch.int32, device="cuda"),
                   torch.zeros((max(n, 1), O), dtype=torch.int64, device="cuda")]
            d = torch.zeros(n * O * S * stride, dtype=torch.uint8, device="cuda") if dump else None
            calls.append((k, at, out, d))
        torch.cuda.synchronize()  # the buffers are zeroed; the calls below queue back to back
        at = 0
        for k, b, out, d in calls:
            if b != at:
                at = b
                x = ws[at]
                fsb.fs_update_bounds(m, x.cap_lo, x.cap_hi, x.tail_lo, x.tail_hi)
            cand, O, S, _ = plans[k]
            fsb.fs_score_candidates_async(m, dev[k], O, S, 9, score_dev=out[0], gamma_t_dev=out[1], best_dev=out[2],
                                          sum_eo_dev=out[3], dump_dev=d, stream=st)
        fsb.fs_check(m)
        torch.cuda.synchronize()
    for k, b, out, _ in calls:
        r, n = ref[(k, b)], len(plans[k][0])
        assert float(out[1][0]) == r.gamma_t and int(out[2][0]) == r.best, (k, b)
        assert np.array_equal(out[3].cpu().numpy()[:n], r.sum_eo), (k, b)
        assert np.array_equal(out[0].cpu().numpy()[:n], r.score), (k, b)


def test_calls_under_capture(fsb, cuda, oracle_lib):
    """Three asynchronous calls captured into one CUDA graph after a single
    warm-up call, the graph replayed between calls made directly."""
    torch = cuda
    w = dataclasses.replace(workloads.make_workload(1), S=1000)
    plans = [(w.candidates, 8, 1000), (w.candidates[::9].copy(), 4, 60), (w.candidates[5:6].copy(), 8, 3000)]
    st = torch.cuda.Stream()
    with load_model(fsb, w) as m:
        ref = [fsb.fs_score_candidates(m, c, O, S, w.seed) for c, O, S in plans]
    m = fsb.fs_load_model(w.cap_lo, w.cap_hi, w.tail_lo, w.tail_hi, w.slo, w.demand, w.G, w.K, w.B, stream=st)
    dev = [torch.from_numpy(c).cuda() for c, _, _ in plans]
    sums = [torch.zeros((len(c), O), dtype=torch.int64, device="cuda") for c, O, _ in plans]
    torch.cuda.synchronize()

    def call(k):
        fsb.fs_score_candidates_async(m, dev[k], plans[k][1], plans[k][2], w.seed, sum_eo_dev=sums[k], stream=st)

    with m:
        call(0)  # the largest: buffers and launch shapes are there
        call(1)
        call(2)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            for k in range(3):
                call(k)
        for _ in range(4):
            for s in sums:
                s.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(st):
                call(0)
                g.replay()
                call(2)
                g.replay()
            torch.cuda.synchronize()
            for k in range(3):
                assert np.array_equal(sums[k].cpu().numpy(), ref[k].sum_eo), k


@pytest.mark.parametrize("at", [0, 7])
@pytest.mark.parametrize("S", [60, 1500])  # few samples and many
def test_list_written_by_the_call_before(fsb, cuda, oracle_lib, at, S):
    """A call whose candidate list holds the best cell of the call queued right
    before it. That call's reduction lets this one start before it has written
    the cell, so the entry read first is another one, and no cell at all."""
    torch = cuda
    rng = np.random.default_rng(at + S)
    w = workloads.make_workload(1)
    n, O, calls = 40, 8, 24
    lists = [rng.permutation(w.cells)[:n].astype(np.int32) for _ in range(calls)]
    stale = [-1, int(w.cells), int(lists[0][at])]  # (what the entry holds until then)
    with load_model(fsb, w) as m:
        ref = []
        for k in range(calls):
            if k:
                lists[k][at] = ref[-1].best
            ref.append(fsb.fs_score_candidates(m, lists[k], O, S, k))
        dev = [torch.from_numpy(c).cuda() for c in lists]
        best = torch.zeros(1, dtype=torch.int32, device="cuda")
        sums = [torch.zeros((n, O), dtype=torch.int64, device="cuda") for _ in range(calls)]
        for _ in range(2):  # (the first calls make the buffers)
            for k in range(1, calls):
                dev[k][at] = stale[k % 3]
            torch.cuda.synchronize()
            for k in range(calls):
                nxt = dev[k + 1][at:at + 1] if k + 1 < calls else best
                fsb.fs_score_candidates_async(m, dev[k], O, S, k, best_dev=nxt, sum_eo_dev=sums[k])
            fsb.fs_check(m)
            torch.cuda.synchronize()
            for k in range(calls):
                assert np.array_equal(dev[k].cpu().numpy(), lists[k]), k
                assert np.array_equal(sums[k].cpu().numpy(), ref[k].sum_eo), k
            assert int(best[0]) == ref[-1].best


def _long_plan(w):
    """Candidates of a call whose scenarios run for milliseconds, its records within the second buffer."""
    return np.tile(w.candidates, 23)[:1450].astype(np.int32), 8, 1 << 19


def test_capture_between_calls(fsb, cuda, oracle_lib):
    """A call captured between two calls queued without a wait does not run, so
    the second must keep clear of the first, whose scenarios are still running;
    the graph gives the captured call's sums later."""
    torch = cuda
    w = workloads.make_workload(1)
    cand, O, S = _long_plan(w)
    plans = [(cand, S, 1), (w.candidates, 1500, 2), (cand[::-1].copy(), 1500, 3)]  # before, captured, after
    st = torch.cuda.Stream()
    with load_model(fsb, w) as m:
        ref = [fsb.fs_score_candidates(m, c, O, s, seed) for c, s, seed in plans]
    m = fsb.fs_load_model(w.cap_lo, w.cap_hi, w.tail_lo, w.tail_hi, w.slo, w.demand, w.G, w.K, w.B, stream=st)
    dev = [torch.from_numpy(c).cuda() for c, _, _ in plans]
    sums = [torch.zeros((len(c), O), dtype=torch.int64, device="cuda") for c, _, _ in plans]

    def call(k):
        fsb.fs_score_candidates_async(m, dev[k], O, plans[k][1], plans[k][2], sum_eo_dev=sums[k], stream=st)

    with m:
        for k in (2, 2, 2):  # buffers of the largest records, both
            call(k)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(st):
            for _ in range(4):
                call(0)
            g.capture_begin()
            call(1)
            g.capture_end()
            running = not st.query()
            call(2)
        torch.cuda.synchronize()
        assert running, "the first call had finished before the capture did: it is too short for this test"
        assert np.array_equal(sums[0].cpu().numpy(), ref[0].sum_eo)
        assert np.array_equal(sums[2].cpu().numpy(), ref[2].sum_eo)
        assert not sums[1].any()
        with torch.cuda.stream(st):
            call(2)
            g.replay()
            call(0)
        torch.cuda.synchronize()
        for k in range(3):
            assert np.array_equal(sums[k].cpu().numpy(), ref[k].sum_eo), k


@pytest.mark.parametrize("what", ["bounds", "floors"])
def test_inputs_replaced_while_calls_run_on_another_stream(fsb, cuda, oracle_lib, what):
    """The model's stream is not the one its calls are queued on: new bounds and
    floors reach the device only once the calls queued with the old have read them."""
    torch = cuda
    w = dataclasses.replace(workloads.make_workload(1), floor=np.array([0.125, 0.0], np.float32))
    if what == "bounds":
        w2 = dataclasses.replace(w, cap_lo=w.cap_lo * np.float32(0.5), cap_hi=w.cap_hi * np.float32(0.75))
    else:
        w2 = dataclasses.replace(w, floor=np.array([0.0, 1.0], np.float32))
    cand, O, S = _long_plan(w)
    st = torch.cuda.Stream()
    with load_model(fsb, w2) as m:
        ref2 = fsb.fs_score_candidates(m, w.candidates, O, 1500, 5)
    with load_model(fsb, w) as m:  # (on the default stream)
        ref = fsb.fs_score_candidates(m, cand, O, S, 5)
        assert not np.array_equal(fsb.fs_score_candidates(m, w.candidates, O, 1500, 5).sum_eo, ref2.sum_eo)
        dev = [torch.from_numpy(c).cuda() for c in (cand, w.candidates)]
        sums = [torch.zeros((len(cand), O), dtype=torch.int64, device="cuda") for _ in range(4)]
        sums2 = torch.zeros((len(w.candidates), O), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        for x in sums:
            fsb.fs_score_candidates_async(m, dev[0], O, S, 5, sum_eo_dev=x, stream=st)
        if what == "bounds":
            fsb.fs_update_bounds(m, w2.cap_lo, w2.cap_hi, w2.tail_lo, w2.tail_hi)
        else:
            fsb.fs_set_floors(m, w2.floor)
        fsb.fs_score_candidates_async(m, dev[1], O, 1500, 5, sum_eo_dev=sums2, stream=st)
        fsb.fs_check(m, st)
    for x in sums:
        assert np.array_equal(x.cpu().numpy(), ref.sum_eo)
    assert np.array_equal(sums2.cpu().numpy(), ref2.sum_eo)


def test_records_past_the_second_buffer(fsb, cuda, oracle_lib):
    """Calls whose records do not fit the second buffer (32 MiB: more than 1842
    candidates here) among calls whose records do, in a mixed order without a wait,
    with plans of many and few samples and bounds replaced in between."""
    torch = cuda
    w = workloads.make_workload(1)
    ws = [w, dataclasses.replace(w, cap_lo=w.cap_lo * np.float32(0.5), cap_hi=w.cap_hi * np.float32(0.75))]
    rng = np.random.default_rng(12)
    O = 8
    plans = [(rng.permutation(np.tile(w.candidates, 32))[:n].astype(np.int32), S)
             for n, S in ((2000, 1500), (1800, 1500), (64, 4096), (2000, 60), (16, 60))]
    ref = {}
    for b, x in enumerate(ws):
        with load_model(fsb, x) as m:
            for k, (cand, S) in enumerate(plans):
                ref[k, b] = fsb.fs_score_candidates(m, cand, O, S, k)
    order = [int(k) for k in rng.integers(len(plans), size=48)]
    order[:8] = [0, 0, 2, 1, 0, 1, 1, 2]  # (large first, then each change of buffer)
    at = [int(b) for b in np.cumsum(rng.random(48) < 0.2) % 2]
    dev = [torch.from_numpy(c).cuda() for c, _ in plans]
    sums = [torch.zeros((len(plans[k][0]), O), dtype=torch.int64, device="cuda") for k in order]
    best = torch.zeros(len(order), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with load_model(fsb, ws[at[0]]) as m:
        for i, k in enumerate(order):
            if i and at[i] != at[i - 1]:
                x = ws[at[i]]
                fsb.fs_update_bounds(m, x.cap_lo, x.cap_hi, x.tail_lo, x.tail_hi)
            fsb.fs_score_candidates_async(m, dev[k], O, plans[k][1], k, best_dev=best[i:i + 1], sum_eo_dev=sums[i])
        fsb.fs_check(m)
        torch.cuda.synchronize()
    for i, k in enumerate(order):
        assert np.array_equal(sums[i].cpu().numpy(), ref[k, at[i]].sum_eo), (i, k)
        assert int(best[i]) == ref[k, at[i]].best, (i, k)
