"""Sweeps of several lattice sizes on the engine's side streams: the priority and
the order of the caller's stream."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

NO_TUNE, SEPARATE = 2, 4


def _mixed(sizes, temps=8):
    out = []
    for k, (L, R) in enumerate(sizes):
        out.append(W.RunDesc(L, W.EA_PMJ if k % 2 else W.FERRO, R, 3, W.schedule(0.7, temps), seed=31, run_id=k,
                             disorder_id=k))
    return out


def test_side_streams_take_the_callers_priority():
    import torch

    low, high = torch.cuda.Stream.priority_range()
    assert high < low
    for priority in (low, high):
        mine = torch.cuda.Stream(priority=priority)
        with _lib.Engine(_mixed([(10, 50), (16, 60), (30, 20)]), stream=mine.cuda_stream, flags=SEPARATE) as eng:
            side = [torch.cuda.ExternalStream(s) for s in _lib.pa_side_streams(eng.h)]
            assert len(side) == 3 and mine.priority == priority
            assert all(s.priority == priority for s in side)
    with _lib.Engine(_mixed([(10, 50), (10, 60)])) as eng:  # one size: nothing to spread
        assert _lib.pa_side_streams(eng.h) == []


SIZES = [(6, 300), (8, 200), (10, 250), (16, 150), (30, 60), (32, 40), (64, 20)]  # more than the streams: a second turn


def _with_overlaps(temps=8):
    descs = _mixed(SIZES, temps)
    descs[1].overlap = descs[4].overlap = W.Q_SHIFT
    descs[3].overlap = W.Q_WANG
    return descs


def _all(eng):
    out = []
    for k, d in enumerate(eng.runs):
        r = eng.records(k, qhist=bool(d.overlap), wang=bool(d.overlap))
        out += list(r) if isinstance(r, tuple) else [r]
        out += list(eng.population(k))
    return out


def _same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)


def test_spread_sweeps_equal_serial_ones():
    descs = _with_overlaps()
    with _lib.Engine(descs, flags=1) as g:  # the byte-plane kernel
        g.run_to_end()
        want = _all(g)
    with _lib.Engine(descs, flags=NO_TUNE | SEPARATE) as eng:
        assert len(_lib.pa_side_streams(eng.h)) == 3
        _lib.pa_set_profiling(eng.h, True)  # one after another on the engine's stream
        eng.step(7)
        _same(_all(eng), want)
        assert _lib.pa_kernel_times(eng.h)["sweep"][1] == 7 * len(SIZES)
        _lib.pa_set_profiling(eng.h, False)
        for graph in (False, True, True):
            eng.reset()
            l0 = eng.launches
            eng.step(2, graph)
            eng.step(5, graph)
            _same(_all(eng), want)
            assert eng.launches > l0
        eng.reset()
        for k in range(7):  # eager, captured and profiled steps in turn
            _lib.pa_set_profiling(eng.h, k % 3 == 2)
            eng.step(1, k % 3 == 0)
        _same(_all(eng), want)


def test_spread_sweeps_while_residents_change():
    descs = _mixed(SIZES, 12)
    from paper_2207_05535_gb300 import serve

    want = []
    for d in descs:
        with _lib.Engine([d], flags=1) as g:
            g.run_to_end()
            want.append(g.records(0))
    srv = serve.Server(serve.config_for_budget(1 << 30, max_runs=8, min_L=6, max_L=64, max_n_beta=12),
                       flags=NO_TUNE | SEPARATE)
    try:
        jobs = [serve.Job(d, 0.0) for d in descs]
        for k, graph in zip(range(3), (True, False, True)):  # from one size to five
            for j in jobs[2 * k:2 * k + 2] if k else jobs[:1]:
                assert srv.try_admit(j)
            _lib.pa_anneal_step(srv.h, 2, graph)
        for j in jobs[1:2] + jobs[6:]:
            if j.slot < 0:
                assert srv.try_admit(j)
        done = []
        for _ in range(40):
            _lib.pa_anneal_step(srv.h, 1, True)
            done += srv.collect()
        assert len(done) == len(jobs)
        for j, w in zip(jobs, want):
            assert np.array_equal(j.records, w)
    finally:
        srv.close()


def test_spread_sweeps_keep_the_order_of_the_callers_stream():
    import torch

    descs = _with_overlaps()
    mine = torch.cuda.Stream()
    with _lib.Engine(descs, flags=NO_TUNE | SEPARATE) as g:
        g.run_to_end()
        want = _all(g)
    with _lib.Engine(descs, stream=mine.cuda_stream, flags=NO_TUNE | SEPARATE) as eng:
        side = [torch.cuda.ExternalStream(s) for s in _lib.pa_side_streams(eng.h)]
        eng.step(1, False)
        eng.step(1, True)
        eng.sync()
        for graph in (False, True):
            with torch.cuda.stream(mine):
                torch.cuda._sleep(100_000_000)  # about 50 ms on the caller's stream ahead of the sweeps
            eng.step(2, graph)
            after = torch.cuda.Event()
            after.record(mine)
            assert not after.query()
            if not graph:
                assert not any(s.query() for s in side)  # the sweeps wait for what the caller had enqueued
            after.synchronize()
            assert all(s.query() for s in side)  # and what follows waits for them
        eng.step(1)
        _same(_all(eng), want)
