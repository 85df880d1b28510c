"""The sweeps' launch shape is chosen for the load and the kind of schedule, not
once for a lattice size: one engine's choice is no other load's, in one process
and in one engine whose resident runs change."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib, serve
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SEPARATE, NO_TUNE = 4, 2
LARGE = 90000  # replicas: at least 8 CTAs per SM of 64 replicas


def _run(L, R, theta, k=0, temps=16):
    return W.RunDesc(L, W.FERRO, R, theta, W.schedule(0.4, temps), seed=17, run_id=k, disorder_id=k)


def _tuned(descs):
    """(choices pending before the first step, children per thread chosen)"""
    with _lib.Engine(descs, flags=SEPARATE) as eng:
        pending = _lib.pa_tuning_pending(eng.h)
        eng.step(11, False)
        assert _lib.pa_tuning_pending(eng.h) == 0
        return pending, _lib.pa_sweep_candidates(eng.h)[0][2]


def test_the_first_engine_does_not_choose_for_every_load():
    L = 22  # tuned at these loads by no other test
    pending, children = _tuned([_run(L, 100, 6)])
    assert children == 1  # 28 us against 48 with two children per thread
    for descs in ([_run(L, LARGE, 6)], [_run(L, LARGE, 2)], [_run(L, 100, 2)]):
        assert _tuned(descs)[0] == 1
    for descs in ([_run(L, LARGE, 7)], [_run(L, LARGE, 1)], [_run(L, 130, 9)]):
        assert _tuned(descs)[0] == 0  # these loads and schedules have been timed


@pytest.mark.parametrize("L", [30, 32, 64, 100, 128, 256])
def test_default_shapes_follow_the_load(L):
    for R, children in ((40, 1), (4000000 // L // L * 40, 2)):
        with _lib.Engine([_run(L, R, 1, temps=2)], flags=SEPARATE | NO_TUNE) as eng:
            assert _lib.pa_sweep_candidates(eng.h)[0][2] == children


def test_a_server_whose_residents_change():
    L = 26
    srv = serve.Server(serve.config_for_budget(2 << 30, max_runs=4, min_L=8, max_L=64, max_n_beta=40), flags=SEPARATE)
    try:
        h = srv.h
        small = _lib.pa_admit(h, [_run(L, 60, 6, 1, 30)])[0]
        _lib.pa_anneal_step(h, 11, False)
        assert _lib.pa_tuning_pending(h) == 0
        large = _lib.pa_admit(h, [_run(L, LARGE, 6, 2, 30)])[0]
        _lib.pa_anneal_step(h, 1, False)
        assert _lib.pa_tuning_pending(h) == 1
        _lib.pa_anneal_step(h, 10, False)
        assert _lib.pa_tuning_pending(h) == 0
        _lib.pa_retire(h, large)
        _lib.pa_anneal_step(h, 1, False)
        assert _lib.pa_tuning_pending(h) == 0 and _lib.pa_sweep_candidates(h)[0][2] == 1
        _lib.pa_anneal_step(h, 40)
        _lib.pa_sync(h)
        got = _lib.pa_records(h, small, 30)
    finally:
        srv.close()
    with _lib.Engine([_run(L, 60, 6, 1, 30)], flags=1) as eng:
        eng.run_to_end()
        assert np.array_equal(eng.records(0), got)
