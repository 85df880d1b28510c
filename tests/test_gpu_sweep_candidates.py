"""Every launch shape of every bit-sliced sweep, whichever the tuner would pick,
against the general byte-plane sweep, bit for bit: schedules on both sides of the
kernels compiled for few sweeps, one and several tiles per CTA."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GENERIC, SEPARATE = 1, 4


def _mixed(L, runs, thetas, temps, R=3):
    b = W.schedule(0.9, temps)
    return [W.RunDesc(L, W.EA_PMJ if k % 3 == 1 else W.FERRO, R + (k * 7) % 40, thetas[k % len(thetas)], b, seed=11,
                      run_id=k, disorder_id=k) for k in range(runs)]


def _outcome(eng, steps, picks):
    ids = np.arange(len(eng.runs), dtype=np.uint32)
    eng.step(steps, False)
    return [eng.step_records(ids)] + [x for k in picks for x in eng.population(k)]


def _each_candidate(descs, steps, several):
    L, picks = descs[0].L, sorted({0, 1, len(descs) // 2, len(descs) - 1})
    with _lib.Engine(descs, flags=GENERIC) as g:
        want = _outcome(g, steps, picks)
    with _lib.Engine(descs, flags=SEPARATE) as eng:
        n = _lib.pa_sweep_candidates(eng.h)[0][1]
        for c in range(n):
            _lib.pa_set_sweep_shape(eng.h, L, c)
            eng.reset()
            assert _lib.pa_tuning_pending(eng.h) == 0
            ran, _, _, tiles = _lib.pa_sweep_candidates(eng.h)[0]
            assert ran == c
            if several and not (L == 12 and c >= n - 2):  # L = 12's padded rows take one tile per CTA
                assert tiles > 1
            for x, y in zip(_outcome(eng, steps, picks), want):
                assert np.array_equal(x, y), c
        with pytest.raises(_lib.PAError):
            _lib.pa_set_sweep_shape(eng.h, L, n)


SIZES = [4, 6, 8, 10, 12, 14, 16, 18, 26, 30, 32, 46, 62, 64, 66, 100, 126, 128, 206, 256]


@pytest.mark.parametrize("thetas", [(6, 9, 5), (1, 0, 3, 2, 4), (25, 5, 11)])
@pytest.mark.parametrize("L", SIZES)
def test_every_candidate(L, thetas):
    _each_candidate(_mixed(L, 5, thetas, 4, R=1), 3, False)


# enough tiles for several per CTA with every candidate's tile size
@pytest.mark.parametrize("L,runs", [(6, 10000), (8, 5000), (10, 10000), (12, 10000), (16, 5000), (30, 5000),
                                    (32, 1500), (46, 2400), (64, 300), (100, 480), (128, 160), (256, 90)])
def test_every_candidate_with_several_tiles_per_cta(L, runs):
    _each_candidate(_mixed(L, runs, (1, 0, 3, 2, 4), 3), 2, True)


def test_a_fixed_shape_is_given_back():
    with _lib.Engine(_mixed(64, 3, (2,), 20), flags=SEPARATE | 2) as eng:
        first = _lib.pa_sweep_candidates(eng.h)
        _lib.pa_set_sweep_shape(eng.h, 64, 1)
        eng.step(2)
        assert _lib.pa_sweep_candidates(eng.h)[0][0] == 1
        _lib.pa_set_sweep_shape(eng.h, 64)
        eng.step(2)
        assert _lib.pa_sweep_candidates(eng.h) == first
        for bad in ((65, 0), (2, 0), (258, 0)):
            with pytest.raises(_lib.PAError):
                _lib.pa_set_sweep_shape(eng.h, *bad)
