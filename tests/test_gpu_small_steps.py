"""Runs that fit a cluster only when several temperatures share a launch: single
steps take the per-stage kernels, several the one launch, alone and beside other
runs, and every mix of the two gives the general sweep's anneal bit for bit."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GENERIC, NO_TUNE = 1, 2


def _descs(L, R, theta, n=1, temps=22):
    return [W.RunDesc(L, W.EA_PMJ if k % 2 else W.FERRO, R, theta, W.schedule(0.5, temps), seed=23, run_id=k,
                      disorder_id=k) for k in range(n)]


def _kinds(eng, n):
    _lib.pa_set_profiling(eng.h, True)
    _lib.pa_kernel_times(eng.h)
    eng.step(n)
    eng.sync()
    k = _lib.pa_kernel_times(eng.h)
    _lib.pa_set_profiling(eng.h, False)
    return k["small"][1], k["sweep"][1]


@pytest.mark.parametrize("L,R,theta,staged", [(16, 1500, 10, True), (8, 2000, 10, True), (16, 1500, 1, False),
                                              (16, 600, 10, False)])
@pytest.mark.parametrize("beside", [[], [(10, 300, 2)]])
def test_single_and_several_steps(L, R, theta, staged, beside):
    descs = _descs(L, R, theta, 2) + [W.RunDesc(a, W.FERRO, b, t, W.schedule(0.5, 22), seed=23, run_id=99)
                                      for a, b, t in beside]
    with _lib.Engine(descs, flags=GENERIC) as g:
        g.run_to_end()
        want = [g.records(0), g.records(1), *g.population(1)]
    with _lib.Engine(descs, flags=NO_TUNE) as eng:
        assert _kinds(eng, 1) == ((0, 1 + len(beside)) if staged else (1, len(beside)))
        if not beside:
            assert _kinds(eng, 4) == (1, 0)
        for n, graph in ((1, True), (3, True), (1, False), (1, True), (2, False), (20, True)):
            eng.step(n, graph)
        eng.sync()
        for x, y in zip([eng.records(0), eng.records(1), *eng.population(1)], want):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("L", [8, 16])
@pytest.mark.parametrize("R", [60, 350, 480, 700, 1000, 1500])
def test_clusters_on_both_sides_of_the_rule(L, R):
    for theta, n in ((1, 1), (3, 5), (6, 1), (14, 9)):
        descs = _descs(L, R, theta, n, 6)
        with _lib.Engine(descs, flags=GENERIC) as g, _lib.Engine(descs) as a, _lib.Engine(descs) as b:
            g.run_to_end()
            a.run_to_end()
            for _ in range(5):
                b.step(1)
            for k in (0, n - 1):
                for eng in (a, b):
                    assert np.array_equal(eng.records(k), g.records(k))
                    for x, y in zip(eng.population(k), g.population(k)):
                        assert np.array_equal(x, y)
