"""Reads of a population in mid-anneal: a few replicas unpacked on the host, more on
the device, and the anneal that goes on afterwards."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SEPARATE = 4


def _engine(L, R, flags=SEPARATE, model=W.EA_PMJ, temps=12):
    return _lib.Engine([W.RunDesc(L, model, R, 2, W.schedule(0.8, temps), seed=29, run_id=1)], flags=flags)


# 2560 sites and one replica more; L/2 a power of two, padded, and repacked rows
@pytest.mark.parametrize("L,n", [(4, 160), (6, 71), (12, 17), (16, 10), (32, 2), (44, 1), (46, 1)])
def test_slices_on_both_sides_of_the_line(L, n):
    with _engine(L, 300) as eng:
        eng.step(5)
        s, E, M, fam, _ = eng.population(0)
        assert np.array_equal(s.sum(axis=1, dtype=np.int64), M)
        for first, count in ((0, 1), (3, n), (3, n + 1), (len(s) - 1, 1), (len(s) - 2, 500)):
            l0 = eng.launches
            p, e, m, f, R, _ = _lib.pa_population_slice(eng.h, 0, first, count, L * L)
            got = min(count, len(s) - first)
            assert eng.launches - l0 == (0 if got * L * L <= 2560 else 1)
            assert R == len(s) and len(p) == got
            for a, b in ((p, s), (e, E), (m, M), (f, fam)):
                assert np.array_equal(a, b[first:first + got])
