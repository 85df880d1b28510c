"""Measurement and resampling with 128 and 512 threads per run: the same runs in
launches on both sides of the rules' lines, and beside a run of another size."""
import numpy as np
import pytest

import oracle as O
from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SEPARATE = 4


def _desc(L, R, k):
    return W.RunDesc(L, W.EA_PMJ if k % 2 else W.FERRO, R, 1, np.array([0.0, 0.05, 0.1, 0.3]), seed=21, run_id=k,
                     disorder_id=k)


@pytest.mark.parametrize("L,R", [(20, 40), (22, 3), (32, 700), (34, 33), (64, 40), (66, 5)])
def test_threads_do_not_change_results(L, R):
    want = None
    for n, extra in ((2, []), (153, []), (305, []), (2, [(8, 1500)]), (153, [(64, 2)])):
        descs = [_desc(L, R, k) for k in range(n)] + [_desc(a, b, 1000) for a, b in extra]
        with _lib.Engine(descs, flags=SEPARATE) as eng:
            eng.run_to_end(use_graph=False)
            got = [eng.records(0), eng.records(1)] + [x for k in (0, 1) for x in eng.population(k)]
        if want is None:
            want = got
            for k in (0, 1):
                o = O.OracleRun.from_desc(descs[k])
                for _ in range(3):
                    assert o.step() == 0
                for f in ("R", "sumE", "sumE2", "sumAbsM", "sumM2", "sum_c2", "n_fam", "max_fam"):
                    assert np.array_equal(got[k][f], o.records()[f]), f
        for x, y in zip(got, want):
            assert np.array_equal(x, y), (n, extra)
