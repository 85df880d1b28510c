"""The parent map of steps that leave few families, in one CTA and split over
several: copy numbers below, at and far above the count from which a whole warp
writes a row's children, against the oracle bit for bit; and its time, which a
replica with very many copies must not multiply."""
import numpy as np
import pytest

import oracle as O
from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SEPARATE = 4


@pytest.mark.parametrize("L,betas", [(4, (0.0, 0.15, 0.3, 2.0)), (12, (0.0, 0.06, 0.2, 0.6)), (32, (0.0, 0.08, 0.16, 0.24))])
@pytest.mark.parametrize("R", [1, 33, 800, 5000, 9001, 20000])
def test_few_families(L, betas, R):
    d = W.RunDesc(L, W.FERRO, R, 1, np.array(betas), seed=13, run_id=R, R_cap=40 * R + 2000 if R < 100 else 0)
    with _lib.Engine([d], flags=SEPARATE) as eng:
        eng.run_to_end(use_graph=False)
        o = O.OracleRun.from_desc(eng.runs[0])
        for _ in range(1, d.n_beta):
            assert o.step() == 0
        g, r = eng.records(0), o.records()
        for f in ("R", "sumE", "sumE2", "n_fam", "max_fam", "sum_c2", "sumAbsM"):
            assert np.array_equal(g[f], r[f]), f
        _, E, M, fam, _ = eng.population(0)
        _, oE, oM, ofam = o.population()
        assert np.array_equal(E, oE) and np.array_equal(M, oM) and np.array_equal(fam, ofam)


def _resample_us(R, beta_f):
    d = [W.RunDesc(32, W.FERRO, R, 1, W.schedule(beta_f, 6), seed=3, run_id=k) for k in range(5)]
    best = 1e9
    with _lib.Engine(d, flags=SEPARATE | 2) as eng:
        for _ in range(6):
            eng.reset()
            eng.sync()
            _lib.pa_set_profiling(eng.h, True)
            _lib.pa_kernel_times(eng.h)
            eng.step(5)
            eng.sync()
            best = min(best, _lib.pa_kernel_times(eng.h)["resample"][0] * 1e3 / 5)
            _lib.pa_set_profiling(eng.h, False)
    return best


# R = 7000: one CTA per run, R = 9000: split.  The quench's steps took 64 us and 224 us when every
# replica wrote its own copies, against 16 to 17 us of the slow schedule's.
@pytest.mark.parametrize("R", [7000, 9000])
def test_a_quench_step_is_not_a_chain_of_copies(R):
    slow, fast = _resample_us(R, 0.05), _resample_us(R, 0.4)
    assert fast < 3 * slow + 5
