"""Resampling, measurement and Wang pairing at the sizes where their launches
change: against the oracle, bit for bit (ln Q and -beta F to 1e-12 relative, a few
ulp of the device's log)."""
import numpy as np
import pytest

import oracle as O
from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _against_oracle(descs, flags=0):
    n = max(d.n_beta for d in descs)
    with _lib.Engine(descs, flags=flags) as eng:
        eng.run_to_end(use_graph=False)
        for k, d in enumerate(descs):
            o = O.OracleRun.from_desc(d)
            for _ in range(1, d.n_beta):
                assert o.step() == 0
            g, r = eng.records(k), o.records()
            for f in g.dtype.names:
                if f in ("lnQ", "minus_betaF"):
                    assert np.allclose(g[f], r[f], rtol=1e-12, atol=1e-12), (k, f)
                elif f in r.dtype.names:
                    assert np.array_equal(g[f], r[f]), (k, f)
            _, E, M, fam, _ = eng.population(k)
            _, oE, oM, ofam = o.population()
            assert np.array_equal(E, oE) and np.array_equal(M, oM) and np.array_equal(fam, ofam)
    assert n > 1


def _multi(L, R, run=0, beta_f=0.4, model=W.FERRO):
    return W.RunDesc(L, model, R, 1, W.schedule(beta_f, 4), seed=3, run_id=run, disorder_id=run, resample=W.MULTINOMIAL)


# one replica, fewer than a warp, chunks that do not divide, the block sizes' edge, more levels
# than shared memory holds (L = 64: up to 4097, of which a population at beta = 0 takes few; a
# second run of another size sets the launch's shared memory), more replicas than it stages
@pytest.mark.parametrize("sizes", [[(8, 1)], [(8, 31), (16, 33)], [(16, 1000), (6, 2048)], [(16, 2049), (8, 5)],
                                   [(30, 3001)], [(64, 700), (8, 400)], [(4, 25000)], [(8, 24576), (8, 24577)]])
def test_multinomial(sizes):
    _against_oracle([_multi(L, R, k) for k, (L, R) in enumerate(sizes)])


# levels far apart: a glass population quenched in one step spreads over many levels
def test_multinomial_many_levels():
    _against_oracle([W.RunDesc(64, W.EA_PMJ, 3000, 1, np.array([0.0, 0.02, 0.7, 0.72]), seed=4, run_id=1,
                               resample=W.MULTINOMIAL)])


# 128-thread and 512-thread launches (capacity up to 1024 and above), with lattice sizes on both
# sides of the counters' shared memory in one launch
@pytest.mark.parametrize("R", [1, 2, 31, 127, 128, 129, 500, 700, 1100])
def test_small_population_launches(R):
    b = W.schedule(0.6, 4)
    _against_oracle([W.RunDesc(L, W.EA_PMJ if L % 4 else W.FERRO, R, 1, b, seed=6, run_id=L) for L in (6, 16, 30, 66)],
                    flags=4)


# pairings whose families near R / 2, so that searches go to the whole block
@pytest.mark.parametrize("R", [40, 200, 1000, 1500])
def test_wang_large_families(R):
    b = np.array([0.0, 0.3, 0.9, 1.2, 1.4])
    _against_oracle([W.RunDesc(8, W.EA_PMJ, R, 1, b, seed=7, run_id=k, disorder_id=k, overlap=W.Q_WANG)
                     for k in range(6)])


# one or a few large populations, split over more CTAs than many of them would be, with a
# population too small to split beside them
@pytest.mark.parametrize("sizes", [[4096], [4097], [9001], [20000, 3], [40000, 17000, 60]])
def test_split_populations(sizes):
    b = W.schedule(0.6, 4)
    _against_oracle([W.RunDesc(6, W.EA_PMJ if k else W.FERRO, R, 1, b, seed=8, run_id=k) for k, R in enumerate(sizes)])


# weighted overlap distributions: more runs than a CTA stages at once, histograms that end inside a
# piece, runs without pairs at some steps; 1e-12 relative, as every weighted average
@pytest.mark.parametrize("M,L", [(1, 8), (7, 12), (256, 8), (300, 10), (513, 4)])
def test_weighted_overlap_distributions(M, L):
    rng = np.random.default_rng(M)
    N, n = L * L, 5
    rec = np.zeros((M, n), dtype=_lib.RECORD_DTYPE)
    rec["beta"] = np.linspace(0.0, 0.4, n)
    rec["lnQ"] = rng.normal(0.3, 0.05, (M, n))
    rec["minus_betaF"] = N * np.log(2.0) + np.cumsum(rec["lnQ"], axis=1)
    rec["R"], rec["R_target"], rec["N"] = rng.integers(40, 60, (M, n)), 50, N
    R = rec["R"].astype(np.int64)
    rec["sumE"], rec["sumE2"], rec["sumAbsM"], rec["sumM2"] = -20 * R, 500 * R, 6 * R, 60 * R
    for f, v in (("sumE3", 9000), ("sumE4", 400000), ("sumAbsM3", 700), ("sumM4", 9000)):
        rec[f][..., 0] = v * R
    rec["n_q"] = rng.integers(0, 30, (M, n))
    rec["n_q_pair"] = rng.integers(0, 2, (M, n)) * 25
    rec["n_q_wang"] = rec["R"]
    qs = [rng.integers(0, 1000, (M, n, N + 1)).astype(np.uint32) for _ in range(3)]
    for q, f in zip(qs, ("n_q", "n_q_pair", "n_q_wang")):
        q[rec[f] == 0] = 0
    g = _lib.pa_weighted_average(rec, N, 0, qs[0], qs[1], qh_wang=qs[2])
    one = _lib.pa_weighted_average(rec, N, 0, None, qs[1])
    o = O.weighted_average(rec, N, 0, qs[0], qs[1], qh_wang=qs[2])
    for a, b in zip(g[1:], o[1:]):
        assert np.allclose(a, b, rtol=1e-12, atol=0)
    assert one[1] is None and np.array_equal(one[2], g[2])
    assert np.allclose(g[0]["W_minus_betaF"], o[0]["W_minus_betaF"], rtol=1e-12, atol=0)
