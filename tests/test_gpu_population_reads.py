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


# Reads of the whole population go through the buffer that the next step's children take, in up to eight
# pieces: the anneal goes on as if nothing had been read
@pytest.mark.parametrize("flags", [SEPARATE, 0, 1])
@pytest.mark.parametrize("L,R", [(6, 500), (8, 700), (16, 900), (30, 300), (64, 90), (128, 40)])
def test_whole_reads_leave_the_anneal_alone(L, R, flags):
    with _engine(L, R, flags) as eng, _engine(L, R, flags) as other:
        for n in (1, 2, 1, 3):
            eng.step(n)
            other.step(n)
            s, E, M, fam, _ = eng.population(0)
            assert np.array_equal(s.sum(axis=1, dtype=np.int64), M)
            cut = eng.checkpoint(0)
            assert cut == other.checkpoint(0)
        eng.run_to_end()
        other.run_to_end()
        assert np.array_equal(eng.records(0), other.records(0))
        for a, b in zip(eng.population(0), other.population(0)):
            assert np.array_equal(a, b)


# results of 1 MB and more: into fresh pages, into pages that hold something, into pinned memory
def test_large_results_into_pageable_and_pinned_memory():
    import ctypes as C

    import torch

    L, R, temps = 32, 3000, 40
    N = L * L
    descs = [W.RunDesc(L, W.EA_PMJ, R, 1, W.schedule(0.8, temps), seed=37, run_id=k, disorder_id=0,
                       overlap=W.Q_SHIFT | W.Q_PAIR, paired=1 - k) for k in range(2)]
    with _lib.Engine(descs) as eng:
        eng.run_to_end()
        rec, qa, qb = eng.records(0, qhist=True)
        assert qa.nbytes < 1 << 20 and np.array_equal(qa.sum(axis=1), rec["n_q"])
        s, E, M, fam, _ = eng.population(0)
        assert s.nbytes > 1 << 20
        cap = eng.runs[0].R_cap
        R_i, step = C.c_uint32(), C.c_uint32()
        for buf in (np.empty((cap, N), np.int8), np.full((cap, N), 9, np.int8),
                    torch.full((cap, N), 9, dtype=torch.int8).pin_memory().numpy()):
            _lib._check(_lib.load().pa_population(eng.h, 0, _lib._p(buf, C.c_int8), None, None, None, C.byref(R_i),
                                                  C.byref(step)), "pa_population")
            assert R_i.value == len(s) and np.array_equal(buf[:len(s)], s)
