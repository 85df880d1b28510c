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
