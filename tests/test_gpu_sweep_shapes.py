"""The bit-sliced sweeps' launch shapes against the general byte-plane sweep, bit
for bit: one and several tiles per CTA, CTAs that span runs of other sizes,
models and sweep counts, shared Philox parts from a table longer and shorter
than the schedule, and more threads than a population fills."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GENERIC, NO_TUNE, SEPARATE = 1, 2, 4


def _same(descs, flags, steps):
    with _lib.Engine(descs, flags=flags | SEPARATE) as a, _lib.Engine(descs, flags=GENERIC) as b:
        ids = np.arange(len(descs), dtype=np.uint32)
        for _ in range(steps):
            a.step(1, False)
            b.step(1, False)
            assert np.array_equal(a.step_records(ids), b.step_records(ids))
        for k in {0, 1, len(descs) // 2, len(descs) - 1}:
            for x, y in zip(a.population(k), b.population(k)):
                assert np.array_equal(x, y), k


def _mixed(L, runs, thetas, temps, R=3):
    b = W.schedule(0.9, temps)
    return [W.RunDesc(L, W.EA_PMJ if k % 3 == 1 else W.FERRO, R + (k * 7) % 40, thetas[k % len(thetas)], b, seed=5,
                      run_id=k, disorder_id=k) for k in range(runs)]


# several tiles per CTA: more than 2432 (compact rows: 4864) tiles of a launch per tile of K
@pytest.mark.parametrize("L,runs", [(8, 5000), (16, 2600), (32, 700), (64, 150), (128, 80), (256, 60),
                                    (6, 10000), (10, 10000), (30, 2600), (46, 1400), (100, 140)])
def test_several_tiles_per_cta(L, runs):
    _same(_mixed(L, runs, (1, 0, 3, 2, 4), 3), NO_TUNE, 2)


# theta above the table's half-sweeps (40, 20, 8 at L = 8, 16, 32), and one below
@pytest.mark.parametrize("L", [8, 16, 32])
def test_table_refills(L):
    _same(_mixed(L, 9, (25, 5, 11), 4), NO_TUNE, 3)
    # a CTA of several tiles whose table is refilled within a tile
    _same(_mixed(L, {8: 5000, 16: 2600, 32: 700}[L], (4,), 2), NO_TUNE, 1)


# every candidate shape takes a step while the tuner times them
@pytest.mark.parametrize("L", [4, 6, 8, 10, 12, 14, 18, 22, 26, 34, 62, 64, 66, 90, 126, 128, 206, 254, 256])
def test_every_shape(L):
    _same(_mixed(L, 5, (6, 1, 9), 12, R=1), 0, 11)
