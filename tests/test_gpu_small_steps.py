"""Small runs whose clusters are chosen on either side of the rule's lines, in one
launch of all temperatures and in single steps: the general sweep's anneal bit for
bit."""
import numpy as np
import pytest

from paper_2207_05535_gb300 import _lib
from paper_2207_05535_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GENERIC = 1


def _descs(L, R, theta, n=1, temps=22):
    return [W.RunDesc(L, W.EA_PMJ if k % 2 else W.FERRO, R, theta, W.schedule(0.5, temps), seed=23, run_id=k,
                      disorder_id=k) for k in range(n)]


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
