"""One persistent construction launch whose classes stage their rows differently: every resident
warp builds ants of several classes, rows by lane copies and by bulk copies in the same shared
memory, and each instance ends as when run alone."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco  # noqa: F401  (fixture)
from test_gpu_pool import alone

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [0, 1])
def test_staging_by_class(aco, first):
    ns = [1000, 800, 517, 300, 100]
    ms = [2000] * len(ns)  # more ants than the launch has warps (8 CTAs of 4 on each SM)
    insts = [I.uniform_instance(n, 1000, seed=900 + n) for n in ns]
    b = aco.aco_batch_create([x.dist for x in insts], ms, [3, 4, 5, 6, 7])
    try:
        widths = (36, 28, 20, 12, 4)
        aco.aco_pool_set_tuning(b, [[[1, 32, c], [1, 32, 4, (first + i) % 2]]
                                    for i, c in enumerate(widths)])
        aco.aco_pool_set_single_launch(b, True)
        aco.aco_batch_iterate(b, 2)
        assert [aco.aco_pool_tiling(b, i)[2:] for i in range(len(ns))] == \
            [(c, (first + i) % 2) for i, c in enumerate(widths)]
        for i, x in enumerate(insts):
            tau_a, (tour_a, len_a) = alone(aco, x.dist, ms[i], 3 + i, 2)
            tour_b, len_b = aco.aco_batch_best(b, i, x.n)
            assert len_b == len_a and np.array_equal(tour_b, tour_a), i
            assert np.array_equal(aco.aco_pool_pheromone(b, i, x.n), tau_a), i
    finally:
        aco.aco_batch_destroy(b)
