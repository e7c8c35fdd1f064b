"""The Ant Colony System kernel that keeps rows in registers, against the oracle, where its
parts meet: sizes around whole blocks of 128 cities and around the widths compiled, ant counts
on both sides of the rows that fit, even and tiny weights (the integer roulette decides)."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _check(aco, orc, dist, m, iters, beta, q0):
    n = dist.shape[0]
    ref = orc.run_acs(dist, m, iters, 17, beta=beta, q0=q0)
    h = aco.aco_create(dist, 1.0, beta, 0.1, m, 17)
    try:
        aco.aco_set_acs(h, q0, 0.1)
        aco.aco_iterate(h, iters)
        tau = aco.aco_get_pheromone(h, n)
        tour, best = aco.aco_best_tour(h, n)
    finally:
        aco.aco_destroy(h)
    assert np.array_equal(tau, ref["tau32"])
    assert best == ref["best_len"] and np.array_equal(tour, ref["best_tour"])


@pytest.mark.parametrize("n,m", [(3, 2), (4, 4), (127, 10), (128, 10), (129, 32), (256, 7), (257, 10),
                                 (512, 32), (513, 16), (513, 17), (769, 10), (1024, 16), (1025, 10),
                                 (1025, 11), (2049, 10), (3073, 3)])
def test_block_edges(aco, orc, n, m):
    _check(aco, orc, I.clustered_instance(n, seed=n, clusters=9, sigma=500).dist, m,
           1 if n > 1000 else 3, 2.0, 0.6)


# beta = 0 leaves equal weights (boundaries everywhere); distances near 2^31 and beta = 3 put the
# sums on both sides of 2^-120.  q0 = 0: every step explores.
@pytest.mark.parametrize("n,beta", [(140, 0.0), (1001, 0.0), (140, 3.0), (601, 3.0)])
def test_exploring_at_the_edge(aco, orc, n, beta):
    rng = np.random.default_rng(n)
    u = np.triu(rng.integers(1 << 30, (1 << 31) - 1, (n, n)), 1).astype(np.int32)
    _check(aco, orc, np.ascontiguousarray(u + u.T), 6, 2, beta, 0.0)
