"""Construction with the whole matrix in shared memory (default tiling, n <= 240) against the
oracle, bit for bit: the smallest and largest n, both chunk widths, ragged rows, ants that leave
warps of the last CTA idle, and weights at which the integer roulette decides."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def _check(aco, orc, d, m, iters, beta, rho):
    n = d.shape[0]
    ref = orc.run(d, m, iters, 23, beta=beta, rho=rho)
    with aco.Colony(d, m, seed=23, beta=beta, rho=rho) as c:
        for _ in range(iters):
            tours, lens = aco.aco_construct_tours(c.h, n, m)
            aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    assert np.array_equal(tours, ref["tours"]) and np.array_equal(lens, ref["lens"])
    assert np.array_equal(tau, ref["tau32"])


@pytest.mark.parametrize("n,m", [(3, 1), (4, 7), (33, 153), (127, 9), (128, 1000), (129, 5),
                                 (238, 300), (239, 33), (240, 4871), (241, 40)])
def test_sizes(aco, orc_all_cores, n, m):
    _check(aco, orc_all_cores, I.clustered_instance(n, seed=n, clusters=7, sigma=400).dist, m, 2,
           2.0, 0.5)


@pytest.mark.parametrize("n", [65, 240])
@pytest.mark.parametrize("beta,rho", [(0.0, 0.5), (3.0, 0.9), (2.0, 1.0)])
def test_even_tiny_and_zero_weights(aco, orc_all_cores, n, beta, rho):
    rng = np.random.default_rng(n)
    u = np.triu(rng.integers(1 << 30, (1 << 31) - 1, (n, n)), 1).astype(np.int32)
    _check(aco, orc_all_cores, np.ascontiguousarray(u + u.T), 20, 4, beta, rho)
