"""The walk's single-precision search against the oracle where it may not decide.

The float search takes a city only when the target lies inside the city's
interval by more than its error bound; otherwise the step runs the integer
roulette.  Everything is bit-exact, so no tolerance is involved.
"""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def _run_both(aco, orc, dist, m, iters, beta, rho, warps, lanes):
    n = dist.shape[0]
    ref = orc.run(dist, m, iters, 13, beta=beta, rho=rho)
    with aco.Colony(dist, m, seed=13, beta=beta, rho=rho) as c:
        aco.aco_set_option(c.h, aco.ACO_OPT_WARPS_PER_ANT, warps)
        aco.aco_set_option(c.h, aco.ACO_OPT_LANES_PER_ANT, lanes)
        for it in range(iters):
            tours, lens = aco.aco_construct_tours(c.h, n, m)
            aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    assert np.array_equal(tours, ref["tours"]) and np.array_equal(lens, ref["lens"])
    assert np.array_equal(tau, ref["tau32"])


# Equal weights (beta = 0): n boundaries spread evenly, so the target falls
# within the error bound of one of them at about 1 % of the steps of large n.
@pytest.mark.parametrize("n,warps,lanes", [(385, 1, 32), (1001, 1, 32), (2432, 1, 32),
                                           (2433, 2, 32), (4093, 2, 32), (701, 1, 16),
                                           (397, 1, 8)])
def test_even_weights(aco, orc_all_cores, n, warps, lanes):
    d = I.uniform_instance(n, 10000, seed=n).dist
    _run_both(aco, orc_all_cores, d, 24, 1, 0.0, 0.5, warps, lanes)


# Distances near 2^31 and beta = 3: the weights start near 2^-124, their sums
# on both sides of 2^-120 (below which the float search steps aside), and the
# second iteration's (rho = 0.9) are subnormal or zero.
@pytest.mark.parametrize("n,warps,lanes", [(401, 1, 32), (1003, 1, 32), (2433, 2, 32), (601, 1, 8)])
def test_tiny_weights(aco, orc_all_cores, n, warps, lanes):
    rng = np.random.default_rng(n)
    u = np.triu(rng.integers(1 << 30, (1 << 31) - 1, (n, n)), 1).astype(np.int32)
    _run_both(aco, orc_all_cores, np.ascontiguousarray(u + u.T), 16, 2, 3.0, 0.9, warps, lanes)
