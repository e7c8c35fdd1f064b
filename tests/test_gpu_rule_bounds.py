"""The per-candidate rules where their bounds decide which cities are drawn for: against the
oracle, bit for bit, at one group per lane and many, with even, tiny, zero and overflowing keys."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", [1, 2])  # data-parallel, exponential race
@pytest.mark.parametrize("n,beta,rho,far", [
    (5, 2.0, 0.5, False), (128, 2.0, 0.5, False), (129, 0.0, 0.5, False), (385, 2.0, 1.0, False),
    (517, 3.0, 0.5, True), (300, 3.0, 0.9, True), (1217, 0.0, 0.5, False), (2433, 2.0, 0.5, False)])
def test_bounds(aco, orc_all_cores, rule, n, beta, rho, far):
    orc = orc_all_cores
    if far:  # weights near 2^-124, then subnormal or zero: keys overflow
        rng = np.random.default_rng(n)
        u = np.triu(rng.integers(1 << 30, (1 << 31) - 1, (n, n)), 1).astype(np.int32)
        d = np.ascontiguousarray(u + u.T)
    else:
        d = I.clustered_instance(n, seed=n + rule, clusters=8, sigma=400).dist
    m, iters = min(n, 16), 3 if n < 600 else 1
    ref = orc.run(d, m, iters, 19, beta=beta, rho=rho, rule={1: 1, 2: 3}[rule])  # the oracle numbers the race 3
    with aco.Colony(d, m, seed=19, beta=beta, rho=rho) as c:
        aco.aco_set_option(c.h, aco.ACO_OPT_SELECTION, rule)
        for _ in range(iters):
            tours, lens = aco.aco_construct_tours(c.h, n, m)
            aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    assert np.array_equal(tours, ref["tours"]) and np.array_equal(lens, ref["lens"])
    assert np.array_equal(tau, ref["tau32"])
