"""List construction's single-precision search and dense fallback against the oracle, bit for bit:
even weights (the target often near a boundary), tiny, subnormal and zero weights, short lists that
are often exhausted, and rows that end inside a block of 128."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nn,beta,rho,far", [
    (33, 32, 0.0, 0.5, False), (129, 2, 2.0, 0.5, False), (1001, 32, 0.0, 0.5, False),
    (401, 9, 3.0, 0.9, True), (253, 5, 2.0, 1.0, False), (2399, 3, 2.0, 0.5, False)])
def test_lists(aco, orc_all_cores, n, nn, beta, rho, far):
    if far:
        rng = np.random.default_rng(n)
        u = np.triu(rng.integers(1 << 30, (1 << 31) - 1, (n, n)), 1).astype(np.int32)
        d = np.ascontiguousarray(u + u.T)
    else:
        d = I.clustered_instance(n, seed=n, clusters=6, sigma=300).dist
    m, iters = 20, 3 if n < 500 else 1
    ref = orc_all_cores.run(d, m, iters, 31, beta=beta, rho=rho, rule=2, nn=nn)
    with aco.Colony(d, m, seed=31, beta=beta, rho=rho) as c:
        aco.aco_set_option(c.h, aco.ACO_OPT_NN_LIST, nn)
        for _ in range(iters):
            tours, lens = aco.aco_construct_tours(c.h, n, m)
            aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    assert np.array_equal(tours, ref["tours"]) and np.array_equal(lens, ref["lens"])
    assert np.array_equal(tau, ref["tau32"])
