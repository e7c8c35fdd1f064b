"""The walk at the edge of compaction (chunks of 28 cities walk the whole row, of 36 list the
unvisited ones) for one and two warps and for segments of 16 and 8 lanes, with both row stagings:
tours and trails equal the oracle's, bit for bit."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,warps,lanes", [(896, 1, 32), (897, 1, 32), (1792, 2, 32), (1793, 2, 32),
                                           (448, 1, 16), (449, 1, 16), (224, 1, 8), (225, 1, 8)])
@pytest.mark.parametrize("stage", [0, 1])
def test_last_without_and_first_with_lists(aco, orc_all_cores, n, warps, lanes, stage):
    d = I.clustered_instance(n, seed=n + lanes, clusters=9, sigma=400).dist
    m = 33
    ref = orc_all_cores.run(d, m, 2, 17)
    with aco.Colony(d, m, seed=17) as c:
        aco.aco_set_option(c.h, aco.ACO_OPT_WARPS_PER_ANT, warps)
        aco.aco_set_option(c.h, aco.ACO_OPT_LANES_PER_ANT, lanes)
        aco.aco_set_option(c.h, aco.ACO_OPT_STAGING, stage)
        for _ in range(2):
            tours, lens = aco.aco_construct_tours(c.h, n, m)
            aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    assert np.array_equal(tours, ref["tours"]) and np.array_equal(lens, ref["lens"])
    assert np.array_equal(tau, ref["tau32"])
