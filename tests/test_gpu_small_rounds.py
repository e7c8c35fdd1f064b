"""The kernel that holds the whole matrix in shared memory near its largest n, where few warps fit
beside the matrix: bits when the ants take two rounds, and no slower than the walk with many ants."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)
from test_gpu_small import _check

pytestmark = pytest.mark.gpu


# one ant more than a round holds, uneven last rounds, the most ants of two rounds, one more
@pytest.mark.parametrize("n,m", [(240, 305), (240, 608), (240, 609), (239, 1000), (238, 1824),
                                 (237, 2433), (236, 4871), (128, 4865), (60, 9000)])
def test_rounds(aco, orc_all_cores, n, m):
    _check(aco, orc_all_cores, I.clustered_instance(n, seed=n, clusters=7, sigma=400).dist, m, 1,
           2.0, 0.5)


# Median of nine event times; runs of one side differ by under 2 %.  (With as many rounds as it
# took, the kernel was 4.0 times slower than the walk at n = 240, m = 4864, and 1.6 at n = 239,
# m = 2048.)
@pytest.mark.parametrize("n,m", [(240, 4864), (239, 2048), (237, 4864), (200, 5000), (128, 5000)])
def test_not_slower_than_the_walk(aco, n, m):
    d = I.uniform_instance(n, 1000, seed=3).dist
    ms = []
    for warps in (0, 1):  # the default, and the walk by an option that names a tiling
        with aco.Colony(d, m, seed=9) as c:
            if warps:
                aco.aco_set_option(c.h, aco.ACO_OPT_WARPS_PER_ANT, warps)
            aco.aco_set_option(c.h, aco.ACO_OPT_PROFILE, 1)
            aco.aco_iterate(c.h, 3)
            t = []
            for _ in range(9):
                aco.aco_iterate(c.h, 1)
                t.append(aco.aco_get_kernel_times(c.h)[0])
            ms.append(np.median(t))
    assert ms[0] <= 1.1 * ms[1], ms
