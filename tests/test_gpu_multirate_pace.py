"""Multi-rate steps by the model of one iteration's time: beside a long instance a short one keeps
most of its own pace, and the long one's step is not stretched by the short one's iterations."""
import time

import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _step_time(aco, kinds, multirate):
    """Median seconds per step, and the slots' rates."""
    ms = [10 if "acs" in k else n for k, n in kinds]
    p = aco.aco_pool_create(len(kinds), sum(aco.aco_pool_bytes_needed(n, m)
                                            for (_, n), m in zip(kinds, ms)) + (1 << 20))
    try:
        aco.aco_pool_set_multirate(p, multirate)
        slots = []
        for (kind, n), m in zip(kinds, ms):
            d = I.uniform_instance(n, 1000 if n < 500 else 10000, seed=n).dist
            s = aco.aco_pool_admit(p, d, 1.0, 2.0, 0.1, m, 5, 5000)
            if "acs" in kind:
                aco.aco_pool_set_acs(p, s, 0.9, 0.1)
            if "nn" in kind:
                aco.aco_pool_set_nn(p, s, 20)
            slots.append(s)
        t = []
        for _ in range(13):
            aco.aco_pool_synchronize(p)
            t0 = time.perf_counter()
            aco.aco_pool_step(p)
            aco.aco_pool_synchronize(p)
            t.append(time.perf_counter() - t0)
        return float(np.median(t)), [aco.aco_pool_rate(p, s) for s in slots]
    finally:
        aco.aco_pool_destroy(p)


# The model's ratios are within 10 % of the measured ones at these sizes, a rate rounds down (at
# most by 1 / 5 here), and the two groups slow each other little: they share no SM.  (With the
# times of earlier kernels the first long step took 2.5 of its time alone and the second short
# instance ran at 0.44 of its pace.)
@pytest.mark.parametrize("long,short", [(("acs", 1002), ("as", 100)), (("as", 1002), ("acs", 100)),
                                        (("acs nn", 1002), ("nn", 100)), (("as", 1500), ("nn", 200))])
def test_pace(aco, long, short):
    alone_long, _ = _step_time(aco, [long], False)
    alone_short, _ = _step_time(aco, [short], False)
    both, rates = _step_time(aco, [long, short], True)
    assert rates[0] == 1 and rates[1] > 1
    assert both <= 1.5 * alone_long, (both, alone_long, rates)
    assert rates[1] * alone_short >= 0.6 * both, (both, alone_short, rates)
