"""Deposits summed over runs of ants before they reach the accumulator: the allocation-free update
on tours that are not permutations (which go edge by edge) and at the edges of its launch, and the
handle's default update where runs, ants and cities end unevenly."""
import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I
from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def _expected(tours, lens, heta, tau, rho):
    """The documented arithmetic: fixed-point deposits, every rounding on its own."""
    n, m = tau.shape[0], tours.shape[0]
    dtau = (1.0 / lens.astype(np.float64)).astype(np.float32)
    shift = 62 - (m - 1).bit_length() - int(np.floor(np.log2(float(dtau.max()))))
    q = [int(float(d) * 2.0 ** shift) for d in dtau]
    acc = np.zeros((n, n), object)
    for k in range(m):
        for a, b in zip(tours[k, :-1], tours[k, 1:]):
            if 0 <= a < n and 0 <= b < n:
                acc[a, b] += q[k]
                acc[b, a] += q[k]
    dep = np.array([[np.float32(np.uint64(v)) for v in row] for row in acc], np.float32)
    dep = dep * np.float32(2.0 ** -shift)
    t = np.float32(np.float32(1) - np.float32(rho)) * tau + dep
    return t, t * heta


@pytest.mark.parametrize("n,m,odd", [(3, 1, False), (32, 5, True), (33, 700, True), (40, 21000 // 8, False),
                                     (129, 17, True), (1024, 3, False)])
def test_noalloc_tours(aco, n, m, odd):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n * m)
    tours = np.stack([rng.permutation(n) for _ in range(m)]).astype(np.int32)
    if m > 3:
        tours[m // 2:] = tours[m // 2]  # shared edges
    tours = np.concatenate([tours, tours[:, :1]], 1)
    if odd:
        tours[0, 1] = tours[0, 0]        # a city twice in a row
        tours[1, n // 2] = tours[1, 3]   # a city twice, another never
        tours[2, 5] = n + 7              # outside
        tours[3, n] = tours[3, 1]        # not closed
        tours[4, 2] = -1
    lens = rng.integers(1000, 9000, m).astype(np.int64)
    heta = rng.uniform(0, 1, (n, n)).astype(np.float32)
    tau = rng.uniform(0, 1, (n, n)).astype(np.float32)
    want_tau, want_choice = _expected(tours, lens, heta, tau, 0.5)
    d = [torch.from_numpy(x).cuda() for x in (tours, lens, heta, tau)]
    choice = torch.empty_like(d[3])
    aco.aco_update_pheromone_noalloc(n, m, *(x.data_ptr() for x in d), choice.data_ptr(), 1.0, 0.5,
                                     torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert np.array_equal(d[3].cpu().numpy(), want_tau)
    assert np.array_equal(choice.cpu().numpy(), want_choice)


# short and long runs (n m below and above 2.5e6), ants that end inside a run and a group of four
@pytest.mark.parametrize("n,m", [(3, 3), (31, 9), (100, 33), (257, 1027), (1501, 1701), (700, 4099)])
def test_default_update(aco, orc_all_cores, n, m):
    d = I.clustered_instance(n, seed=n + m, clusters=5, sigma=300).dist
    with aco.Colony(d, m, seed=29) as c:
        tau0, _ = aco.aco_get_tau0(c.h)
        tours, lens = aco.aco_construct_tours(c.h, n, m)
        aco.aco_update_pheromone(c.h)
        tau = aco.aco_get_pheromone(c.h, n)
    start = np.full((n, n), tau0, np.float32)
    np.fill_diagonal(start, 0)
    assert np.array_equal(tau, orc_all_cores.update_mirror(start, tours, lens, 0.5))
