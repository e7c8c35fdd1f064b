"""Kernels that start before their predecessors in the stream have ended (programmatic dependent
launch): what they take as read-only, and calls that follow each other without a synchronisation,
directly and in a captured graph."""
import glob
import os
import re

import numpy as np
import pytest

from test_gpu_parity import aco, orc_all_cores  # noqa: F401  (fixtures)

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1101_2678_gb300", "csrc")


def _kernels(text):
    """(name, parameters, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void\s+(?:__\w+__\([^)]*\)\s*)?(\w+)\(([^)]*)\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), [p.strip() for p in m.group(2).split(",")], text[m.end():i]


# const ... __restrict__ promises that nobody writes the data while the kernel lives; a kernel that
# waits inside for its predecessors may not say that of what they write.
def test_no_read_only_promise_on_data_still_being_written():
    seen = 0
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        kernels = list(_kernels(open(path).read()))
        written = {p.split()[-1].lstrip("*") for _, params, _ in kernels for p in params
                   if "*" in p and "const" not in p}
        for name, params, body in kernels:
            if "grid_wait()" not in body:
                continue
            seen += 1
            for p in params:
                if "const" in p and "__restrict__" in p:
                    assert p.split()[-1].lstrip("*") not in written, (name, p)
    assert seen >= 2


def _args(torch, rng, n, m):
    tours = np.stack([rng.permutation(n) for _ in range(m)]).astype(np.int32)
    tours = np.concatenate([tours, tours[:, :1]], 1)
    lens = rng.integers(1000, 9000, m).astype(np.int64)
    up = np.triu(rng.uniform(0, 1, (n, n)).astype(np.float32), 1)
    tau, heta = up + up.T, rng.uniform(0, 1, (n, n)).astype(np.float32)
    return tours, lens, heta, tau


def _call(aco, torch, d, n, m, rho):
    aco.aco_update_pheromone_noalloc(n, m, *(x.data_ptr() for x in d), 1.0, rho,
                                     torch.cuda.current_stream().cuda_stream)


@pytest.mark.gpu
def test_calls_back_to_back(aco, orc_all_cores):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    sizes = [(300, 2000), (5, 1), (1002, 400), (64, 4096), (1024, 700), (3, 9), (257, 257)] * 3
    calls = []
    for i, (n, m) in enumerate(sizes):
        host = _args(torch, rng, n, m)
        dev = [torch.from_numpy(x).cuda() for x in host]
        dev.append(torch.empty_like(dev[3]))
        calls.append((n, m, 0.1 + 0.04 * i, host, dev))
    torch.cuda.synchronize()
    for n, m, rho, _, dev in calls:
        _call(aco, torch, dev, n, m, rho)
    torch.cuda.synchronize()
    for n, m, rho, (tours, lens, heta, tau), dev in calls:
        want = orc_all_cores.update_mirror(tau, tours, lens, rho)
        assert np.array_equal(dev[3].cpu().numpy(), want), (n, m)
        assert np.array_equal(dev[4].cpu().numpy(), want * heta), (n, m)


@pytest.mark.gpu
def test_captured_and_replayed(aco, orc_all_cores):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(6)
    sizes = [(300, 700), (1002, 64), (40, 3000)]
    host = [_args(torch, rng, n, m) for n, m in sizes]
    dev = [[torch.from_numpy(x).cuda() for x in h] for h in host]
    for d in dev:
        d.append(torch.empty_like(d[3]))
    keep = [d[3].clone() for d in dev]
    for (n, m), d in zip(sizes, dev):  # (the first call looks the scratch up)
        _call(aco, torch, d, n, m, 0.3)
    for d, k in zip(dev, keep):
        d[3].copy_(k)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for (n, m), d in zip(sizes, dev):
            _call(aco, torch, d, n, m, 0.3)
    want = [h[3] for h in host]
    for rep in range(3):
        new = [_args(torch, rng, n, m) for n, m in sizes]
        for d, h in zip(dev, new):  # other tours and lengths in the same arrays
            d[0].copy_(torch.from_numpy(h[0]))
            d[1].copy_(torch.from_numpy(h[1]))
        graph.replay()
        torch.cuda.synchronize()
        for i, h in enumerate(new):
            want[i] = orc_all_cores.update_mirror(want[i], h[0], h[1], 0.3)
            assert np.array_equal(dev[i][3].cpu().numpy(), want[i]), (rep, sizes[i])
            assert np.array_equal(dev[i][4].cpu().numpy(), want[i] * host[i][2]), (rep, sizes[i])
