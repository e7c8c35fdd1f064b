"""The Eq. 1 walk with compaction under any order of its threads, on the CPU.

host_warp/walk_emulator.cpp compiles the kernel's own header for the host with a fibre per GPU
thread and a random scheduler, so a missing synchronisation between lanes shows as a wrong tour or
as lanes that part for good.  Tours are compared with the oracle's, bit for bit.
"""
import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from paper_1101_2678_gb300 import instances as I

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1101_2678_gb300", "csrc")


def _cuda_include():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def emulate(tmp_path_factory):
    if not os.path.exists(os.path.join(_cuda_include(), "cuda_runtime.h")):
        pytest.skip("needs the CUDA headers")
    tmp = tmp_path_factory.mktemp("walk")
    for f in ("aco_device.cuh", "construct_phased.cuh"):
        shutil.copy(os.path.join(CSRC, f), tmp)
    # the two PTX statements of construct.cuh
    text = open(os.path.join(CSRC, "construct.cuh")).read()
    text, a = re.subn(r'asm volatile\("bar\.sync.*?\);\n', "emu::bar_sync(bar_id, nthreads);\n",
                      text, flags=re.S)
    text, b = re.subn(r'asm volatile\(\s*"\{\\n\\t\.reg \.pred p;\\n\\t\.reg \.f32 t;.*?\(mask\)\);',
                      "{ const float t = shfl_up(x, o); if (hl >= o) x += t; }", text, flags=re.S)
    assert (a, b) == (1, 1)
    (tmp / "construct.cuh").write_text(text)
    so = tmp / "walk.so"
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I", str(tmp), "-isystem", _cuda_include(),
                    os.path.join(HERE, "host_warp", "walk_emulator.cpp"), "-o", str(so)], check=True)
    lib = C.CDLL(str(so))

    def run(c, g, h, choice, dist, ants, lane_copy, seed, schedule, stall=-1):
        n = dist.shape[0]
        tours, lens = np.zeros((ants, n + 1), np.int32), np.zeros(ants, np.int64)
        lane_copy = np.asarray(lane_copy, np.int32)
        counts = np.zeros(4, np.int32)
        p = lambda x: x.ctypes.data_as(C.c_void_p)  # noqa: E731
        rc = lib.emulate_walk(c, g, h, n, ants, p(lane_copy), p(choice), p(dist),
                              C.c_ulonglong(seed), schedule, stall, p(tours), p(lens), p(counts))
        return rc, tours, lens, counts
    return run


def _instance(orc, n, beta=2.0):
    dist = np.ascontiguousarray(I.clustered_instance(n, seed=n, clusters=5, sigma=300).dist, np.int32)
    heta = orc.heta(dist, beta)
    tau = np.full((n, n), orc.tau0(dist, n), np.float32)
    np.fill_diagonal(tau, 0)
    return dist, np.ascontiguousarray(orc.choice(tau, heta, 1.0))


# every group shape that compacts, sizes that start in the direct and in a listed phase; even
# weights (beta = 0) send steps to the integer roulette
@pytest.mark.parametrize("c,g,h,n", [(36, 1, 32, 450), (36, 1, 32, 61), (36, 1, 16, 230),
                                     (36, 1, 8, 150), (36, 2, 32, 850), (76, 1, 32, 700),
                                     (12, 1, 32, 100)])
@pytest.mark.parametrize("beta", [2.0, 0.0])
@pytest.mark.parametrize("lane_copy", [0, 1])
def test_walk_in_any_order(orc, emulate, c, g, h, n, beta, lane_copy):
    dist, choice = _instance(orc, n, beta)
    ants = 32 // h + 1
    want = orc.construct(choice, dist, ants, seed=5, iteration=0)
    rc, tours, lens, counts = emulate(c, g, h, choice, dist, ants, [lane_copy] * 2, 5, n)
    assert rc == 0 and counts[2] == 0
    assert np.array_equal(tours, want[0]) and np.array_equal(lens, want[1])


# A persistent launch builds one ant after another in the same shared memory, and classes may
# differ in their row staging: every thread that copied rows itself has to fence its writes before
# the copy engine writes there.
@pytest.mark.parametrize("c,g,h,n", [(36, 1, 32, 120), (12, 1, 32, 100), (36, 1, 8, 90),
                                     (36, 2, 32, 200)])
def test_bulk_copy_after_lane_copies_is_fenced(orc, emulate, c, g, h, n):
    dist, choice = _instance(orc, n)
    ants = 2 * (32 // h)
    want = orc.construct(choice, dist, ants, seed=9, iteration=0)
    rc, tours, lens, counts = emulate(c, g, h, choice, dist, ants, [1, 0], 9, n)
    assert rc == 0 and np.array_equal(tours, want[0]) and np.array_equal(lens, want[1])
    assert counts[0] == 0 and counts[2] == 0


# A copy that never arrives: the wait gives up and the status says so; no copy is issued after it
# (the shared memory goes away at the CTA's end), and the tour is still one.
@pytest.mark.parametrize("c,g,h,n", [(36, 1, 32, 450), (36, 1, 8, 90), (36, 2, 32, 200),
                                     (12, 1, 32, 100)])
def test_no_copies_after_a_wait_gave_up(orc, emulate, c, g, h, n):
    dist, choice = _instance(orc, n)
    ants = 32 // h
    rc, tours, _, counts = emulate(c, g, h, choice, dist, ants, [0], 7, n, stall=n // 2)
    assert rc == 0 and counts[2] == 1
    assert counts[1] == 0
    assert all(sorted(t[:-1]) == list(range(n)) and t[-1] == t[0] for t in tours)


# A persistent launch initialises a barrier in the same place for ant after ant: each has to be
# invalidated first.
@pytest.mark.parametrize("c,g,h,n", [(36, 1, 32, 120), (12, 1, 32, 100), (36, 1, 8, 90),
                                     (36, 2, 32, 200)])
def test_barriers_end_with_their_ant(orc, emulate, c, g, h, n):
    dist, choice = _instance(orc, n)
    ants = 3 * (32 // h)
    want = orc.construct(choice, dist, ants, seed=11, iteration=0)
    rc, tours, _, counts = emulate(c, g, h, choice, dist, ants, [0, 0, 0], 11, n)
    assert rc == 0 and np.array_equal(tours, want[0])
    assert counts[2] == 0 and counts[3] == 0
