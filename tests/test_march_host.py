"""The host side of the multi-step kernel without a GPU (march_host.cu: its launches are recorded or
answered with an error): which steps of a call it takes, what happens where the launch is not possible, and
its order of tiles, in which every tile comes after those it waits for."""
import ctypes
import os
import subprocess

import pytest

from paper_2608_23786_gb300 import build, mclbm

HERE = os.path.dirname(os.path.abspath(__file__))
INVALID_CONFIGURATION, COOPERATIVE_TOO_LARGE, LAUNCH_FAILURE = 9, 720, 719


@pytest.fixture(scope="module", params=[19, 27])
def host(request, tmp_path_factory):
    out = os.path.join(tmp_path_factory.mktemp("march"), f"host{request.param}.so")
    cmd = [build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-shared", "-Xcompiler", "-fPIC",
           *(["-DMCLBM_D3Q27"] if request.param == 27 else []), os.path.join(HERE, "march_host.cu"), "-o", out]
    subprocess.run(cmd, check=True, capture_output=True)
    lib = ctypes.CDLL(out)
    lib.take.restype = ctypes.c_int64
    lib.take.argtypes = [ctypes.c_int] * 4 + [ctypes.c_int64, ctypes.c_int, ctypes.c_int64, ctypes.c_int]
    lib.order.argtypes = [ctypes.c_int] * 3 + [ctypes.c_int64]
    return lib


@pytest.mark.parametrize("answer", [INVALID_CONFIGURATION, COOPERATIVE_TOO_LARGE])
@pytest.mark.parametrize("pattern", [mclbm.PULL, mclbm.AA])
def test_a_launch_that_is_not_possible_leaves_the_steps_to_single_launches(host, answer, pattern):
    """Too many blocks for the part of the GPU that is there; a build with another number of registers
    than the kernel's split needs (-G, another compiler)."""
    for precision, N in ((mclbm.FP32, 64), (mclbm.FP16, 32), (mclbm.FP64, 32)):
        assert host.take(N, 2, precision, pattern, 20, answer, 0, 0) == 0
        assert host.take(N, 2, precision, pattern, 20, 0, 0, 0) == 20


def test_other_errors_are_returned(host):
    assert host.take(64, 2, mclbm.FP32, mclbm.PULL, 20, LAUNCH_FAILURE, 0, 0) == -LAUNCH_FAILURE


def _launches(host):
    buf = (ctypes.c_int64 * (5 * 4096))()
    n = host.launches(buf, 4096)
    return [tuple(buf[5 * k:5 * k + 5]) for k in range(min(n, 4096))]


# measured microseconds of a step
@pytest.mark.parametrize("precision,N,M,us", [
    (mclbm.FP32, 8, 1, 2.6), (mclbm.FP32, 32, 1, 2.9), (mclbm.FP32, 64, 64, 271.0), (mclbm.FP32, 256, 8, 2700.0),
    (mclbm.FP16, 8, 1, 2.4), (mclbm.FP16, 64, 2, 12.9), (mclbm.FP64, 8, 1, 13.9), (mclbm.FP64, 32, 16, 312.0)])
@pytest.mark.parametrize("pattern", [mclbm.PULL, mclbm.AA])
def test_a_launch_takes_about_a_second_at_most(host, precision, N, M, us, pattern):
    steps = int(4e6 / us) & ~1  # four seconds
    assert host.take(N, M, precision, pattern, steps, 0, 0, 0) == steps
    taken = [k for k, *_ in _launches(host)]
    assert sum(taken) == steps and 4 <= len(taken) <= 20
    assert max(taken) * us <= 1.2e6


@pytest.mark.parametrize("limit,want", [(0, [26]), (1, []), (2, [2] * 13), (7, [6, 6, 6, 6, 2]), (12, [12, 12, 2]),
                                        (26, [26]), (100, [26])])
@pytest.mark.parametrize("pattern,nsteps", [(mclbm.PULL, 26), (mclbm.PULL, 27), (mclbm.AA, 26)])
def test_the_limit_splits_a_call(host, limit, want, pattern, nsteps):
    assert host.take(32, 7, mclbm.FP32, pattern, nsteps, 0, limit, 0) == sum(want)
    got = _launches(host)
    assert [k for k, *_ in got] == want
    # in place, in the lattice of the state; pull lattices start with the odd-type step
    assert {(dst, par) for _, _, dst, par, _ in got} <= {(1 << 40, 0 if pattern == mclbm.AA else 1)}


@pytest.mark.parametrize("limit", [0, 8])
def test_a_split_trajectory_goes_on_where_it_stopped(host, limit):
    assert host.take(32, 7, mclbm.FP32, mclbm.PULL, 20, 0, limit, 1) == 20
    hop = 4 * host.velocities() * 32**3 * 7
    at = 0
    for k, src, dst, _, _ in _launches(host):
        assert dst == (1 << 40) + at * hop
        assert src == (1 << 39 if at == 0 else dst - hop)
        at += k
    assert at == 20


# planes of several tiles and tiles of several planes, ensembles within L2 and windows of 2 to 12 steps,
# one sample, odd counts
@pytest.mark.parametrize("precision,N,M,steps", [
    (mclbm.FP32, 8, 1, 20), (mclbm.FP32, 8, 5, 13), (mclbm.FP32, 16, 3, 12), (mclbm.FP32, 32, 1, 12),
    (mclbm.FP32, 32, 7, 13), (mclbm.FP32, 32, 40, 9), (mclbm.FP32, 64, 1, 6), (mclbm.FP32, 64, 4, 3),
    (mclbm.FP32, 64, 9, 23), (mclbm.FP32, 128, 2, 7), (mclbm.FP32, 128, 3, 50), (mclbm.FP32, 256, 1, 5),
    (mclbm.FP16, 8, 1, 7), (mclbm.FP16, 32, 7, 9), (mclbm.FP16, 64, 3, 13), (mclbm.FP16, 128, 1, 12),
    (mclbm.FP64, 8, 1, 16), (mclbm.FP64, 16, 3, 17), (mclbm.FP64, 32, 1, 17), (mclbm.FP64, 32, 16, 8)])
def test_every_tile_comes_after_the_tiles_it_waits_for(host, precision, N, M, steps):
    assert host.order(N, M, precision, steps) == 0
