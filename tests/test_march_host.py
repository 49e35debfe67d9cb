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
    lib.take.argtypes = [ctypes.c_int] * 4 + [ctypes.c_int64, ctypes.c_int]
    lib.order.argtypes = [ctypes.c_int] * 3 + [ctypes.c_int64]
    return lib


@pytest.mark.parametrize("answer", [INVALID_CONFIGURATION, COOPERATIVE_TOO_LARGE])
@pytest.mark.parametrize("pattern", [mclbm.PULL, mclbm.AA])
def test_a_launch_that_is_not_possible_leaves_the_steps_to_single_launches(host, answer, pattern):
    """Too many blocks for the part of the GPU that is there; a build with another number of registers
    than the kernel's split needs (-G, another compiler)."""
    for precision, N in ((mclbm.FP32, 64), (mclbm.FP16, 32), (mclbm.FP64, 32)):
        assert host.take(N, 2, precision, pattern, 20, answer) == 0
        assert host.take(N, 2, precision, pattern, 20, 0) == 20


def test_other_errors_are_returned(host):
    assert host.take(64, 2, mclbm.FP32, mclbm.PULL, 20, LAUNCH_FAILURE) == -LAUNCH_FAILURE


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
