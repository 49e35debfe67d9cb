"""The FP64 reciprocal of the plain collision against the correctly rounded one.  Bound: the starting value
is within 2^-20, one third-order step leaves 2^-60 of it, and the step's own roundings (e and e + e^2, both
below 2^-19, and the last fused operation) add at most 2^-72 to the last one's half unit in the last place: one
unit from the correctly rounded value, and that only within 2^-60 + 2^-72 of a tie, in at most 2^-60 / 2^-53 =
1% of the values."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2608_23786_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = os.path.join(tmp_path_factory.mktemp("rcp64"), "rcp64.so")
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler",
                    "-fPIC", os.path.join(HERE, "rcp64_check.cu"), "-o", out],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(out)
    lib.rcp64_check.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    return lib


# densities and products of populations; the normal range whose reciprocals are normal; one binade
@pytest.mark.parametrize("lo,hi", [(-12, 3), (-1000, 1000), (0, 1), (-1, 0)])
def test_within_one_unit_of_the_correctly_rounded_reciprocal(lib, lo, hi):
    n = 1 << 27
    out = torch.zeros(2, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    assert lib.rcp64_check(n, 12345, lo, hi, out.data_ptr()) == 0
    ulps, differ = out.tolist()
    print(f"exponents {lo}..{hi - 1}: largest distance {ulps}, {differ} of {n} differ")
    assert ulps <= 1 and differ <= 0.01 * n
