"""The field transport's bit-level arithmetic on the GPU, bit for bit against
the native operations: the float division by a length near 1 (emt_unit.cuh,
with the hardware's estimate) for every squared length of its range, the
float -> double conversion for every float, and the integer conversion, the
ceiling and the ordered keys (emt_device.cuh) over their ranges."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib():
    out_dir = os.path.join(HERE, "_build")
    os.makedirs(out_dir, exist_ok=True)
    so = os.path.join(out_dir, "libbits_check.so")
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-o", so, os.path.join(HERE, "csrc", "bits_gpu.cu")])
    L = ctypes.CDLL(so)
    L.bits_check.argtypes = [ctypes.c_int, ctypes.c_void_p]
    return L


@pytest.mark.parametrize("which,at_least", [("unit division", 9e7), ("widen", 2 ** 32), ("rest", 6e6)])
def test_bit_level_arithmetic_equals_native(lib, which, at_least):
    counts = np.zeros(2, np.uint64)
    assert lib.bits_check(["unit division", "widen", "rest"].index(which), counts.ctypes.data) == 0
    assert counts[0] >= at_least and counts[1] == 0, counts
