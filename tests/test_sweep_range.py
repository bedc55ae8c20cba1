"""The fixed-point sweeps (csrc/amrfd_sweep.cuh) at the ends of their range, on the CPU: wide
sums, windows of far more than 110 bits, cells that are exactly equal."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1407_2052_gb300", "csrc")

HARNESS = """
#include "amrfd_sweep.cuh"
using namespace amrfd;
extern "C" double wide(long long hi, unsigned long long lo) {
  return wide_double((__int128)(((unsigned __int128)(unsigned long long)hi << 64) | lo));
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("range")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run([gxx, "-O1", "-std=gnu++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    L.wide.restype, L.wide.argtypes = ctypes.c_double, [ctypes.c_longlong, ctypes.c_ulonglong]
    return L


@pytest.mark.parametrize("bits", [53, 54, 95, 96, 97, 120, 121, 122, 123, 124, 125])
def test_wide_sums_round_once(lib, bits):
    """Whole numbers of `bits` bits, near ties of the conversion among them."""
    rng = np.random.default_rng(bits)
    for _ in range(2000):
        a = (1 << (bits - 1)) | int(rng.integers(0, 1 << 52)) << max(0, bits - 53)
        a += (1 << max(0, bits - 54)) + int(rng.integers(-2, 3))  # half a unit in the last place, about
        a = min(a, (1 << bits) - 1) * int(rng.choice((-1, 1)))
        assert lib.wide(a >> 64, a & (2 ** 64 - 1)) == float(Fraction(a)), a
