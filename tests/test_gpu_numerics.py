"""The library's own FP64 root, division by three and local solve against CUDA's correctly rounded operations, value by
value on the GPU: random bits, the range that solves work in, exact squares, powers of two, next to the midpoint
between two roots, and subnormal numbers."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
N = 1 << 27


@pytest.fixture(scope="module")
def lib(gpu, tmp_path_factory):
    from paper_1805_04198_gb300 import _build
    so = str(tmp_path_factory.mktemp("numerics") / "numerics.so")
    subprocess.run([_build.nvcc_path()] + _build.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                   _build.CSRC, "-o", so, os.path.join(HERE, "numerics_check.cu"), "-lcudart"], check=True)
    l = ctypes.CDLL(so)
    for f in (l.root_mismatches, l.third_mismatches, l.third_f32_mismatches, l.solve_mismatches):
        f.restype = ctypes.c_longlong
    return l


@pytest.mark.parametrize("kind", range(6))
def test_root_and_third(lib, kind):
    n, seed = ctypes.c_ulonglong(N), ctypes.c_ulonglong(1000003 * (kind + 1))
    assert lib.root_mismatches(n, seed, kind) == 0
    assert lib.third_mismatches(n, seed, kind) == 0


def test_third_of_every_float(lib):
    assert lib.third_f32_mismatches() == 0


def test_local_solve_over_the_range(lib):
    assert lib.solve_mismatches(ctypes.c_ulonglong(N), ctypes.c_ulonglong(7)) == 0
