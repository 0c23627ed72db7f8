"""The larger radices of the line transforms (`csrc/fft_radix.cuh`), compiled for the host (no
GPU), against direct DFTs.  An R-point transform of values of size one in FP64 is off by a few
log2(R) rounding errors of the result's norm: 1e-14 of it for R <= 15."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="nvcc not available")


@pytest.fixture(scope="module")
def radix(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("hostradix") / "libradix.so")
    subprocess.run([NVCC, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-I" + os.path.join(ROOT, "paper_2601_02172_gb300", "csrc"), "-o", out,
                    os.path.join(ROOT, "tests", "host", "radix_host.cu")], check=True, capture_output=True)
    lib = C.CDLL(out)
    lib.host_radix.argtypes = [C.c_int, C.c_int, C.POINTER(C.c_double)]
    return lib


@pytest.mark.parametrize("R", [9, 10, 12, 15])
@pytest.mark.parametrize("inv", [0, 1])
def test_radix_matches_direct_dft(radix, R, inv):
    rng = np.random.default_rng(R)
    x = rng.normal(size=R) + 1j * rng.normal(size=R)
    v = np.ascontiguousarray(np.stack([x.real, x.imag], 1).ravel())
    assert radix.host_radix(R, inv, v.ctypes.data_as(C.POINTER(C.c_double))) == 1
    k = np.arange(R)
    ref = np.exp((2j if inv else -2j) * np.pi * (np.outer(k, k) % R) / R) @ x
    assert np.abs(v[0::2] + 1j * v[1::2] - ref).max() < 1e-14 * np.linalg.norm(ref)
