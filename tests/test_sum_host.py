"""The FP32 lane sums of the one-kernel Arnoldi step (sum2.cuh), run on the host: as accurate as one FP64 addition per
term, whatever the number of terms.  The harness is built with nvcc as host code."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1303_1377_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("sumh") / "libsumh.so"
    subprocess.run([nvcc, "-x", "cu", "-shared", "-Xcompiler", "-fPIC", "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", CSRC,
                    os.path.join(ROOT, "tests", "ml_host", "sum_harness.cu"), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


@pytest.mark.parametrize("cnt", [1, 31, 33, 517, 1024])
@pytest.mark.parametrize("signed", [False, True])
def test_lane_sums_lose_nothing(lib, cnt, signed):
    """Entries of 12 bits make every product exact in FP32, and a term with one product per part is exact too; the 32
    additions of a lane may then err by 32 (2^-24) of an error term of at most 32 (2^-24) of the sum: 2^-38.  Plain FP32
    sums err by up to 2^-19."""
    rng = np.random.default_rng(cnt)
    a, w = np.zeros((cnt, 4), dtype=np.float32), np.zeros((cnt, 4), dtype=np.float32)
    a[:, 0] = rng.integers(2048, 4096, cnt)
    w[:, :2] = rng.integers(2048, 4096, (cnt, 2))
    if signed:
        w *= rng.choice([-1, 1], w.shape)
    out = np.zeros((32, 4), dtype=np.float32)
    p = ctypes.POINTER(ctypes.c_float)
    lib.sum_lane_dot(a.ctypes.data_as(p), w.ctypes.data_as(p), cnt, out.ctypes.data_as(p))
    for lane in range(32):
        t = a[lane::32, :1].astype(np.float64) * w[lane::32, :2].astype(np.float64)
        for part in range(2):
            got = float(out[lane, 2 * part]) + float(out[lane, 2 * part + 1])
            assert abs(got - t[:, part].sum()) <= 2.0**-38 * np.abs(t[:, part]).sum()
