"""State kept per device (device_once.h), against a fake of the runtime calls: kernels' shared-memory limits are set on
every device that a process uses, once, and errors are returned.  The harness is built with nvcc as host code."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1303_1377_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    out = tmp_path_factory.mktemp("devh") / "libdevh.so"
    subprocess.run([nvcc, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-Xcompiler", "-fPIC", "-O2", "-std=c++17", "-I", CSRC,
                    os.path.join(ROOT, "tests", "ml_host", "device_harness.cpp"), "-o", str(out)], check=True)
    return ctypes.CDLL(str(out))


def test_limits_are_set_on_every_device_once(lib):
    sets = lib.device_sets

    def ask(which, device, get=0, set_=0):
        n = sets()
        return lib.device_allow(which, device, 1000 + device, get, set_), sets() - n

    assert ask(0, 0) == (0, 1) and lib.device_bytes() == 1000
    assert ask(0, 0) == (0, 0)
    assert ask(0, 1) == (0, 1)  # a second device of the same process
    assert ask(1, 0) == (0, 1)  # another kernel
    assert ask(0, 0) == (0, 0) and ask(0, 1) == (0, 0)
    assert ask(0, 2, set_=1) == (1, 1)  # a failed call is reported and tried again
    assert ask(0, 2) == (0, 1) and ask(0, 2) == (0, 0)
    assert ask(0, 3, get=2) == (2, 0)
    assert ask(0, 63) == (0, 1) and ask(0, 63) == (0, 0)
    assert ask(0, 64) == (0, 1) and ask(0, 64) == (0, 1)


def test_no_kernel_state_is_set_once_per_process():
    """No function-local static of the kernels' sources keeps that a device was set up."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".inc", ".cuh")):
            with open(os.path.join(CSRC, f)) as s:
                assert not re.search(r"static (const )?bool \w+ = (\[\]|false)", s.read()), f
