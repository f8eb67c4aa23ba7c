"""Shared-memory limits are raised once on every device of the process (csrc/smem_limit.cuh, built for the host
against a fake runtime), and every launcher goes through that header."""
import ctypes
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2205_09104_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    out = tmp_path_factory.mktemp("smem") / "libsmem_limit_host.so"
    cuda_inc = os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda_inc,
                           os.path.join(HERE, "smem_limit_host_harness.cpp"), "-o", str(out)])
    return ctypes.CDLL(str(out))


def test_once_per_device(lib):
    def raise_on(dev, fail=0):
        calls, last = ctypes.c_int(), ctypes.c_int()
        rc = lib.host_raise(dev, 55296, fail, ctypes.byref(calls), ctypes.byref(last))
        assert last.value in (0, 55296)
        return rc, calls.value

    assert raise_on(0) == (0, 1)
    assert raise_on(0) == (0, 1)
    assert raise_on(3) == (0, 2)          # another device of the process
    assert raise_on(0) == (0, 2)
    assert raise_on(5, fail=1)[0] != 0    # a failure is reported and tried again
    assert raise_on(5) == (0, 4)
    assert raise_on(5) == (0, 4)
    assert raise_on(64) == (0, 5) and raise_on(64) == (0, 6)  # beyond the record: every time


def test_every_launcher_uses_it():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if name != "smem_limit.cuh":
            assert not re.search(r"cudaFuncSetAttribute\s*\(", text), name
