"""When an operator's digit copy is built, refused, kept and given back (csrc/dig_store.cu, built for the host against
a fake runtime)."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
UNDECIDED, DIGITS, ASKED, MEMORY = 0, 1, 2, 3


@pytest.fixture
def lib(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    out = tmp_path / "libdig_store_host.so"
    cuda_inc = os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include"
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda_inc,
                           os.path.join(HERE, "dig_store_host_harness.cpp"), "-o", str(out)])
    L = ctypes.CDLL(str(out))
    vp, sz = ctypes.c_void_p, ctypes.c_size_t
    L.host_device.argtypes = [sz, ctypes.c_int, ctypes.c_int, ctypes.c_int]
    L.host_used.restype = sz
    L.host_store.restype = L.host_use.restype = vp
    L.host_use.argtypes = L.host_refill.argtypes = [vp, sz]
    L.host_alloc.argtypes = [sz]
    for f in ("host_delete", "host_retry", "host_path", "host_has", "host_done"):
        getattr(L, f).argtypes = [vp]
    L.host_device(1000, 0, 0, 0)
    return L


def call(L, st, size):
    """One FP64 stencil: whether it goes through digits."""
    u = L.host_use(st, size)
    has = L.host_has(u)
    L.host_done(u)
    return bool(has)


def test_built_on_first_use_and_freed(lib):
    st = lib.host_store(0, 0)
    assert lib.host_path(st) == UNDECIDED and lib.host_used() == 0
    assert lib.host_refill(st, 200) == 0 and lib.host_packs() == 0  # blocks change before any use: nothing to do
    assert call(lib, st, 200) and call(lib, st, 200)
    assert lib.host_path(st) == DIGITS and lib.host_used() == 200 and lib.host_packs() == 1
    lib.host_refill(st, 200)
    assert lib.host_packs() == 2
    lib.host_delete(st)
    assert lib.host_used() == 0


def test_left_out(lib):
    st = lib.host_store(0, 1)
    assert not call(lib, st, 100) and lib.host_path(st) == ASKED and lib.host_used() == 0
    lib.host_retry(st)
    assert not call(lib, st, 100)


def test_at_most_a_quarter_of_the_memory(lib):
    a, b, c = (lib.host_store(0, 0) for _ in range(3))
    assert call(lib, a, 150)
    assert not call(lib, b, 150) and lib.host_path(b) == MEMORY  # 300 of 1000
    assert call(lib, c, 100)
    lib.host_delete(a)
    assert not call(lib, b, 150)  # an operator keeps its way
    lib.host_retry(b)             # until its blocks change
    assert call(lib, b, 150) and lib.host_path(b) == DIGITS


def test_no_room(lib):
    st = lib.host_store(0, 0)
    assert lib.host_alloc(900)
    assert not call(lib, st, 200) and lib.host_path(st) == MEMORY and lib.host_used() == 900


def test_given_back_to_an_allocation_that_fails(lib):
    a, b = lib.host_store(0, 0), lib.host_store(0, 0)
    assert call(lib, a, 120) and call(lib, b, 120)
    assert lib.host_alloc(900) and lib.host_used() == 900
    assert lib.host_path(a) == MEMORY and not call(lib, b, 120)
    assert not lib.host_alloc(200)


def test_not_taken_from_calls_graphs_and_other_devices(lib):
    used, captured, other = lib.host_store(0, 0), lib.host_store(0, 0), lib.host_store(1, 0)
    assert call(lib, captured, 80) and call(lib, other, 80)
    running = lib.host_use(used, 80)
    lib.host_device(1000, 1, 0, 0)
    assert call(lib, captured, 80)  # a graph now holds its pointers
    lib.host_device(1000, 0, 0, 0)
    assert not lib.host_alloc(900)
    assert [lib.host_path(s) for s in (used, captured, other)] == [DIGITS] * 3
    lib.host_done(running)
    lib.host_device(1000, 0, 0, 1)  # the device cannot be waited for
    assert not lib.host_alloc(800)
    lib.host_device(1000, 0, 0, 0)
    assert lib.host_alloc(800)
    assert [lib.host_path(s) for s in (used, captured, other)] == [MEMORY, DIGITS, DIGITS]


def test_nothing_is_built_under_capture(lib):
    st = lib.host_store(0, 0)
    lib.host_device(1000, 1, 0, 0)
    assert not call(lib, st, 100) and lib.host_path(st) == UNDECIDED
    lib.host_device(1000, 0, 0, 0)
    assert call(lib, st, 100)
