"""Which device uploads load the caller's vertices in place: only memory of the context's own GPU at an
int2's alignment (host code, compiled alone)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3  # cudaMemoryType


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text('#include "upload.cuh"\nextern "C" int rule(int type, int at, int device, uint64_t a)\n'
                             '{ return pmh_reads_in_place(type, at, device, (uintptr_t)a); }\n')
    subprocess.run([cxx, "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2511_16576_gb300", "csrc"), str(d / "r.cpp"), "-o",
                    str(d / "r.so")], check=True)
    lib = ctypes.CDLL(str(d / "r.so"))
    return lambda t, at, dev, a: bool(lib.rule(t, at, dev, ctypes.c_uint64(a)))


@pytest.mark.parametrize("address,aligned", [(0x7F0000000000, True), (0x7F0000000008, True),
                                             (0x7F0000000004, False), (0x7F0000000001, False)])
def test_own_device_memory_only(rule, address, aligned):
    for device in (0, 1, 3):
        assert rule(DEVICE, device, device, address) == aligned
        for other in (-2, -1, 0, 1, 2, 3, 7):
            if other != device:
                assert not rule(DEVICE, other, device, address)
        for kind in (UNREGISTERED, HOST, MANAGED):
            assert not rule(kind, device, device, address)
