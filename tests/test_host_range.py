"""Which host buffers kernels may access directly: the decision alone, on made-up ranges, compiled for the host."""
import ctypes
import os
import shutil
import subprocess

import pytest

import conftest

CSRC = os.path.join(conftest.ROOT, "paper_2410_03111_b200", "csrc")


@pytest.fixture(scope="module")
def address(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("host_range")
    src, lib = d / "t.cpp", d / "t.so"
    src.write_text('#include "host_range.cuh"\n'
                   'extern "C" uint64_t f(unsigned type, unsigned managed, uint64_t device, uint64_t start, uint64_t size,'
                   ' uint64_t host, uint64_t bytes) {\n'
                   '    return lorc_mapped_address({type, managed, device, start, size}, host, bytes);\n}\n')
    subprocess.run([cxx, "-shared", "-fPIC", "-I", CSRC, "-o", str(lib), str(src)], check=True)
    f = ctypes.CDLL(str(lib)).f
    f.restype = ctypes.c_uint64
    f.argtypes = [ctypes.c_uint] * 2 + [ctypes.c_uint64] * 5
    return lambda host, nbytes, start, size, type=1, managed=0, device=None: f(
        type, managed, host if device is None else device, start, size, host, nbytes)


def test_inside_one_range(address):
    assert address(0x10000, 4096, 0x10000, 4096) == 0x10000          # the whole of it
    assert address(0x10010, 16, 0x10000, 4096) == 0x10010
    assert address(0x10ff0, 16, 0x10000, 4096) == 0x10ff0            # its last bytes
    assert address(0x10000, 64, 0x90000, 64, device=0x90000) == 0x90000


def test_two_registrations_with_a_gap_or_side_by_side(address):
    # first page registered by itself, the buffer ends in another registration: only the first one's range counts
    assert address(0x10000, 3 * 4096, 0x10000, 4096) == 0
    assert address(0x10ff0, 32, 0x10000, 4096) == 0
    assert address(0x10000, 4096, 0x10000, 4096 - 1) == 0


def test_what_is_not_plain_pinned_host_memory(address):
    assert address(0x10000, 64, 0, 0, type=0, device=0) == 0         # pageable
    assert address(0x10000, 64, 0x10000, 4096, type=2) == 0          # device memory
    assert address(0x10000, 64, 0x10000, 4096, managed=1) == 0
    assert address(0x10000, 64, 0x10000, 4096, device=0) == 0        # pinned, not mapped
    assert address(0x10008, 64, 0x10000, 4096) == 0                  # not 16-byte aligned
    assert address(0x10000, 64, 0x20000, 4096) == 0                  # a range that does not hold the byte
    assert address(0x10000, 2 ** 64 - 16, 0x10000, 4096) == 0        # no overflow
