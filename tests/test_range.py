"""Which device buffers a kernel may read in place (csrc/nsli_range.h, compiled
for the host): a buffer that is shorter than what the call reads is left to
the staging copy, whose range the driver checks."""
import ctypes
import os
import subprocess

import pytest

from conftest import ROOT

CSRC = os.path.join(ROOT, "paper_2003_09956_gb300", "csrc")


@pytest.fixture(scope="module")
def covers(tmp_path_factory):
    d = tmp_path_factory.mktemp("range")
    src = d / "range.cpp"
    src.write_text('#include "nsli_range.h"\n'
                   'extern "C" int covers(std::uintptr_t b, std::size_t s, std::uintptr_t p, std::size_t n,'
                   ' std::size_t e) { return nsli::range_covers(b, s, p, n, e); }\n')
    lib = d / "range.so"
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).covers
    fn.argtypes = [ctypes.c_size_t] * 5
    return fn


BASE, TOP = 0x7f0000000000, 2 ** 64


@pytest.mark.parametrize("size,offset,count,want", [
    (8, 0, 1, 1), (8, 0, 2, 0), (15, 0, 1, 1), (15, 0, 2, 0), (800, 0, 100, 1), (800, 0, 101, 0),
    (800, 8, 99, 1), (800, 8, 100, 0), (800, 792, 1, 1), (800, 800, 0, 1), (800, 800, 1, 0), (800, 808, 1, 0),
    (800, -8, 1, 0), (0, 0, 1, 0), (1 << 40, 0, 1 << 37, 1), (1 << 40, 0, (1 << 37) + 1, 0),
    (800, 0, TOP // 8, 0), (800, 0, TOP // 8 + 1, 0), (800, 0, TOP - 1, 0)])
def test_range(covers, size, offset, count, want):
    assert covers(BASE, size, BASE + offset, count, 8) == want
