"""Where a decode call's kernels may store their results straight to the
caller's host memory: the whole result inside one page-locked, writable range.
The decision is a function of the driver's answer about the pointer, compiled
here from the library's header and given made-up answers (no GPU)."""
import ctypes
import os
import subprocess

import pytest

from conftest import ROOT

SRC = """
#include "forest.h"
extern "C" int stores_ok(int locked, int writable, unsigned long long device, unsigned long long start,
                         unsigned long long size, unsigned long long p, unsigned long long bytes,
                         unsigned long long align) {
    tp::HostRange r;
    r.page_locked = locked, r.writable = writable, r.device = device, r.start = start, r.size = size;
    return tp::host_stores_ok(r, p, bytes, align);
}
"""
TOP = 1 << 64


@pytest.fixture(scope="module")
def ok(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_range")
    (d / "r.cpp").write_text(SRC)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", cuda, "-I",
                           os.path.join(ROOT, "paper_2508_17445_gb300", "csrc"), str(d / "r.cpp"), "-o", str(d / "r.so")])
    fn = ctypes.CDLL(str(d / "r.so")).stores_ok
    fn.argtypes = [ctypes.c_int] * 2 + [ctypes.c_ulonglong] * 6
    return lambda p, n, start=0x10000, size=0x8000, locked=1, writable=1, device=None, align=16: bool(
        fn(locked, writable, p if device is None else device, start, size, p % TOP, n, align))


def test_whole_result_inside_the_range(ok):
    assert ok(0x10000, 0x8000) and ok(0x10010, 0x7FF0) and ok(0x17FF0, 16) and ok(0x10000, 1)


@pytest.mark.parametrize("p,n", [(0x10000, 0x8001), (0x10010, 0x7FF1), (0x17FF0, 17), (0x18000, 16), (0x18010, 16),
                                 (0xFFF0, 16), (0xFFF0, 0x8000), (0x10000, TOP - 1), (TOP - 16, 32)])
def test_results_that_leave_the_range(ok, p, n):
    assert not ok(p, n)


def test_memory_that_is_not_page_locked_or_writable(ok):
    assert not ok(0x10000, 16, locked=0) and not ok(0x10000, 16, writable=0) and not ok(0x10000, 16, device=0)
    assert not ok(0x10000, 16, device=0x20008) and ok(0x10000, 16, device=0x20008, align=4)
    assert not ok(0x10000, 16, start=0, size=0)  # no range in the driver's answer
