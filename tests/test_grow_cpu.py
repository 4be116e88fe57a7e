"""Per-molecule scratch of a handle after a failed allocation: every region still lies inside the buffer it belongs to.
The host code is compiled with a fake allocator that fails when told to."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdlib>
#include "jk_grow.h"
static long fail_after, live;
static int fake_alloc(size_t bytes, void **p)
{
    if (fail_after-- == 0) return 2;
    *p = std::malloc(bytes);
    ++live;
    return 0;
}
static void fake_free(void *p) { if (p) --live; std::free(p); }
static JkPerMol<double> buf;
extern "C" {
int grow(size_t n, size_t total, long fail) { fail_after = fail; return buf.grow(n, total, fake_alloc, fake_free); }
size_t held() { return buf.ndm; }
long allocations() { return live; }
long long offset(size_t unit) { return buf.base ? (long long)(buf.at(unit) - buf.base) : -1; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("grow")
    (d / "g.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2507_09772_gb300", "csrc"),
                    str(d / "g.cpp"), "-o", str(d / "g.so")], check=True)
    g = ctypes.CDLL(str(d / "g.so"))
    g.grow.argtypes = [ctypes.c_size_t, ctypes.c_size_t, ctypes.c_long]
    g.held.restype = ctypes.c_size_t
    g.offset.argtypes, g.offset.restype = [ctypes.c_size_t], ctypes.c_longlong
    return g


def test_regions_stay_inside_the_buffer_they_belong_to(lib):
    nao = np.array([5, 40, 3, 17])
    unit = np.concatenate([[0], np.cumsum(nao ** 2)])
    total = int(unit[-1])

    def build(ndm, fail=-1):
        """A call with ndm densities: grow where needed, then place every molecule."""
        rc = lib.grow(ndm, total, fail)
        if rc:
            return rc
        n = lib.held()
        assert n >= ndm
        end = 0
        for m in range(len(nao)):
            o = lib.offset(int(unit[m]))
            assert o >= end                          # regions do not overlap
            end = o + ndm * int(nao[m]) ** 2
        assert end <= n * total                      # nor leave the allocation
        return 0

    assert build(1) == 0 and build(2) == 0 and build(1) == 0
    assert build(4, fail=0) == 2                     # the growth fails
    assert lib.held() == 0 and lib.offset(0) == -1 and lib.allocations() == 0   # and leaves nothing behind
    assert build(1) == 0 and lib.held() == 1         # the next call allocates again
    assert build(3) == 0 and build(2) == 0 and lib.allocations() == 1
