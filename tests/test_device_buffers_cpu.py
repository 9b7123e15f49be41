"""Whether a caller's device buffer lies whole in memory that is there (the check
that comes before a kernel reads or writes it), against made-up allocations on the
host."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
WHOLE, PIECES, SHORT, UNKNOWN = range(4)

SOURCE = r"""
#include "device_buffers.h"
extern "C" int extent(const unsigned long long* base, const unsigned long long* size, int n, unsigned long long p,
                      unsigned long long bytes) {
  return (int)brahms::extent_of((uintptr_t)p, (size_t)bytes, [&](uintptr_t a, uintptr_t* b, size_t* s) {
    for (int i = 0; i < n; ++i)
      if (a >= base[i] && a - base[i] < size[i]) {
        *b = (uintptr_t)base[i];
        *s = (size_t)size[i];
        return true;
      }
    return false;
  });
}
"""


@pytest.fixture(scope="module")
def extent(tmp_path_factory):
    d = tmp_path_factory.mktemp("extent")
    src, so = d / "extent.cpp", d / "extent.so"
    src.write_text(SOURCE)
    from paper_2609_08384_gb300 import build
    nvcc = shutil.which(build._nvcc()) or build._nvcc()
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I" + build.CSRC, "-I" + include, str(src), "-o", str(so)],
                   check=True)
    fn = ctypes.CDLL(str(so)).extent

    def call(allocations, p, size):
        u = ctypes.c_ulonglong
        n = len(allocations)
        return fn((u * n)(*[a for a, _ in allocations]), (u * n)(*[s for _, s in allocations]), n, u(p), u(size))

    return call


@pytest.mark.parametrize("allocations, p, size, want", [
    ([(4096, 4096)], 4096, 4096, WHOLE),            # the whole allocation
    ([(4096, 4096)], 4104, 4088, WHOLE),            # its end, from inside
    ([(4096, 4096)], 4104, 4096, SHORT),            # eight bytes too many
    ([(4096, 4096)], 8191, 2, SHORT),
    ([(4096, 4096), (8192, 64)], 4096, 4160, PIECES),   # the next one follows without a gap
    ([(4096, 4096), (8192, 64)], 4096, 4161, SHORT),
    ([(4096, 4096), (8192, 64), (8256, 64)], 5000, 3320, PIECES),
    ([(4096, 4096), (8448, 4096)], 4096, 8192, SHORT),  # a gap
    ([(4096, 4096)], 64, 64, UNKNOWN),              # no device allocation
    ([(4096, 4096)], 4096, 2**64 - 64, SHORT),      # beyond the address space
], ids=str)
def test_extent_of_a_buffer(extent, allocations, p, size, want):
    assert extent(allocations, p, size) == want
