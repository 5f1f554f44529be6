"""The host rule for the rows that a build keeps (row_copy_cap in
csrc/fim_common.cuh), compiled and run without a GPU."""
import ctypes
import os
import subprocess

import pytest

from paper_2412_19420_gb300 import build as b

SRC = r"""
#include "fim_common.cuh"
extern "C" unsigned long long cap_of(long long n) { return row_copy_cap(n); }
// steps of 32 that the row pass takes over ids [b0, b1), or -1 when an index
// wraps (more steps than ids)
extern "C" long long steps(unsigned b0, unsigned b1) {
    long long k = 0;
    for (uint32_t e0 = b0; e0 < b1; e0 += 32)
        if (++k > (long long)(b1 - b0)) return -1;
    return k;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rowcopy")
    src, so = d / "t.cpp", d / "t.so"
    src.write_text(SRC)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", b.CSRC, "-I", cuda, str(src), "-o", str(so)],
                   check=True)
    so = ctypes.CDLL(str(so))
    so.cap_of.restype, so.cap_of.argtypes = ctypes.c_ulonglong, [ctypes.c_longlong]
    so.steps.restype, so.steps.argtypes = ctypes.c_longlong, [ctypes.c_uint, ctypes.c_uint]
    return so


def test_ids_of_kept_rows_never_wrap_a_step(lib):
    assert lib.steps(2 ** 32 - 100, 2 ** 32 - 2) == -1  # what the cap is for
    n_most = (2 ** 32 - 64) // 24
    for n in (1, 1000, n_most, n_most + 1, n_most + 2, 2 ** 31 - 1):
        cap = lib.cap_of(n)
        assert cap == (24 * n if n <= n_most else 0)
        for back in range(1, 70):
            if cap > back:
                assert lib.steps(cap - back, cap) == (back + 31) // 32
