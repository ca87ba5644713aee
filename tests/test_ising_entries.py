"""The numbering of an Ising op's table entries (csrc/ising_table.h), checked on
the CPU: every entry of the table is formed by exactly one thread, and a warp's
threads form entries of one kind, so that no warp waits for an outside energy
(n_free^2 / 2 additions) beside fields (n_free each)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from test_planner_emulated import CSRC, ROOT, _cuda_include

SOURCE = """
#include "ising_table.h"
using namespace qsim;
extern "C" uint64_t threads(int tb, int rb, int k, int n_free) { return ising_threads(tb, rb, k, n_free); }
extern "C" uint64_t pairs(int tb, int rb, int k, int n_free) { return ising_thr_stride(rb, 1 << tb, k, n_free) / 2; }
extern "C" void entries(int tb, int rb, int k, int n_free, int64_t *out) {
    for (uint64_t i = 0; i < ising_threads(tb, rb, k, n_free); ++i) {
        const IsingEntry e = ising_entry(i, tb, rb, k, n_free);
        const int64_t v[4] = {e.kind, e.row, e.col, (int64_t)e.at};
        for (int j = 0; j < 4; ++j) out[4 * i + j] = v[j];
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc, cxx = _cuda_include(), shutil.which("g++")
    if inc is None or cxx is None:
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("ising")
    src, out = str(d / "ising.cpp"), str(d / "libising.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", inc, "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, src, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    lib = ctypes.CDLL(out)
    lib.threads.restype = lib.pairs.restype = ctypes.c_uint64
    return lib


# thread and register bits of complex64 and complex128 tiles
@pytest.mark.parametrize("tb,rb", [(8, 5), (8, 4)])
@pytest.mark.parametrize("n_free", [0, 1, 4, 5, 9, 13])
def test_every_entry_once_and_warps_of_one_kind(lib, tb, rb, n_free):
    k = tb + rb
    count, threads = lib.pairs(tb, rb, k, n_free), lib.threads(tb, rb, k, n_free)
    out = np.empty((threads, 4), dtype=np.int64)
    lib.entries(tb, rb, k, n_free, out.ctypes.data_as(ctypes.c_void_p))
    kind, row, col, at = out.T
    used = kind > 0
    np.testing.assert_array_equal(np.sort(at[used]), np.arange(count))
    # what an entry is follows from its place in the table
    for y, x, c, a in out[used][:: max(1, count // 5000)]:
        p = (1 + rb) << tb
        if a < p:
            assert (x, y) == (a // (1 + rb), 5 if a % (1 + rb) == 0 else 2) and (y == 5 or c == a % (1 + rb) - 1)
        elif a < p + (1 << rb):
            assert (x, y) == (a - p, 3)
        else:
            t = a - p - (1 << rb)
            assert (x, y) == (t // (k + 1), 4 if t % (k + 1) == k else 1) and (y == 4 or c == t % (k + 1))
    assert threads % 32 == 0 and len(kind) == threads
    for w in kind.reshape(-1, 32):
        assert len(set(w[w > 0])) <= 1
