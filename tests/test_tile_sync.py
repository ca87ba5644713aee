"""Barriers of the specialised passes' transposes (csrc/tile_sync.h), on the CPU:
over several tiles, no warp may write a shared-memory position that another warp
reads or writes unless the CTA met in between. Stage lists are random; a warp's
positions are those with its warp bits where a transpose stays inside warps, and
any position where it does not. The same check finds the hazard when the barrier
before a tile's first transpose is left out of the flags."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

from test_planner_emulated import CSRC, ROOT, _cuda_include

SOURCE = """
#include <cstring>
#include "tile_sync.h"
using namespace qsim;
template <typename R> void flags(int stages, const int *warp, char *out) {
    static TileParams<R> P;
    std::memset(&P, 0, sizeof(P));
    P.n_stages = stages;
    for (int s = 0; s < stages; ++s) {
        int j = 0;
        for (int b = 0; b < 16; ++b)
            if ((warp[s] >> b) & 1) P.st[s].wloc[j++] = b;
    }
    const std::vector<char> f = transpose_sync<R>(P);
    std::memcpy(out, f.data(), stages);
}
extern "C" void flags64(int n, const int *w, char *out) { flags<float>(n, w, out); }
extern "C" void flags128(int n, const int *w, char *out) { flags<dd>(n, w, out); }
"""
LOCAL, BEFORE = 1, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    inc, cxx = _cuda_include(), shutil.which("g++")
    if inc is None or cxx is None:
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("sync")
    src, out = str(d / "sync.cpp"), str(d / "libsync.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-I", inc, "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, src, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(out)


def flags_of(lib, name, warps):
    out = ctypes.create_string_buffer(len(warps))
    getattr(lib, name)(len(warps), (ctypes.c_int * len(warps))(*warps), out)
    return list(out.raw)


def overlap(a, b):
    """Whether two different warps can touch one position: a, b are the warp bits of local accesses, None of others."""
    return a is None or b is None or a != b  # the same bits: each warp has positions of its own


def hazard(flags, warps, tiles=3):
    """Two accesses of different warps to one position, one of them a write, with no meeting of the CTA in between."""
    since = []  # (warp bits or None, is a write) since the CTA last met
    for _ in range(tiles):
        for s in range(1, len(warps)):
            local = warps[s] if flags[s] & LOCAL else None
            if flags[s] & BEFORE:
                since = []
            for write in (True, False):
                if any((write or w) and overlap(local, b) for b, w in since):
                    return True
                since.append((local, write))
                if local is None:  # the CTA meets after the writes and after the reads
                    since = []
    return False


@pytest.mark.parametrize("name,k,low", [("flags64", 13, 4), ("flags128", 12, 3)])
def test_no_hazard_within_and_across_tiles(lib, name, k, low):
    r = random.Random(k)
    wrapped = 0
    for _ in range(4000):
        pool = [sum(1 << b for b in r.sample(range(r.choice([0, low]), k), 3)) for _ in range(r.randint(1, 3))]
        warps = [r.choice(pool) for _ in range(r.randint(1, 12))]
        flags = flags_of(lib, name, warps)
        assert flags[0] == 0
        for s in range(1, len(warps)):
            assert bool(flags[s] & LOCAL) == (warps[s] == warps[s - 1] and warps[s] & ((1 << low) - 1) == 0)
        assert not hazard(flags, warps)
        if len(warps) > 1 and flags[1] & BEFORE:
            assert hazard([0, flags[1] & ~BEFORE] + flags[2:], warps)
            wrapped += 1
    assert wrapped > 100
