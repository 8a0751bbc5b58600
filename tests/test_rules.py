"""The rules and places of csrc/rules.h, compiled for the host. What the fixed-point mode adds up in floating point must not
depend on the device, so neither may its choice between kernels that add in another order."""
import ctypes
import os
import subprocess

import pytest

from paper_2011_01207_gb300 import build

SRC = """#include "rules.h"
// the lists of n candidates, which lie anywhere in the room of nt tiles, as long as they can get: whether each
// chunk's lists end before the first mask that is still to be read and inside the room, and the places of the
// chunks in the room of theirs
extern "C" int lists_fit(int nt, int mult, int n) {
    const long room = (long)(list_entry_base(nt, 1, mult) - list_entry_base(0, 0, mult));
    const long mask0 = (long)list_mask_base(nt, mult);
    if (mask0 + 8L * 32 * nt * mult != room || mask0 % 8) return 0;
    const int per = list_chunk_size(n);
    long done = 0;
    for (int c = 0; c < list_chunks(n); ++c) {
        const int k0 = c * per, kc = n - k0 < per ? n - k0 : per;
        if (kc < 1 || kc > AP_CHUNK) return 0;
        done += 16L * ((kc + 15) / 16 * 16);
        if (done > room || (k0 + kc < n && done > mask0 + 8L * (k0 + kc))) return 0;
    }
    for (int tile0 = 0; tile0 < 64; ++tile0)
        if (list_meta_base(tile0 + nt, 1, mult) - list_meta_base(tile0, 0, mult) < (size_t)list_chunks(n)) return 0;
    return 1;
}
extern "C" int segments(int nt) {
    for (int w = 0; w < 4; ++w) {
        int mine = 0;
        for (int t = w; t < nt; t += 4) ++mine;
        if (segment_tile(nt, w + 1) - segment_tile(nt, w) != mine) return 0;
    }
    return segment_tile(nt, 0) == 0 && segment_tile(nt, 4) == nt;
}
extern "C" int five(long n, int sms, int fixed) { return gather_five(n, sms, fixed != 0); }
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, lib = os.path.join(d, "rules.cpp"), os.path.join(d, "rules.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + build.CSRC, src, "-o", lib], check=True)
    r = ctypes.CDLL(lib)
    r.five.argtypes = [ctypes.c_long, ctypes.c_int, ctypes.c_int]
    return r


def test_fixed_mode_is_the_same_on_every_device(rules):
    for n in (1, 648, 27033, 27034, 40000, 62259, 62260, 96000, 100000000):
        assert len({rules.five(n, sms, 1) for sms in (1, 66, 108, 132, 148, 152, 160, 208)}) == 1
        assert rules.five(n, 152, 1) == rules.five(n, 152, 0)


def test_gather_line(rules):
    assert rules.five(62259, 152, 0) and not rules.five(62260, 152, 0)
    assert rules.five(27033, 66, 0) and not rules.five(27034, 66, 0)


def test_lists_stay_in_their_room(rules):
    """Every number of candidates up to all of the tiles' atoms; for large blocks the numbers around each step."""
    for mult in (1, 2, 4, 8):
        for nt in list(range(1, 40)) + [60, 86, 87, 120, 301, 1000]:
            cap = 32 * nt * mult
            some = range(cap + 1) if cap <= 8000 else {k + d for k in range(0, cap + 1, 160) for d in (-1, 0, 1)} | {cap}
            assert all(rules.lists_fit(nt, mult, n) for n in some if 0 <= n <= cap), (mult, nt)


def test_segments_are_the_warps_tiles(rules):
    assert all(rules.segments(nt) for nt in range(1, 500))
