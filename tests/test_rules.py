"""The rules of csrc/rules.h, compiled for the host. What the fixed-point mode adds up in floating point must not
depend on the device, so neither may its choice between kernels that add in another order."""
import ctypes
import os
import subprocess

import pytest

from paper_2011_01207_gb300 import build

SRC = """#include "rules.h"
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
