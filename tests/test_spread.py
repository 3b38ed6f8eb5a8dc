"""The shared memory that holds every SM at its even share of a grid (csrc/spread.h), compiled for the host."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2202_05008_b200", "csrc")
SMS, SM_BYTES, UNIT = 148, 228 * 1024, 128


@pytest.fixture(scope="module")
def spread(tmp_path_factory):
    d = tmp_path_factory.mktemp("spread")
    src, lib = str(d / "spread.cc"), str(d / "libspread.so")
    with open(src, "w") as f:
        f.write('#include "spread.h"\nextern "C" size_t spread(size_t d, size_t f, uint64_t b, uint32_t n, size_t m)'
                "{ return evo::spread_bytes(d, f, b, n, m); }\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
    fn = C.CDLL(lib).spread
    fn.argtypes, fn.restype = [C.c_size_t, C.c_size_t, C.c_uint64, C.c_uint32, C.c_size_t], C.c_size_t
    return fn


def _resident(dynamic, fixed):
    block = (dynamic + fixed + UNIT - 1) // UNIT * UNIT
    return SM_BYTES // block


@pytest.mark.parametrize("static", [0, 128, 2432, 9728, 13568, 17280])
def test_an_sm_holds_its_share_and_no_more(spread, static):
    fixed = static + 1024
    for share in range(1, 9):
        for blocks in (SMS * (share - 1) + 1, SMS * share - 37, SMS * share):
            for dynamic in (0, 1544, 6560, 14848, 26144):
                got = spread(dynamic, fixed, blocks, SMS, SM_BYTES)
                assert got >= dynamic
                if _resident(dynamic, fixed) >= share:              # the share fits: it still does, and nothing above it
                    assert _resident(got, fixed) == share, (share, blocks, dynamic)
                else:
                    assert got == dynamic


def test_larger_grids_are_left_alone(spread):
    assert spread(5000, 1024, SMS * 8 + 1, SMS, SM_BYTES) == 5000
    assert spread(5000, 1024, 0, SMS, SM_BYTES) == 5000
