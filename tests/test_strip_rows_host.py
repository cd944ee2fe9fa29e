"""Rows per strip of the 16-bit row pipeline: the search over the splits that differ gives what
the search over every split gives, in few enough steps for each launch to ask."""
import ctypes
import random
import subprocess
import time

import pytest

from paper_2009_12279_gb300 import build

SRC = """
#include "lbve_launch.h"
extern "C" int strip_rows(int ny, int nz, long long places) { return lbve::strip_rows(ny, nz, places); }
"""


@pytest.fixture(scope="module")
def strip_rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cu").write_text(SRC)
    so = d / "rows.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-I", build.INCLUDE, "-o", str(so), str(d / "rows.cu")], check=True, capture_output=True)
    f = ctypes.CDLL(str(so)).strip_rows
    f.argtypes, f.restype = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong], ctypes.c_int
    return f


def _every_split(ny, nz, places):
    best, yc, n = None, ny, 1
    while n <= ny and (n == 1 or n * nz <= 32 * places):
        rows = -(-ny // n)
        cost = -(-(-(-ny // rows) * nz) // places) * (2 * rows + 3)
        if best is None or cost < best:
            best, yc = cost, rows
        n += 1
    return yc


def test_equal_to_the_search_over_every_split(strip_rows):
    rng = random.Random(5)
    cases = [(ny, nz, p) for ny in (1, 2, 3, 7, 64, 128, 255, 256, 512) for nz in (1, 3, 64, 512) for p in (152, 304, 760)]
    cases += [(int(2 ** rng.uniform(0, 12)), int(2 ** rng.uniform(0, 12)), rng.randint(1, 1500)) for _ in range(400)]
    cases += [(65535, 1, 304), (32768, 1, 608), (16384, 2, 608)]
    for c in cases:
        assert strip_rows(*c) == _every_split(*c), c


def test_long_sides_are_cheap(strip_rows):
    strip_rows(65535, 1, 608)
    t = time.perf_counter()
    for _ in range(2000):
        strip_rows(65535, 1, 608)
    assert (time.perf_counter() - t) / 2000 < 20e-6  # about 2 us; every split takes over 60
