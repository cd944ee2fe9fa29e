"""Host side of the grid barrier (csrc/lbve_gridbar.cuh): a call's steps are split into
launches whose barrier count stays inside its 32-bit word."""
import ctypes
import subprocess

import pytest

from paper_2009_12279_gb300 import build

SRC = """
#include "lbve_gridbar.cuh"
extern "C" int launch_steps(int steps, long long blocks) { return lbve::launch_steps(steps, blocks); }
"""


@pytest.fixture(scope="module")
def launch_steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("gridbar")
    (d / "split.cu").write_text(SRC)
    so = d / "split.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-o", str(so), str(d / "split.cu")], check=True, capture_output=True)
    f = ctypes.CDLL(str(so)).launch_steps
    f.argtypes, f.restype = [ctypes.c_int, ctypes.c_longlong], ctypes.c_int
    return f


# 912 blocks wrap a 32-bit count after 4.7 M steps, 343 (196^2 cells) after 12.5 M
@pytest.mark.parametrize("steps", [1, 2, 4095, 4096, 4097, 4_709_394, 12_521_771, 2**31 - 1])
@pytest.mark.parametrize("blocks", [1, 2, 343, 912, 152 * 32, 2**20, 2**31 - 1])
def test_barrier_count_stays_in_its_word(launch_steps, steps, blocks):
    left, first = steps, None
    m = launch_steps(left, blocks)
    assert 1 <= m <= min(left, 4096)
    assert m == 1 or m * blocks <= 2**30  # every arrival of the launch's barriers
    # the same length again and again, then the rest: the sum is the call's steps
    rest = left % m
    assert launch_steps(left - m, blocks) in (m, rest, left - m) if left > m else True
    if rest:
        assert launch_steps(rest, blocks) == rest
