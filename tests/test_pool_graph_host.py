"""The steps of a pool's replayed graph: an even number, its kernels bounded for any call."""
import ctypes
import subprocess

import pytest

from paper_2009_12279_gb300 import build

SRC = """
#include "lbve_launch.h"
extern "C" int block_steps(long long nodes) { return lbve::graph_block_steps(nodes); }
"""


@pytest.fixture(scope="module")
def block_steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("graph")
    (d / "block.cu").write_text(SRC)
    so = d / "block.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-I", build.INCLUDE, "-o", str(so), str(d / "block.cu")], check=True, capture_output=True)
    f = ctypes.CDLL(str(so)).block_steps
    f.argtypes, f.restype = [ctypes.c_longlong], ctypes.c_int
    return f


@pytest.mark.parametrize("nodes", [0, 1, 2, 3, 130, 256, 320, 683, 1023, 1024, 1025, 10**6])
def test_block_is_even_and_bounded(block_steps, nodes):
    b = block_steps(nodes)
    assert b >= 2 and b % 2 == 0
    assert b == 2 or b * nodes <= 2048
    # 1 to b steps are left for the call's last graph
    for nsteps in (1, 2, b - 1, b, b + 1, 2 * b, 2 * b + 1, 10**6 + 1):
        assert nsteps < 1 or 1 <= nsteps - (nsteps - 1) // b * b <= b
