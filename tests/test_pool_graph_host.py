"""The steps of a pool's replayed graph: an even number, its kernels bounded for any call."""
import ctypes
import subprocess

import pytest

from paper_2009_12279_gb300 import build

SRC = """
#include "lbve_launch.h"
extern "C" int block_steps(long long nodes, int nsteps) { return lbve::graph_block_steps(nodes, nsteps); }
"""


@pytest.fixture(scope="module")
def block_steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("graph")
    (d / "block.cu").write_text(SRC)
    so = d / "block.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-I", build.INCLUDE, "-o", str(so), str(d / "block.cu")], check=True, capture_output=True)
    f = ctypes.CDLL(str(so)).block_steps
    f.argtypes, f.restype = [ctypes.c_longlong, ctypes.c_int], ctypes.c_int
    return f


@pytest.mark.parametrize("nodes", [0, 1, 2, 3, 130, 256, 320, 683, 1023, 1024, 1025, 10**6])
def test_block_is_even_and_bounded(block_steps, nodes):
    most = block_steps(nodes, 1)  # a call that fits is one graph
    assert most >= 2 and most % 2 == 0 and (most == 2 or most * nodes <= 4096)
    for nsteps in (1, 2, most - 1, most):
        assert nsteps < 1 or block_steps(nodes, nsteps) == most
    for nsteps in (most + 1, most + 2, 2 * most, 2 * most + 1, 25, 100, 1000, 10**6 + 1, 2**31 - 1):
        if nsteps <= most:
            continue
        b = block_steps(nodes, nsteps)
        left = nsteps - (nsteps - 1) // b * b
        assert b % 2 == 0 and 2 <= b <= most and 2 * b >= most
        assert 1 <= left <= b  # the call's last graph
        assert b + left <= most + (nsteps - 1) % most + 1


def test_few_steps_to_capture(block_steps):
    assert block_steps(130, 30) == 30 and block_steps(130, 100) == 16
