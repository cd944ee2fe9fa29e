"""The grid barrier of multi-step launches (csrc/lbve_gridbar.cuh): steps meet, and a wait
that runs out ends the launch with a status and leaves the context usable.  The wait runs out
because the barrier expects one block more than the launch has; every wait is bounded by the
barrier itself."""
import ctypes
import subprocess
import time

import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu

SRC = """
#include "lbve_gridbar.cuh"
// Blocks of 64 threads meet `steps` times on the words out[0..1]; out[2] is the status word,
// out[3 + b] becomes the number of barriers block b passed.  Block 0 waits at most first_ns0 at the
// first barrier, the others first_ns.
__global__ void k_meet(unsigned *out, int steps, unsigned blocks, unsigned long long first_ns0,
                       unsigned long long first_ns, unsigned long long wait_ns) {
    unsigned passed = 0;
    for (int s = 0; s < steps; ++s) {
        if (!lbve::grid_barrier(out, (unsigned)s, blocks, out + 2, blockIdx.x == 0 ? first_ns0 : first_ns, wait_ns)) break;
        ++passed;
    }
    if (threadIdx.x == 0) out[3 + blockIdx.x] = passed;
}
extern "C" int meet(unsigned *host, int nblocks, int steps, unsigned blocks, unsigned long long first_ns0,
                    unsigned long long first_ns, unsigned long long wait_ns) {
    unsigned *d = nullptr;
    const size_t bytes = sizeof(unsigned) * (3 + (size_t)nblocks);
    if (cudaMalloc((void **)&d, bytes) != cudaSuccess) return -1;
    cudaError_t e = cudaMemset(d, 0, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(d + 1, host + 1, sizeof(unsigned), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        void *args[] = {&d, &steps, &blocks, &first_ns0, &first_ns, &wait_ns};
        e = cudaLaunchCooperativeKernel((const void *)k_meet, dim3(nblocks), dim3(64), args, 0, nullptr);
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(host, d, bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return (int)e;
}
"""
MS = 10**6


@pytest.fixture(scope="module")
def meet(tmp_path_factory):
    require_gpu()
    from paper_2009_12279_gb300 import build

    d = tmp_path_factory.mktemp("gridbar")
    (d / "meet.cu").write_text(SRC)
    so = d / "meet.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", build.CSRC,
                    "-o", str(so), str(d / "meet.cu")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))
    u64 = ctypes.c_ulonglong
    lib.meet.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_uint, u64, u64, u64]

    def call(nblocks, steps, blocks, first0, first, wait, given_up=0):
        out = (ctypes.c_uint * (3 + nblocks))()
        out[1] = given_up
        t = time.monotonic()
        assert lib.meet(out, nblocks, steps, blocks, first0, first, wait) == 0
        assert out[1] == (1 if given_up or out[2] else 0)
        return out[0], out[2], list(out[3:]), time.monotonic() - t

    return call


@pytest.mark.parametrize("nblocks,steps", [(1, 3), (7, 50), (152, 1000)])
def test_every_block_passes_every_barrier(meet, nblocks, steps):
    word, status, passed, _ = meet(nblocks, steps, nblocks, 1000 * MS, 1000 * MS, 1000 * MS)
    assert (word, status, passed) == (nblocks * steps, 0, [steps] * nblocks)


@pytest.mark.parametrize("nblocks", [1, 5, 152])
def test_a_wait_that_runs_out_sets_the_status(meet, nblocks):
    word, status, passed, _ = meet(nblocks, 4, nblocks + 1, 20 * MS, 20 * MS, 20 * MS)
    assert status == 2 and passed == [0] * nblocks and word >> 31 == 1


def test_no_wait_after_a_launch_that_gave_up(meet):
    """The second word still set: the launches behind one that gave up return at once."""
    meet(1, 1, 1, MS, MS, MS)
    word, status, passed, seconds = meet(64, 4, 65, 5000 * MS, 5000 * MS, 20 * MS, given_up=1)
    assert status == 0 and passed == [0] * 64 and seconds < 2.5


def test_one_block_that_gives_up_ends_the_waits_of_the_others(meet):
    """Block 0 gives up after 20 ms, the others would wait for 5 s: they see it and leave."""
    meet(1, 1, 1, MS, MS, MS)  # the context exists before the clock starts
    word, status, passed, seconds = meet(64, 4, 65, 20 * MS, 5000 * MS, 20 * MS)
    assert status == 2 and passed == [0] * 64
    assert seconds < 2.5
    # the context is usable: the same blocks meet in a further launch
    assert meet(64, 4, 64, 1000 * MS, 1000 * MS, 1000 * MS)[2] == [4] * 64
