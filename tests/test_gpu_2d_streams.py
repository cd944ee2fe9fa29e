"""Two two-dimensional solves stepped on streams of their own, each launch filling most of the
device, beside a third stream's work: the launches take turns, and both results are those of
the solves stepped alone.  (Every wait of the launches is bounded: blocks that could not all
start would end in LBVE_ETIMEOUT.)"""
import time

import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _solver(seed, stream):
    from paper_2009_12279_gb300.lbve import Solver2D

    shape = (300, 300)  # 750 tiles of some 900 resident ones
    s = Solver2D(shape, precision="f32", periodic=(1, 1), eta=0.3, beta=0.4, lambda_p=150.0, stream=stream.cuda_stream)
    s.init_fields(u=np.random.default_rng(seed).uniform(-2e-3, 2e-3, (2, 300, 300)))
    return s


def test_two_solves_on_two_streams():
    import torch

    streams = [torch.cuda.Stream() for _ in range(3)]
    refs = []
    for k in range(2):
        s = _solver(k, streams[0])
        s.step(600)
        refs.append(s.read_fields())
        s.close()
    pair = [_solver(k, streams[k]) for k in range(2)]
    x = torch.zeros(1 << 24, device="cuda")
    torch.cuda.synchronize()
    t = time.monotonic()
    for n in [2, 3, 5, 10, 20, 40, 70] * 4:
        with torch.cuda.stream(streams[2]):
            x.add_(1.0)
        for s in pair:
            s.step(n)
    got = [s.read_fields() for s in pair]
    assert time.monotonic() - t < 10.0  # no launch ran into its first barrier's limit
    for r, g in zip(refs, got):
        for a, b in zip(r, g):
            assert np.array_equal(a, b)
    for s in pair:
        s.close()
