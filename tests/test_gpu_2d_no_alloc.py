"""lbve2d_step allocates nothing, also in the first call that takes several steps in one launch:
a capture of another stream in the mode that forbids every thread's allocations goes on
undisturbed."""
import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_first_multi_step_call_beside_a_capture(precision):
    import torch

    from paper_2009_12279_gb300.lbve import Solver2D

    def solver():
        s = Solver2D((40, 24), precision=precision, periodic=(1, 1), stream=torch.cuda.Stream().cuda_stream)
        s.init_fields(u=1e-3 * np.random.default_rng(3).standard_normal((2, 24, 40)))
        return s

    ref = solver()
    for _ in range(6):
        ref.step(1)
    warm = solver()  # the kernels are loaded before the capture begins
    warm.step(6)
    warm.read_fields()
    s = solver()
    x = torch.ones(1000, device="cuda")
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side, capture_error_mode="global"):
        x.mul_(3.0)
        s.step(6)
    graph.replay()
    out = s.read_fields()
    torch.cuda.synchronize()
    assert bool((x == 3.0).all())
    for a, b, c in zip(ref.read_fields(), out, warm.read_fields()):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    for t in (ref, warm, s):
        t.close()
