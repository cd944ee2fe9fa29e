"""The tuners time and record only what a kernel of the solve or the pool reads."""
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _solver(shape, precision, schedule, **kw):
    from paper_2009_12279_gb300 import Solver

    return Solver(shape, precision=precision, schedule=schedule, eta=1.0 / 6.0, beta=0.5, lambda_p=200.0, **kw)


def test_z_chunks_only_where_a_stress_kernel_has_them():
    from paper_2009_12279_gb300 import lbve

    shape = (46, 22, 40)  # block widths 32 and 64
    for precision in ("f64", "f32"):  # per-cell stress kernel
        s = _solver(shape, precision, lbve.SCHED_AUTO)
        r = s.autotune(steps=2)
        assert r["candidates"] == 2 and r["fv_zchunk"] == 1
        s.close()
    # the tiled stress kernel of the same shape and precision: nothing recorded for it yet
    s = _solver(shape, "f32", lbve.SCHED_SPLIT)
    assert s.autotune(steps=0)["fv_zchunk"] > 1
    r = s.autotune(steps=2)
    assert r["candidates"] > 2 and r["fv_zchunk"] > 1
    s.close()
    # nor for another stress update
    s = _solver(shape, "f32", lbve.SCHED_SPLIT, giesekus_alpha=0.2)
    assert s.autotune(steps=2)["candidates"] > 2
    s.close()
    s = _solver(shape, "f32", lbve.SCHED_SPLIT)
    assert s.autotune(steps=2)["candidates"] == 0
    s.close()


def test_default_chunk_is_the_running_kernels():
    """The two-cell stress kernel has a chunk rule of its own: the schedule measured first is
    the one that runs untuned, and it is reported as such."""
    from paper_2009_12279_gb300 import lbve

    a = _solver((64, 16, 200), "f32", lbve.SCHED_PIPELINED)
    b = _solver((64, 16, 200), "f32", lbve.SCHED_SPLIT)
    assert (a.stress_kernel, b.stress_kernel) == ("pairs", "tiles")
    assert a.autotune(steps=0)["fv_zchunk"] != b.autotune(steps=0)["fv_zchunk"]
    a.close()
    b.close()


@pytest.mark.parametrize("graphs", [True, False])
def test_pool_tiles_only_where_batched_kernels_run(graphs):
    import torch

    from paper_2009_12279_gb300 import lbve, serve
    from test_gpu_pool import _members

    reqs = _members("f32")
    stream = torch.cuda.Stream()
    pool = lbve.Pool("f32", budget_bytes=10**10, stream=stream.cuda_stream, graphs=graphs)
    solvers = [serve.build_solver(r, "f32", stream.cuda_stream) for r in reqs]
    for s in solvers:
        pool.admit(s)
    r = pool.autotune(steps=2)
    assert len(r["classes"]) == len({q.shape[0] for q in reqs})
    if graphs:  # kernels of their own: the present schedule is timed, nothing else
        assert solvers[0].time == 6 and r["ms_per_step_after"] == r["ms_per_step_before"]
    else:
        assert solvers[0].time > 6
    pool.close()
