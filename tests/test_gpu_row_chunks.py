"""Per-cell kernels on planes of several row chunks, against the row pipeline (bitwise).

Tiles of the per-cell kernels sweep z within chunks of rows (49152 cells a plane in FP32,
24576 in 16-bit storage and FP64).  The shapes have two to four chunks, even and ragged, and
a last chunk that the rows do not fill.
"""
import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("precision", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("shape,periodic", [((96, 601, 3), (1, 1, 1)), ((64, 1600, 4), (1, 0, 0)), ((128, 385, 2), (1, 0, 1))])
def test_chunked_planes_equal_the_row_pipeline(precision, shape, periodic):
    from paper_2009_12279_gb300 import Solver, lbve, workloads

    fl = workloads.random_obstacles(shape, 0.05, 3)
    if not periodic[1]:
        fl[:, 0, :], fl[:, -1, :] = 1, 2  # a moving lid
    if not periodic[2]:
        fl[0], fl[-1] = 1, 1
    u0 = workloads.random_velocity(shape, 2e-3, 4) * (fl == 0)
    out = []
    for schedule in (lbve.SCHED_SPLIT, lbve.SCHED_PIPELINED):
        s = Solver(shape, precision=precision, schedule=schedule, periodic=periodic, lambda_p=200.0, beta=0.5,
                   body_force=(1e-6, 0.0, -2e-6))
        s.set_geometry(fl, [(0.02, 0.0, 0.01)])
        s.init_fields(u=u0)
        s.step(3)
        assert s.stream_collide_kernel == ("cells" if schedule == lbve.SCHED_SPLIT else "rows")
        out.append((s.read_pdfs(), *s.read_fields()[:3], s.body_forces()))
        s.close()
    for name, x, y in zip(("pdfs", "rho", "u", "tau", "body forces"), *out):
        assert np.array_equal(x, y), name
