"""Kernels that small grids take, against the kernels they replace there (bitwise).

Below 3 * 2^18 cells schedule AUTO updates the stress with the per-cell kernel; schedule
SPLIT keeps the tiled one.  Rows that are no multiple of the block width (37, 83, 5 cells)
run the per-cell kernels over cells in memory order.
"""
import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _case(shape, periodic, seed):
    from paper_2009_12279_gb300 import workloads

    nx, ny, nz = shape
    fl = workloads.random_obstacles(shape, 0.06, seed)
    if not periodic[0]:
        fl[:, :, 0] = fl[:, :, -1] = 1
    if not periodic[1]:
        fl[:, 0, :], fl[:, -1, :] = 1, 2  # a moving lid
    if not periodic[2]:
        fl[0], fl[-1] = 1, 1
    fluid = fl == 0
    u0 = workloads.random_velocity(shape, 2e-3, seed + 1) * fluid
    t0 = workloads.random_stress(shape, 1e-5, seed + 2) * fluid
    return fl, [(0.02, 0.0, 0.01)], u0, t0


def _run(shape, periodic, precision, schedule, steps, **kw):
    from paper_2009_12279_gb300 import Solver

    fl, wall, u0, t0 = _case(shape, periodic, 31)
    s = Solver(shape, precision=precision, schedule=schedule, periodic=periodic, eta=1.0 / 6.0, beta=0.5,
               lambda_p=200.0, body_force=(1e-6, 0.0, -2e-6), **kw)
    s.set_geometry(fl, wall)
    s.init_fields(u=u0, tau=t0)
    for n in steps:
        s.step(n)
    out = (s.read_pdfs(), *s.read_fields()[:3], s.body_forces())
    s.close()
    return out


@pytest.mark.parametrize("kw", [{}, {"fv_terms": 15, "giesekus_alpha": 0.2}, {"fene_L2": 80.0}, {"fv_terms": 2}])
@pytest.mark.parametrize("precision", ["f32", "bf16"])
@pytest.mark.parametrize("shape,periodic", [((37, 20, 18), (1, 0, 1)), ((64, 9, 7), (1, 1, 1)),
                                            ((5, 6, 35), (0, 0, 0)), ((83, 11, 6), (0, 1, 1)), ((1, 40, 3), (1, 1, 1))])
def test_per_cell_stress_equals_tiled_bitwise(precision, shape, periodic, kw):
    from paper_2009_12279_gb300 import lbve

    a = _run(shape, periodic, precision, lbve.SCHED_AUTO, (1, 4, 2), **kw)
    b = _run(shape, periodic, precision, lbve.SCHED_SPLIT, (1, 4, 2), **kw)
    for name, x, y in zip(("pdfs", "rho", "u", "tau", "body forces"), a, b):
        assert np.array_equal(x, y), name
