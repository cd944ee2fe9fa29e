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


@pytest.mark.parametrize("precision", ["bf16", "f32"])
def test_pool_members_of_both_kinds_equal_alone(precision):
    """70 members: the large ones step by kernels of their own, the small ones by the batched
    kernels; in a pool of 3 every member has its own.  Calls of 1, 4 and 4 steps (graphs of
    both parities, one replayed).  Fields and PDFs are those of the same solves alone."""
    import torch

    from paper_2009_12279_gb300 import Pool, Solver, workloads

    shapes = [(64, 40, 32), (48, 48, 32), (16, 12, 10)] + [(9 + k % 7, 8, 7) for k in range(67)]

    def solver(k, stream):
        shape = shapes[k]
        fl = workloads.channel_flags(shape, 1)
        fl |= workloads.random_obstacles(shape, 0.03, k).astype(fl.dtype)
        fl[2, 3, 4] = 2  # a tracked wall cell
        s = Solver(shape, precision=precision, stream=stream, periodic=(1, 0, 1), lambda_p=150.0, beta=0.4,
                   body_force=(1e-5, 0.0, 0.0), giesekus_alpha=0.2 if k == 1 else 0.0)
        s.set_geometry(fl, [(0.01, 0.0, 0.0)])
        s.init_fields(u=workloads.random_velocity(shape, 1e-3, k) * (fl == 0))
        return s

    for members in (70, 3):
        stream = torch.cuda.Stream()
        pool = Pool(precision, stream=stream.cuda_stream)
        mine = [solver(k, stream.cuda_stream) for k in range(members)]
        for s in mine:
            pool.admit(s)
        for n in (1, 4, 4):
            pool.step(n)
        res = pool.residuals()
        for k in list(range(4)) + [members - 1]:
            if k >= members:
                continue
            alone = solver(k, 0)
            for n in (1, 4, 4):
                alone.step(n)
            assert np.array_equal(alone.read_pdfs(), mine[k].read_pdfs()), (members, k)
            for a, b in zip(alone.read_fields(), mine[k].read_fields()):
                assert np.array_equal(a, b), (members, k)
            assert np.array_equal(alone.body_forces(), mine[k].body_forces()), (members, k)
            assert alone.residual() == tuple(res[k]), (members, k)
            alone.close()
        for s in mine:
            pool.remove(s)
            s.close()
        pool.close()
