"""Two-dimensional steps: several in one launch, one by one, and the grids too large for
one launch give the same fields (bitwise), and those of the FP64 oracle."""
import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _setup(shape, periodic, seed):
    nx, ny = shape
    rng = np.random.default_rng(seed)
    fl = (rng.random((ny, nx)) < 0.05).astype(np.uint8)
    if not periodic[0]:
        fl[:, 0] = fl[:, -1] = 1
    if not periodic[1]:
        fl[0] = fl[-1] = 1
    ub = rng.uniform(-0.01, 0.01, (2, ny, nx)) * fl
    u0 = rng.uniform(-2e-3, 2e-3, (2, ny, nx)) * (fl == 0)
    t0 = 1e-5 * rng.standard_normal((3, ny, nx)) * (fl == 0)
    F = rng.uniform(-1e-6, 1e-6, (2, ny, nx))
    prm = dict(periodic=periodic, eta=0.3, beta=0.4, lambda_p=150.0)
    return fl, ub, u0, t0, F, prm


def _gpu_run(shape, periodic, precision, steps):
    from paper_2009_12279_gb300.lbve import Solver2D

    fl, ub, u0, t0, F, prm = _setup(shape, periodic, 11)
    s = Solver2D(shape, precision=precision, body_force=(1e-6, 0.0), **prm)
    s.set_geometry(fl, ub)
    s.set_force_field(F)
    s.init_fields(u=u0, tau=t0)
    for n in steps:
        s.step(n)
    out = s.read_fields()
    assert s.time == sum(steps)
    s.close()
    return out


# tiles of 32 x 4: ragged in x and y, single cells, closed and periodic sides
@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("shape,periodic", [((33, 5), (1, 1)), ((64, 8), (0, 0)), ((1, 9), (1, 1)), ((70, 3), (0, 1)),
                                            ((31, 41), (1, 0)), ((196, 196), (0, 0))])
def test_many_steps_in_one_launch(precision, shape, periodic):
    from oracle import oracle as o2

    one = _gpu_run(shape, periodic, precision, [1] * 13)
    many = _gpu_run(shape, periodic, precision, [13])
    mixed = _gpu_run(shape, periodic, precision, [4, 1, 8])
    for a, b, c in zip(one, many, mixed):
        assert np.array_equal(a, b) and np.array_equal(a, c)
    fl, ub, u0, t0, F, prm = _setup(shape, periodic, 11)
    o = o2.Oracle2D(shape, g=(1e-6, 0.0), **prm)
    o.set_geometry(fl, ub)
    o.set_force(F)
    o.init_fields(u=u0, tau=t0)
    o.step(13)
    for a, b in zip(many, o.read_fields()):
        if precision == "f64":
            assert np.array_equal(a, b)
        else:
            assert np.linalg.norm(a - b) <= 1e-5 * max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_grid_too_large_for_one_launch(precision):
    """A 900 x 700 grid has more tiles than the device holds: a launch (FP64: two) per step."""
    from oracle import oracle as o2

    shape, periodic = (900, 700), (1, 0)
    got = _gpu_run(shape, periodic, precision, [5])
    fl, ub, u0, t0, F, prm = _setup(shape, periodic, 11)
    o = o2.Oracle2D(shape, g=(1e-6, 0.0), **prm)
    o.set_geometry(fl, ub)
    o.set_force(F)
    o.init_fields(u=u0, tau=t0)
    o.step(5)
    for a, b in zip(got, o.read_fields()):
        if precision == "f64":
            assert np.array_equal(a, b)
        else:
            assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
