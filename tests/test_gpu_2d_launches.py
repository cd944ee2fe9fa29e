"""Two-dimensional calls of more steps than one multi-step launch takes."""
import numpy as np
import pytest

from gpu_helpers import require_gpu
from test_gpu_2d_steps import _setup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


def _run(precision, steps):
    from paper_2009_12279_gb300.lbve import Solver2D

    shape, periodic = (33, 6), (1, 0)
    fl, _, u0, t0, F, prm = _setup(shape, periodic, 11)
    s = Solver2D(shape, precision=precision, body_force=(1e-6, 0.0), **prm)
    s.set_geometry(fl)  # walls at rest: the fields stay finite for as long as the test runs
    s.set_force_field(F)
    s.init_fields(u=u0, tau=t0)
    for n in steps:
        s.step(n)
    out = s.read_fields()
    assert s.time == sum(steps)
    s.close()
    return out


@pytest.mark.parametrize("precision", ["f64", "f32"])
def test_call_of_several_launches(precision):
    """A call of more steps than one launch takes (4096), even and odd remainders, against
    calls of one launch each."""
    ref = _run(precision, [1000] * 8 + [195])
    assert all(np.isfinite(a).all() for a in ref)
    for steps in ([8195], [4096, 4099], [4097, 4098]):
        for a, b in zip(ref, _run(precision, steps)):
            assert np.array_equal(a, b)
