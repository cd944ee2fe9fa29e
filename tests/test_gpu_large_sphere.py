"""Spheres whose particle phase goes past the first chunk of its lists: boxes of more cells per
block than the link pass keeps directions for (2048, from R = 10 on), and steps that convert
more cells than one impulse chunk holds (64)."""
import numpy as np
import pytest

from gpu_helpers import TOL_F32, TOL_F64, compare, pair, rel_l2, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("precision,tol", [("f64", TOL_F64), ("f32", TOL_F32)])
@pytest.mark.parametrize("R,closed", [(10.3, False), (12.4, True)])
def test_large_moving_sphere_matches_the_oracle(precision, tol, R, closed):
    from paper_2009_12279_gb300 import workloads

    shape = (36, 34, 33)
    nx, ny, nz = shape
    fl = np.zeros((nz, ny, nx), np.uint8)
    if closed:
        fl[0] = fl[-1] = 1
    prm = dict(periodic=(1, 1, 0 if closed else 1), eta=1.0 / 6.0, beta=0.5, lambda_p=100.0)
    u0 = workloads.random_velocity(shape, 1e-3, 21) * (fl == 0)
    t0 = workloads.random_stress(shape, 1e-5, 22) * (fl == 0)
    g, o = pair(shape, prm, fl, precision=precision)
    for s in (g, o):  # heavy: it keeps its pace
        s.add_particle((17.4, 16.6, 16.3), R, 30.0, v=(0.12, -0.09, 0.0), w=(1e-3, -2e-3, 5e-4))
        s.init_fields(u=u0, tau=t0)
    most = before = 0
    for _ in range(30):
        g.step(1)
        o.step(1)
        c, d = g.conversions(), o.diag()
        assert (c["created"], c["destroyed"]) == (d["created"], d["destroyed"])
        most, before = max(most, c["created"] + c["destroyed"] - before), c["created"] + c["destroyed"]
    assert most > 64
    pg, po = g.read_particle(0), o.read_particle(0)
    assert max(rel_l2(pg[k], po[k]) for k in ("X", "v", "w")) <= tol
    assert rel_l2(pg["F"], po["F"]) <= 10 * tol and rel_l2(pg["T"], po["T"]) <= 10 * tol
    e = compare(g, o)
    assert max(e["u"], e["tau"]) <= tol, e
    g.close()
