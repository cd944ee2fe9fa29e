"""Two spheres that overlap: a cell that one of them frees deep inside the other bounces back
at the other's present surface velocity (Eq. (ubb))."""
import numpy as np
import pytest

from gpu_helpers import require_gpu

pytestmark = pytest.mark.gpu

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
             + [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1) if abs(a) + abs(b) + abs(c) == 2])
W = np.where(np.abs(C).sum(1) == 0, 1 / 3, np.where(np.abs(C).sum(1) == 1, 1 / 18, 1 / 36))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    require_gpu()


@pytest.mark.parametrize("precision,tol", [("f64", 1e-12), ("f32", 1e-5)])
def test_cell_freed_inside_another_sphere(precision, tol):
    """The second sphere gives up one cell four cells below the first one's surface; the first
    one spins up meanwhile.  All 18 neighbours of the freed cell are the first sphere's, so one
    step turns its momentum j = rho u into -j + 6 rho sum_i w_i c_i (c_i . u_b(r + c_i)), and the
    first sphere, which takes the cell in that step, receives exactly that impulse."""
    from paper_2009_12279_gb300 import Solver

    shape, X0, R0, rho_p = (32, 28, 28), np.array([14.1, 14.2, 13.9]), 6.0, 50.0
    inertia = 0.4 * rho_p * 4.0 / 3.0 * np.pi * R0**5
    s = Solver(shape, precision=precision, eta=1.0 / 6.0, beta=0.0, lambda_p=0.0)
    s.add_particle(X0, R0, rho_p, Text=(0.0, 0.0, 2e-3 * inertia))
    s.add_particle(X0 + [6.5, 0.0, 0.0], 2.5, rho_p)
    # hand the cell to the second sphere, which it does not cover
    cell = (16, 14, 14)
    flags = s.read_fields()[3].astype(np.uint8)
    r = cell[0] + shape[0] * (cell[1] + shape[1] * cell[2])
    assert flags.reshape(-1)[r] == 64
    rec = bytearray(s.save())
    at = rec.find(flags.tobytes())
    rec[at + r] = 65
    s.restore(bytes(rec))
    s.step(1)
    assert s.conversions()["created"] == 1 and s.read_fields()[3].reshape(-1)[r] == 0
    p = s.read_particle(0)
    assert p["w"][2] > 1e-3 and not p["dP"].any()
    out = s.probe([r])[0]
    rho, u = out[19], out[20:23]
    s.step(1)
    assert s.conversions()["destroyed"] == 1
    expected = -rho * u
    for c, w in zip(C, W):
        ub = p["v"] + np.cross(p["w"], np.array(cell) + c - p["X"])
        expected = expected + 6.0 * rho * w * c * (c @ ub)
    got = s.read_particle(0)["dP"]
    assert np.abs(got - expected).max() <= tol * np.abs(expected).max()
    s.close()
