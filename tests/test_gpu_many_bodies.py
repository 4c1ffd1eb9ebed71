"""More bodies than the short cuts hold (8 with a thread per collision partner,
16 centres on hand in the force sums), against the FP64 oracle: on slices, on
the moving slice and on the general path."""
import numpy as np
import pytest

from _helpers import field_errors, gpu_lattice, oracle_lattice, relerr
from paper_1803_09380_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = 1e-12
TOL_MOVING = 1e-10          # as for two disks: rounding of the corrections over velocities of 1e-3


def _spots(n, pitch):
    """n places of a square grid, every third one pushed against its neighbour."""
    side = int(np.ceil(np.sqrt(n)))
    xy = [(pitch * (k % side + 1) + 0.13 * k % 1.0, pitch * (k // side + 1) + 0.29 * k % 1.0) for k in range(n)]
    return xy, int(pitch * (side + 1)) + 2


def _fixed(n):
    """Rings of 20 markers turning both ways: chunks of 128 hold parts of bodies."""
    at, size = _spots(n, 11.0)
    bodies = []
    for k, c in enumerate(at):
        xy, ds = wl.ring(c[0], c[1], 3.2, count=20)
        bodies.append(wl.Body(xy, ds, wl.BODY_FIXED, xc=c, u=(0.002 * (-1) ** k, 0.001), omega=1e-3 * (k % 5 - 2),
                              radius=3.2))
    return wl.Case("fixed", size, size, 0.8, bodies=bodies)


def _free(n, diameter, density):
    """Free disks in a box, two pairs in touch, one prescribed and one fixed body."""
    at, size = _spots(n, diameter + 7.0)
    reach = diameter * 1.02                             # inside the collision force's range of 1.05
    at[1] = (at[0][0] + reach, at[0][1])
    at[n - 1] = (at[n - 2][0], at[n - 2][1] + reach)
    bodies = [wl.disk(c[0], c[1], diameter, density, 2e-4) for c in at]
    bodies[3].kind, bodies[3].u = wl.BODY_PRESCRIBED, (0.004, -0.003)
    bodies[5].kind = wl.BODY_FIXED
    return wl.Case("free", size, size, 0.8, bc=(wl.BOUNCEBACK,) * 4, bodies=bodies)


def _drifting():
    """Sixteen small disks on prescribed ways and two free ones in touch: 90 markers."""
    at, size = _spots(18, 9.0)
    bodies = []
    for k, c in enumerate(at[:16]):
        b = wl.disk(c[0], c[1], 1.4, 2.0, 0.0, kind=wl.BODY_PRESCRIBED)
        b.u, b.omega = (0.003 * (-1) ** k, 0.001 * (k % 3)), 2e-3 * (k % 4 - 1.5)
        bodies.append(b)
    for c in (at[16], (at[16][0] + 4.08, at[16][1])):
        bodies.append(wl.disk(c[0], c[1], 4.0, 10.0, 2e-4))
    return wl.Case("drifting", size, size, 0.8, bc=(wl.BOUNCEBACK,) * 4, bodies=bodies)


CASES = {
    # launches a step: slices 2; one moving slice 3; the general path 11
    "fixed 20": (lambda: _fixed(20), 2),
    "drifting 18": (_drifting, 3),
    "free 9": (lambda: _free(9, 10.0, 3.0), 11),
    "free 20": (lambda: _free(20, 6.0, 5.0), 11),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_many_bodies_against_the_oracle(name):
    make, launches = CASES[name]
    case = make()
    moving = launches != 2
    ora, gpu = oracle_lattice(case), gpu_lattice(case, "fp64")
    ora.step(30)
    gpu.step(30)
    assert gpu.counters()[0] == 30 * launches
    errs = field_errors(gpu, ora)
    tol = TOL_MOVING if moving else TOL
    assert errs["rho"] < TOL and errs["f"] < TOL and max(errs["ux"], errs["uy"]) < tol, errs
    bg, bo = gpu.bodies, ora.bodies
    assert np.max(np.abs(bg[:, 0:2] - bo[:, 0:2])) < 1e-10
    assert np.all(np.any(bo[:, 6:9] != 0.0, axis=1))
    for c in (slice(2, 4), slice(6, 8), slice(8, 9)):
        assert relerr(bg[:, c], bo[:, c]) < 1e-10
    assert relerr(gpu.markers, ora.markers) < 1e-14
    gpu.close()
