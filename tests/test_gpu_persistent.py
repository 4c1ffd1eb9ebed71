"""The persistent correction kernel with its grid barrier in global memory, which
boundaries without slices run (moving ones above 256 markers, more than 60
iterations, other CTA sizes): bitwise the launch form with one kernel a phase."""
import numpy as np
import pytest

from _helpers import gpu_lattice
from paper_1803_09380_gb300 import ibm
from paper_1803_09380_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

GRIDS = (0, 76, 95, 152, 57, 114)
PERSISTENT = 3              # launches a step: correction, band collide, collide+stream (slices: 2)


def _ref(case, prec, steps):
    lat = gpu_lattice(case, prec)
    ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, 1)
    lat.step(steps)
    out = (lat.f, lat.resid, lat.bodies, *lat.moments())
    lat.close()
    assert np.all(np.isfinite(out[0]))
    return out


def _step(lat, n):
    l0 = lat.counters()[0]
    lat.step(n)
    assert lat.counters()[0] - l0 == PERSISTENT * n


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("threads,n_corr", [(512, 10), (1024, 10), (256, 61)])
def test_grids_of_the_persistent_kernel_on_a_live_lattice(prec, threads, n_corr):
    """878 markers; grid sizes that are not multiples of each other, switched
    between steps: the barrier's counter restarts for each."""
    case = wl.couette(256)
    case.n_corr = n_corr
    lat = gpu_lattice(case, prec)
    if threads != 256:
        lat.set_ib_threads(threads)
    for ctas in GRIDS:
        lat.set_ib_ctas(ctas)
        _step(lat, 3)
    ref = _ref(case, prec, 3 * len(GRIDS))
    for a, b in zip((lat.f, lat.resid, lat.bodies, *lat.moments()), ref):
        assert np.array_equal(a, b)
    lat.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", ["couette1024", "channel_mrt"])
def test_persistent_kernel_by_default_above_sixty_iterations(prec, name):
    case = wl.couette(1024) if name == "couette1024" else wl.paper_cylinder(20.0, diameter=16, mrt=True)
    case.n_corr = 61
    lat = gpu_lattice(case, prec)
    l0 = lat.counters()[0]
    lat.step(10)
    # the channel's extrapolation columns are a launch of their own
    assert lat.counters()[0] - l0 == 10 * (PERSISTENT if name == "couette1024" else PERSISTENT + 1)
    for a, b in zip((lat.f, lat.resid, lat.bodies, *lat.moments()), _ref(case, prec, 10)):
        assert np.array_equal(a, b)
    lat.close()
