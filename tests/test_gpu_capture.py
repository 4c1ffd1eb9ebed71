"""Steps that the caller captures into a graph of its own, mixed with plain
calls: whatever the order, the lattice is bitwise where the same number of
plain steps puts it."""
import numpy as np
import pytest

from _helpers import gpu_lattice
from paper_1803_09380_gb300 import ibm
from paper_1803_09380_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = {
    "fixed": lambda: wl.couette(128),
    "pair": lambda: wl.settling_pair(nx=64, ny=130, diameter=10.0, density_ratio=1.2, gravity=2e-4),
}


def _capture(lat, n):
    """A graph of n steps of lat (n even: a replay begins where it ended)."""
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=lat._stream, capture_error_mode="relaxed"):
        lat.step(n, ibm.STEP_NO_GRAPH)

    def replay():
        with torch.cuda.stream(lat._stream):
            g.replay()
    replay.graph = g                     # lives as long as the function
    return replay


def _same(lat, case, prec, steps):
    ref = gpu_lattice(case, prec)
    ibm.ibm_set_option(ref.h, ibm.IBM_OPT_IB_PHASES, 1)
    ref.step(steps)
    assert np.all(np.isfinite(ref.f)) and np.any(ref.bodies[:, 6:] != 0.0)
    for a, b in ((lat.f, ref.f), (lat.bodies, ref.bodies), (lat.markers, ref.markers), (lat.resid, ref.resid),
                 *zip(lat.moments(), ref.moments())):
        assert np.array_equal(a, b)
    ref.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_replays_of_a_captured_first_call_mixed_with_plain_steps(name, prec):
    """The captured call is the lattice's first: replays, plain calls and
    changes of the correction grid in turn."""
    case = CASES[name]()
    lat = gpu_lattice(case, prec)
    replay = _capture(lat, 2)
    replay()
    replay()
    lat.step(4)
    replay()
    lat.step(2)
    lat.set_ib_ctas(1)
    lat.step(2)
    replay()
    replay()
    lat.step(1)
    _same(lat, case, prec, 19)
    lat.close()
