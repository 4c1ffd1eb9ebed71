"""Edge nodes of the odd step (closed sides, outlet pairs, ragged row ends), which
go one per thread beside the vector path: widths around the vectors and warp
spans (FP64: 2 and 64 nodes, FP32: 4 and 128), every kind of side, against the
oracle after both step kinds.  FP64 to 1e-12 and FP32 to 1e-4 of the largest
velocity, the bounds of the other parity tests; 16-bit storage runs the same
paths and is checked for agreement between two step groupings."""
import numpy as np
import pytest

from _helpers import field_errors, gpu_lattice, oracle_lattice
from paper_1803_09380_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SIDES = {
    "box": ((wl.BOUNCEBACK,) * 4, (0, 0, 0, 0, 0, 0, 0.03, 0), (0.0, 0.0)),
    "slip": ((wl.FREESLIP,) * 4, (0,) * 8, (0.0, 0.0)),
    "channel": ((wl.INLET_EQ, wl.OUTLET_ZEROGRAD, wl.FREESLIP, wl.FREESLIP), (0,) * 8, (0.03, 0.0)),
    "walled": ((wl.INLET_EQ, wl.OUTLET_ZEROGRAD, wl.BOUNCEBACK, wl.BOUNCEBACK), (0,) * 8, (0.03, 0.0)),
    "tube": ((wl.PERIODIC, wl.PERIODIC, wl.BOUNCEBACK, wl.FREESLIP), (0, 0, 0, 0, 0.02, 0, 0, 0), (0.0, 0.0)),
    "pipe": ((wl.FREESLIP, wl.BOUNCEBACK, wl.PERIODIC, wl.PERIODIC), (0, 0, 0, 0.02, 0, 0, 0, 0), (0.0, 0.0)),
}


def _case(side, nx, ny):
    bc, wall_u, inlet = SIDES[side]
    return wl.Case(side, nx, ny, 0.8, bc=bc, wall_u=wall_u, inlet_u=inlet)


@pytest.mark.parametrize("side", sorted(SIDES))
@pytest.mark.parametrize("nx", [4, 5, 6, 7, 63, 64, 65, 66, 67, 127, 128, 129, 130, 131, 257])
def test_edge_nodes_match_the_oracle(side, nx):
    case = _case(side, nx, 9)
    start = wl.random_fields(nx, 9, 11, du=0.01, drho=0.001)
    ora = oracle_lattice(case)
    ora.init_equilibrium(*start)
    ora.step(7)
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-4)):
        gpu = gpu_lattice(case, prec)
        gpu.init_equilibrium(*start)
        gpu.step(7)
        e = field_errors(gpu, ora)
        assert max(e["ux"], e["uy"], e["rho"], e["f"]) < tol, (prec, e)
        gpu.close()


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("nx", [5, 66, 129, 257])
def test_edge_nodes_in_16_bits_do_not_depend_on_the_call(prec, nx):
    case = _case("walled", nx, 11)
    start = wl.random_fields(nx, 11, 12, du=0.01, drho=0.001)
    out = []
    for calls in ((12,), (3, 1, 8)):
        lat = gpu_lattice(case, prec)
        lat.init_equilibrium(*start)
        for n in calls:
            lat.step(n)
        out.append(lat.f)
        lat.close()
    assert np.all(np.isfinite(out[0])) and np.array_equal(*out)
