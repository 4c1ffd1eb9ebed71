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


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_options_set_after_a_capture_keep_what_the_graph_holds(name, prec):
    """The slices run before the capture: options and the autotuner leave their
    lists (and the form) alone, and the memory is not handed out again."""
    import torch
    case = CASES[name]()
    lat = gpu_lattice(case, prec)
    lat.step(3)
    lat.step(1)
    per_step = lat.counters()[0]
    replay = _capture(lat, 2)
    per_step = (lat.counters()[0] - per_step) // 2
    assert per_step == (3 if name == "pair" else 2)          # slices
    for option, value in ((ibm.IBM_OPT_IB_CTAS, 2), (ibm.IBM_OPT_IB_THREADS, 512),
                          (ibm.IBM_OPT_IB_PHASES, 1), (ibm.IBM_OPT_BARRIER_LIMIT_US, 3000000)):
        ibm.ibm_set_option(lat.h, option, value)
    with torch.cuda.stream(lat._stream):
        junk = [torch.full((1 << k,), 255, dtype=torch.uint8, device="cuda") for k in range(12, 25) for _ in range(4)]
    replay()
    replay()
    lat.step(2)                                              # steps so far: 4 + 4 + 2
    lat.autotune_ib([1, 3], steps_each=2)                    # 2 x (2 + 2)
    replay()
    l0 = lat.counters()[0]
    lat.step(1)
    assert lat.counters()[0] - l0 == per_step
    _same(lat, case, prec, 21)
    assert all(bool((j == 255).all()) for j in junk)
    lat.close()


def test_markers_added_after_a_capture_open_the_form_again():
    case = wl.couette(128)
    lat = gpu_lattice(case, "fp32")
    _capture(lat, 2)
    lat.step(2)
    b = wl.couette(96).bodies[0]
    lat.add_markers(b.xy + 16.0, b.ds, **b.as_kwargs())
    l0 = lat.counters()[0]
    lat.step(1)
    assert lat.counters()[0] - l0 == 2
    lat.close()


@pytest.mark.parametrize("planned", [False, True])
def test_a_plain_call_before_the_first_replay_has_a_band(planned):
    """The captured call finds no band (none yet, or a pose was written): its
    build runs with the replays only, so a plain call ahead of them builds its
    own."""
    case = CASES["pair"]()
    lat = gpu_lattice(case, "fp32")
    if planned:
        lat.step(2)
        state = lat.read(ibm.FIELD_BODY_STATE)
        state[:, 0] += 3.4
        lat.write(ibm.FIELD_BODY_STATE, state)
    replay = _capture(lat, 2)
    lat.step(2)
    replay()
    ref = gpu_lattice(case, "fp32")
    if planned:
        ref.step(2)
        ref.write(ibm.FIELD_BODY_STATE, state)
    ref.step(4)
    assert np.array_equal(lat.f, ref.f) and np.array_equal(lat.bodies, ref.bodies)
    lat.close()
    ref.close()


def test_the_captured_grid_of_the_persistent_kernel_stays():
    """878 markers on 114 CTAs that wait at the barrier in global memory, whose
    arrival counter is a multiple of the grid: another size set between the
    replays would leave it a multiple of that one."""
    case = wl.couette(256)
    lat = gpu_lattice(case, "fp32")
    ibm.ibm_set_option(lat.h, ibm.IBM_OPT_BARRIER_LIMIT_US, 200000)
    replay = _capture(lat, 2)
    replay()
    lat.set_ib_ctas(95)
    lat.step(2)
    replay()
    lat.step(1)
    _same(lat, case, "fp32", 7)
    lat.close()


@pytest.mark.parametrize("name", sorted(CASES))
def test_first_steps_while_another_stream_is_captured(name):
    """The slices' lists are allocated by the first steps, here with cudaMalloc
    while the caller captures another stream in the strictest mode: neither
    the steps nor the capture fail."""
    import torch
    case = CASES[name]()
    alloc, release = ibm._torch_hooks if ibm.use_torch_allocator() else (None, None)
    x = torch.zeros(1000, device="cuda")
    side = torch.cuda.Stream()
    ref = gpu_lattice(case, "fp32")
    ref.step(5)
    want = (ref.f, ref.bodies)
    ref.close()
    ibm.ibm_set_allocator(None, None)
    try:
        lat = ibm.Lattice(case.nx, case.ny, case.tau, case.rho0, "fp32", case.bc, case.wall_u, case.inlet_u,
                          case.n_corr, torch_stream=False)
        for b in case.bodies:
            lat.add_markers(b.xy, b.ds, **b.as_kwargs())
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side, capture_error_mode="global"):
            x += 1
            lat.step(2, ibm.STEP_NO_GRAPH)
            x += 1
        g.replay()
        lat.step(3)
        assert np.array_equal(lat.f, want[0]) and np.array_equal(lat.bodies, want[1])
        lat.close()
    finally:
        ibm.ibm_set_allocator(alloc, release)
    torch.cuda.synchronize()
    assert bool((x == 2).all())
