"""The barrier-free correction (each CTA iterates its slice of markers with
the neighbourhood it depends on) against the launch form with one kernel per
phase: the same arithmetic per element in the same order, so every result is
bitwise the same, whatever the slices."""
import math

import numpy as np
import pytest

from _helpers import gpu_lattice
from paper_1803_09380_gb300 import ibm
from paper_1803_09380_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _rings(n, radii, spacing=1.0, at=None, **kw):
    """Fixed rings of the given radii around one point, turning alternately."""
    bodies = []
    for k, r in enumerate(radii):
        m = max(3, int(round(2 * math.pi * r / spacing)))
        c = (n / 2.0 + 0.3, n / 2.0 - 0.2) if at is None else at[k]
        xy, ds = wl.ring(c[0], c[1], r, count=m)
        bodies.append(wl.Body(xy, ds, wl.BODY_FIXED, xc=c, omega=0.01 / r * (-1) ** k, radius=r))
    return wl.Case("rings", n, n, 0.8, bodies=bodies, **kw)


CASES = {
    # two rings of 878 markers, the default slices; one slice; many
    "couette256": lambda: wl.couette(256),
    # rings 1.5 apart: every marker couples with both rings
    "near": lambda: _rings(96, (20.0, 21.5)),
    # a ring across the periodic edges
    "edge": lambda: _rings(64, (17.0,), at=[(1.2, 62.9)]),
    # half a unit apart (rows of about twenty), and markers that share no node
    "dense": lambda: _rings(96, (30.0,), spacing=0.5),
    "sparse": lambda: _rings(96, (40.0,), spacing=5.0),
    # a single marker; a bare triangle
    "one": lambda: wl.Case("one", 32, 32, 0.8, bodies=[
        wl.Body(np.array([[15.3, 16.6]]), np.ones(1), wl.BODY_FIXED, xc=(15.3, 16.6), u=(0.01, 0.005))]),
    "three": lambda: _rings(32, (2.0,), spacing=4.0),
    # closed and open sides, odd sizes; the lattice's last rows and columns in the supports
    "box": lambda: _rings(61, (27.9,), at=[(30.0, 30.0)], bc=(wl.BOUNCEBACK,) * 4, wall_u=(0,) * 6 + (0.03, 0)),
    "channel": lambda: wl.cylinder(nx=161, ny=77, diameter=20.0, center=(40.2, 38.1), markers=63),
    "channel_nee": lambda: wl.paper_cylinder(40.0, diameter=12),
    # other delta functions and iteration counts
    "delta2": lambda: _delta(2),
    "delta3": lambda: _delta(3),
    "n1": lambda: _rings(128, (25.0, 50.0), n_corr=1),
    "n2": lambda: _rings(128, (25.0, 50.0), n_corr=2),
    "n25": lambda: _rings(128, (25.0, 50.0), n_corr=25),
}


def _delta(points):
    c = _rings(96, (30.0,))
    c.delta_points = points
    return c


def _run(case, prec, steps, phases=0, ctas=0):
    lat = gpu_lattice(case, prec)
    rho, ux, uy = wl.random_fields(case.nx, case.ny, 5, du=0.01, drho=0.001)
    lat.init_equilibrium(rho, ux, uy)
    if phases:
        ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, phases)
    if ctas:
        lat.set_ib_ctas(ctas)
    lat.step(steps)
    out = (lat.f, lat.resid, lat.bodies, *lat.moments())
    lat.close()
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_slices_are_bitwise_the_phase_kernels(name, prec):
    case = CASES[name]()
    ref = _run(case, prec, 11, phases=1)
    assert np.all(np.isfinite(ref[0]))
    for got, want in zip(_run(case, prec, 11), ref):
        assert np.array_equal(got, want)


@pytest.mark.parametrize("ctas", [4, 7, 33, 152])
def test_slice_sizes_do_not_change_results(ctas):
    """878 markers in 4 slices (220 of a CTA's 256 local markers are owned:
    they do not fit, the persistent kernel runs), 7, 33 and 147."""
    case = wl.couette(256)
    ref = _run(case, "fp32", 9, phases=1)
    for got, want in zip(_run(case, "fp32", 9, ctas=ctas), ref):
        assert np.array_equal(got, want)


def test_slices_follow_added_bodies_and_marker_velocities():
    """Adding a body and prescribing velocities between steps: the slices are
    rebuilt for the new band."""
    out = []
    for phases in (0, 1):
        case = _rings(128, (25.0, 50.0))
        lat = ibm.Lattice(case.nx, case.ny, case.tau, prec="fp32")
        if phases:
            ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, phases)
        for b in case.bodies:
            lat.add_markers(b.xy, b.ds, **b.as_kwargs())
            lat.step(5)
        m = sum(len(b.xy) for b in case.bodies)
        uv = 0.01 * np.random.default_rng(3).standard_normal((m, 2))
        lat.set_marker_velocities(uv)
        lat.step(4)
        out.append((lat.f, lat.resid, lat.bodies))
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


MOVING = {
    # two disks, one free disk near a wall, prescribed motion across the periodic edge
    "pair": lambda: wl.settling_pair(nx=64, ny=130, diameter=10.0, density_ratio=1.2, gravity=2e-4),
    "wall": lambda: wl.Case("wall", 41, 90, 0.8, bc=(wl.BOUNCEBACK,) * 4,
                            bodies=[wl.disk(9.2, 70.0, 14.0, 1.3, 3e-4)]),
    "edge": lambda: _prescribed((1.3, 60.2)),
    # touching disks: nodes covered by both rings
    "touch": lambda: wl.Case("touch", 72, 72, 0.8, bc=(wl.BOUNCEBACK,) * 4,
                             bodies=[wl.disk(28.0, 36.0, 16.0, 1.2, 1e-4), wl.disk(44.6, 36.0, 16.0, 1.2, 1e-4)]),
    # a fixed ring around a free disk; 256 markers; half a unit apart (lists too long: the general path)
    "mixed": lambda: _mixed(),
    "most": lambda: _free_ring(40.0, 256),
    "dense": lambda: _free_ring(16.0, 200),
}


def _prescribed(at):
    xy, ds = wl.ring(at[0], at[1], 9.0)
    b = wl.Body(xy, ds, wl.BODY_PRESCRIBED, xc=at, u=(0.08, -0.05), omega=0.01, radius=9.0)
    return wl.Case("prescribed", 64, 61, 0.8, bodies=[b])


def _mixed():
    c = _rings(80, (30.0,))
    c.bodies.append(wl.disk(40.0, 41.0, 12.0, 1.2, 1e-4))
    return c


def _free_ring(radius, count):
    b = wl.disk(60.2, 59.7, 2 * radius, 1.2, 1e-4)
    xy, ds = wl.ring(60.2, 59.7, radius, count=count)
    b.xy, b.ds = xy, ds
    return wl.Case("free", 121, 120, 0.8, bc=(wl.BOUNCEBACK,) * 4, bodies=[b])


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", sorted(MOVING))
def test_moving_bodies_on_a_rebuilt_slice_are_bitwise_the_phase_kernels(name, prec):
    case = MOVING[name]()
    out = []
    for phases in (0, 1):
        lat = gpu_lattice(case, prec)
        if phases:
            ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, phases)
        lat.step(19)
        lat.step(1, ibm.STEP_NO_GRAPH)
        band = lat.sizes()
        # a pose written between steps, and a switch of the launch form on the way
        lat.write(ibm.FIELD_BODY_STATE, lat.read(ibm.FIELD_BODY_STATE))
        lat.step(3)
        if not phases:
            ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, 1)
        lat.step(2)
        out.append((lat.f, lat.resid, lat.bodies, lat.markers, np.array(band), *lat.moments()))
        lat.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def _window_counts(xy):
    """Most markers that cover a node, and most markers that one couples with
    (4 x 4 windows from floor(X) - 1 on, away from the sides)."""
    o = np.floor(xy).astype(int) - 1
    near = np.abs(o[:, None, :] - o[None, :, :])
    rows = int(np.max(np.sum(np.all(near <= 3, axis=2), axis=1)))
    grid = np.zeros(o.max(axis=0) + 4, int)
    for x, y in o:
        grid[x:x + 4, y:y + 4] += 1
    return int(grid.max()), rows


def _plates(k, at=((32.4, 31.3), (30.45, 29.35), (34.35, 31.4))):
    """Three plates of k x k markers two units apart in relative motion.  A node
    is covered by at most four markers of a plate; a marker couples with nine
    of its own plate and, as the window origins fall, with 9, 12 or 16 of each
    other: at most 41, more than the lists' 32 rows in some poses."""
    g = 2.0 * np.arange(k) - (k - 1)
    xy = np.stack(np.meshgrid(g, g), -1).reshape(-1, 2)
    bodies = []
    for xc, u in zip(at, ((0.0, 0.0), (0.13, 0.02), (-0.03, 0.11))):
        bodies.append(wl.Body(xy + xc, np.ones(k * k), wl.BODY_PRESCRIBED, xc=xc, u=u, radius=float(k)))
    return wl.Case("plates", 64, 64, 0.8, bodies=bodies)


def _crossing(r, m):
    """Four rings on their way to one point: apart, at most six markers cover a
    node; where they cross, up to 24, more than the lists hold."""
    bodies = []
    for dx, dy in ((-1, 0), (1, 0), (0, -1), (0, 1)):
        at = (32.3 + (r + 2.2) * dx, 32.7 + (r + 2.2) * dy)
        xy, ds = wl.ring(at[0], at[1], r, count=m)
        bodies.append(wl.Body(xy, ds, wl.BODY_PRESCRIBED, xc=at, u=(-0.1 * dx, -0.1 * dy), radius=r))
    return wl.Case("crossing", 64, 64, 0.8, bodies=bodies)


@pytest.mark.parametrize("prec,make,limit", [
    ("fp32", lambda: _plates(7), (12, 32)), ("fp64", lambda: _plates(5), (12, 32)),
    ("fp32", lambda: _crossing(6.4, 40), (12, 32)), ("fp64", lambda: _crossing(4.0, 25), (12, 32))])
def test_moving_bodies_in_and_out_of_what_the_slice_holds(prec, make, limit):
    """Poses whose covering lists or rows do not fit the slice's take the general
    path inside the same three launches a step, and the next pose that fits
    comes back: every step bitwise the phase kernels."""
    fast, ref = gpu_lattice(make(), prec), gpu_lattice(make(), prec)
    ibm.ibm_set_option(ref.h, ibm.IBM_OPT_IB_PHASES, 1)
    fit = []
    for k in range(28):
        if k == 14:                      # the way back
            for lat in (fast, ref):
                s = lat.read(ibm.FIELD_BODY_STATE)
                s[:, 2:5] *= -1.0
                lat.write(ibm.FIELD_BODY_STATE, s)
        cover, rows = _window_counts(fast.markers)
        fit.append(cover <= limit[0] and rows <= limit[1])
        l0 = fast.counters()[0]
        fast.step(1)
        ref.step(1)
        assert fast.counters()[0] - l0 == 3
        assert np.array_equal(fast.bodies, ref.bodies) and np.array_equal(fast.resid, ref.resid)
    assert fit[0] and fit[-1] and not all(fit)
    assert np.all(np.isfinite(ref.f)) and np.array_equal(fast.f, ref.f)
    assert np.array_equal(fast.markers, ref.markers)
    fast.close()
    ref.close()


# bodies on the slice (3 launches a step) and on the general path (collide+stream,
# correction, band collide, body update, marker move, six of the band: 11)
FORMS = {
    "fp32 256 markers": ("fp32", lambda: _free_ring(40.0, 256), 3),
    "fp32 257 markers": ("fp32", lambda: _free_ring(40.0, 257), 11),
    "fp64 128 markers": ("fp64", lambda: _free_ring(20.0, 128), 3),
    "fp64 129 markers": ("fp64", lambda: _free_ring(20.0, 129), 11),
    # lists too short from the first pose on: five units apart (16 nodes a marker),
    # a third of a unit apart (17 markers on a node), 41 coupled markers
    "sparse": ("fp32", lambda: _free_ring(32.0, 40), 11),
    "covered": ("fp32", lambda: _free_ring(11.0, 210), 11),
    "rows": ("fp32", lambda: _plates(7, ((32.4, 31.3), (31.4, 30.3), (31.4, 32.3))), 11),
}


@pytest.mark.parametrize("name", sorted(FORMS))
def test_moving_bodies_run_the_form_that_their_first_pose_fits(name):
    prec, make, launches = FORMS[name]
    fast, ref = gpu_lattice(make(), prec), gpu_lattice(make(), prec)
    ibm.ibm_set_option(ref.h, ibm.IBM_OPT_IB_PHASES, 1)
    for n in (1, 8, 2):
        l0 = fast.counters()[0]
        fast.step(n)
        assert fast.counters()[0] - l0 == launches * n
        ref.step(n)
    assert np.array_equal(fast.f, ref.f) and np.array_equal(fast.bodies, ref.bodies)
    assert np.array_equal(fast.resid, ref.resid) and np.array_equal(fast.markers, ref.markers)
    fast.close()
    ref.close()


@pytest.mark.parametrize("count,ctas,slices", [(256, 1, True), (257, 1, False), (513, 2, False)])
def test_slices_too_large_to_hold_their_own_markers_are_not_tried(count, ctas, slices):
    """As many CTAs as the per-case server pins for so many markers: above 256 a
    CTA the first step allocates nothing and runs the persistent kernel."""
    xy, ds = wl.ring(60.2, 59.7, count / (2 * math.pi), count=count)
    case = wl.Case("ring", 256, 256, 0.8, bodies=[
        wl.Body(xy + 64.0, ds, wl.BODY_FIXED, xc=(124.2, 123.7), omega=2e-4, radius=10.0)])
    assert ibm.use_torch_allocator()
    alloc, release = ibm._torch_hooks
    sizes = []

    def counted(nbytes, device, stream, ctx):
        sizes.append(nbytes)
        return alloc(nbytes, device, stream, ctx)
    hook = ibm._ALLOC_FN(counted)
    lat = gpu_lattice(case, "fp32")
    lat.set_ib_ctas(ctas)
    ibm.ibm_set_allocator(hook, release)
    try:
        lat.step(1)
        lat.sync()
    finally:
        ibm.ibm_set_allocator(alloc, release)
    assert bool(sizes) == slices
    lat.close()


def test_server_counts_the_slices_in_the_memory_of_a_case():
    """The first step of a served case allocates its slices' lists, 349 KB each
    in FP64: 16 slices of 16 markers against one slice of 256."""
    xy, ds = wl.ring(64.2, 63.7, 40.0, count=256)
    case = wl.Case("ring", 128, 128, 0.8, bodies=[
        wl.Body(xy, ds, wl.BODY_FIXED, xc=(64.2, 63.7), omega=2e-4, radius=40.0)])
    held = []
    for per_cta in (16, 256):
        with ibm.Server(max_active=1, steps_per_launch=4, ib_markers_per_cta=per_cta) as srv:
            i = srv.submit(case, 40, prec="fp64")
            srv.progress()
            held.append(srv.stats()["device_bytes"])
            srv.wait(i)
            assert srv.stats()["device_bytes"] == 0
    assert 15 * 340e3 < held[0] - held[1] < 15 * 360e3


@pytest.mark.parametrize("name", ["couette", "pair"])
def test_autotuner_tries_the_default_choice(name):
    """The default candidates: the library's own choice of slices (0), 1, 8 and 16
    CTAs, 1/2, 3/4 and all of the SMs, each for 2 + 4 steps."""
    import torch
    make = (lambda: wl.couette(96)) if name == "couette" else MOVING["pair"]
    lat = gpu_lattice(make(), "fp32")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    candidates = {0, 1, 8, 16, sms // 2, (3 * sms + 3) // 4, sms}
    best, us = lat.autotune_ib(None, steps_each=4)
    assert best in candidates and us > 0
    assert lat.counters()[1] == 6 * len(candidates)
    ref = gpu_lattice(make(), "fp32")
    ref.step(6 * len(candidates))
    assert np.array_equal(lat.f, ref.f) and np.array_equal(lat.bodies, ref.bodies)
    lat.close()
    ref.close()


def test_launches_are_counted_where_a_step_does_not_fit_one_grid():
    """16 x 65535 nodes between walls: edge rows and lattice rows of the odd step
    go as two launches, and with markers the step forks (slices, band segments,
    collide+stream)."""
    def make(bodies):
        return wl.Case("tall", 16, 65535, 0.8, bc=(wl.BOUNCEBACK,) * 4, wall_u=(0,) * 6 + (0.03, 0), bodies=bodies)
    xy, ds = wl.ring(7.6, 65520.3, 4.0, count=25)
    ring = wl.Body(xy, ds, wl.BODY_FIXED, xc=(7.6, 65520.3), omega=1e-3, radius=4.0)
    for bodies, even, odd in (([], 1, 2), ([ring], 3, 4)):
        out = []
        for phases in (0, 1):
            lat = gpu_lattice(make(bodies), "fp32")
            ibm.ibm_set_option(lat.h, ibm.IBM_OPT_IB_PHASES, phases)
            for n, want in ((1, even), (1, odd), (9, 5 * even + 4 * odd)):
                l0 = lat.counters()[0]
                lat.step(n)
                if not phases:
                    assert lat.counters()[0] - l0 == want
            out.append((lat.f, lat.bodies, lat.resid))
            lat.close()
        for a, b in zip(*out):
            assert np.all(np.isfinite(a)) and np.array_equal(a, b)


def _launches(lat):
    l0 = lat.counters()[0]
    lat.step(2)
    return (lat.counters()[0] - l0) // 2


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "bf16"])
def test_the_cases_above_run_on_slices(prec):
    """What is compared with the phase kernels above is the slices: two launches a
    step with fixed markers, three with moving ones.  FP64 holds 128 moving
    markers: the three cases with more run the general path."""
    for name in sorted(CASES):
        assert _launches(gpu_lattice(CASES[name](), prec)) == 2, name
    for name in sorted(MOVING):
        general = prec == "fp64" and name in ("mixed", "most", "dense")
        assert _launches(gpu_lattice(MOVING[name](), prec)) == (11 if general else 3), name
