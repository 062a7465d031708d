"""The FP32-mixed kernel's back-to-back steps (csrc/trace.cu): rays whose steps end in every
possible event -- exits, the cap, the zone, re-projection, the ring, stage angles beyond the
series -- within one warp, against the same rays traced alone and against the FP64 mode."""
import math

import numpy as np
import pytest

from paper_2310_15183_gb300 import workloads as W

from .parity import mixed_report, neighbour_band, to_numpy

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
KEYS = ("t", "r", "th", "ph", "status", "nsteps")


@pytest.fixture(scope="module")
def tracer():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15183_gb300 import build, geotrace
    build.build()
    t = geotrace.Tracer(0)
    yield t
    t.close()


# M, S, Q, r0, theta0, fov, nx, ny, steps, sp, options
FORMS = {
    "escape, horizon and cap": (0.5, 0.2, 0.0, 8.0, 1.3, 60.0, 9, 7, 9000, 2e-3, {}),
    "re-projection every step": (0.5, 0.2, 0.0, 8.0, 1.3, 60.0, 9, 7, 3000, 2e-3,
                                 {"reproject_every": 1}),
    "re-projection between caps": (0.5, 0.2, 0.0, 8.0, 1.3, 60.0, 9, 7, 1001, 2e-3,
                                   {"reproject_every": 333}),
    "zone hand-overs": (0.5, 0.24, 2.0, 6.0, 1.3, 75.0, 9, 7, 6000, 2e-3, {}),
    "through the axis": (0.5, 0.1, 0.0, 8.0, 0.02, 75.0, 9, 7, 3000, 5e-3, {}),
    "one step": (0.5, 0.24, 2.0, 15.0, 1.3, 75.0, 5, 3, 1, 1.5e-4, {}),
    "128 steps": (0.5, 0.24, 2.0, 15.0, 1.3, 75.0, 5, 3, 128, 1.5e-4, {}),
    "129 steps": (0.5, 0.24, 0.0, 15.0, 1.3, 75.0, 33, 1, 129, 1.5e-4, {}),
    "coarse steps": (0.5, 0.1, 0.0, 8.0, 0.4, 75.0, 9, 7, 60, 0.7, {}),
}


@pytest.mark.parametrize("name", sorted(FORMS))
def test_rays_do_not_depend_on_their_warp(tracer, name):
    """A ray of a warp full of other rays, and the same ray in a launch of its own (its warp
    runs no other lane's events): the same bits, step counts and statuses."""
    M, S, Q, r0, th0, fov, nx, ny, steps, sp, opts = FORMS[name]
    tracer.set_spacetime(M, S, Q)
    tracer.set_camera(r0, th0, fov, nx, ny)
    tracer.set_options(**opts)
    full = to_numpy(tracer.trace(steps, sp, 1))
    for k in range(0, nx * ny, max(1, nx * ny // 9)):
        one = to_numpy(tracer.trace_range(k, 1, steps, sp, 1))
        for key in KEYS:
            assert np.array_equal(one[key], full[key][k:k + 1], equal_nan=True), (name, k, key)
    assert np.all(full["nsteps"] >= 1) and np.all(full["nsteps"] <= steps)


def test_ring_is_tested_after_every_step(tracer):
    """With a ring as an exit the step loop stops after each step: hits on the step the FP64
    mode hits on, for rays that cross the ring plane once at a steep angle."""
    tracer.set_spacetime(0.5, 0.2, 0.0)
    tracer.set_camera(10.0, 0.6, 60.0, 16, 12)
    tracer.set_options()
    out = [to_numpy(tracer.trace_disk(1.5, 4.0, 0.05, 20000, 1e-3, mode)) for mode in (0, 1)]
    hit = out[0]["status"] == 5
    assert hit.sum() > 20
    assert np.mean(out[0]["status"] == out[1]["status"]) >= 0.999
    both = hit & (out[1]["status"] == 5)
    assert np.max(np.abs(out[0]["nsteps"][both].astype(int) - out[1]["nsteps"][both].astype(int))) <= 1


def test_watchdog_stops_the_step_loop(tracer):
    """A launch of minutes under a 0.2 s limit returns the timeout code; the context goes on."""
    from paper_2310_15183_gb300 import geotrace as g
    cam = W.sub_camera(W.MN_1000, 64, 64)
    tracer.set_spacetime(0.5, 0.2, 0.0)
    tracer.set_camera(1e4, cam.theta0, 75.0, 512, 512)
    tracer.set_options(timeout_seconds=0.2)
    with pytest.raises(g.GeotraceError) as e:
        tracer.trace(1 << 31, 1e-6, 1)
    assert e.value.code == -5
    tracer.set_options()
    tracer.set_camera(15.0, 1.2, 75.0, 8, 8)
    assert np.all(to_numpy(tracer.trace(100, 1.5e-4, 1))["nsteps"] == 100)


@pytest.mark.parametrize("flags", [0, 16])
@pytest.mark.parametrize("n", [1, 33, 200])
def test_rays_of_either_kind_with_their_own_spacetimes(tracer, n, flags):
    """Kerr and Manko-Novikov rays side by side in a warp: the bits of each ray in a launch of
    its own, and the FP64 mode by the mixed mode's criterion of 1e-3 rad."""
    a = list(W.surrogate_samples(n, seed=3, q_max=2.0))
    a[3] = np.where(np.arange(n) % 3 == 0, 0.0, a[3])
    dev = [torch.tensor(v, device="cuda") for v in a]
    tracer.set_options(flags=flags)

    def rays(sel, mode):
        return to_numpy(tracer.trace_rays(*[d[sel].contiguous() for d in dev], M=0.5, r0=15.0,
                                          n_steps=600, step_precision=2e-2, mode=mode))

    full, ref = rays(slice(None), 1), rays(slice(None), 0)
    for k in range(0, n, max(1, n // 9)):
        one = rays(slice(k, k + 1), 1)
        for key in KEYS:
            assert np.array_equal(one[key], full[key][k:k + 1], equal_nan=True), (k, key)
    far = ref["r"] > 4.0
    rep = mixed_report({k: v[far] for k, v in full.items()}, {k: v[far] for k, v in ref.items()})
    assert far.sum() >= 0.8 * n and rep["agree"] >= 0.999 and rep["max_angle"] <= 1e-3, rep


@pytest.mark.parametrize("exponent", [-20, -9, 9, 11, 20])
@pytest.mark.parametrize("Q", [0.0, 2.0])
def test_units_of_length_on_both_sides_of_the_range(tracer, Q, exponent):
    """Camera rays of ordinary scale run the flush-to-zero build of the FP32 kernel, other units
    of length the one that keeps denormals (the line lies at M = 1e-3 and 1e3): frames of
    either against the FP64 mode by the mixed mode's criteria, statuses of 99.9 % and end angles
    within 1e-3 rad away from the shadow's edge.  (The pixel grid is not the same in every unit:
    at 2^-11 its rays pass through the axis, where the two modes part.)"""
    u = 2.0 ** exponent
    nx, ny = 24, 18
    tracer.set_spacetime(u, 0.48 * u * u, Q)  # S is an area, Q a pure number
    tracer.set_camera(20.0 * u, 1.2, 60.0, nx, ny)
    tracer.set_options()
    ref, got = [to_numpy(tracer.trace(4000, 2e-2 * u, mode)) for mode in (0, 1)]
    band = neighbour_band(ref["status"], nx, ny) | (ref["r"] < 4.0 * u)
    rep = mixed_report(got, ref, exclude=band)
    assert rep["n"] > 100 and rep["agree"] >= 0.999 and rep["max_angle"] <= 1e-3, rep
