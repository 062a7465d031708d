"""The double-float step (csrc/pair.cuh): its arithmetic, rates and trajectories on the host
against long double, and on the GPU GT_MODE_FP64's route through it against the FP64 kernels.
"""
import json
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2310_15183_gb300 import build
from paper_2310_15183_gb300 import workloads as W

from .parity import neighbour_band, rel_err, to_numpy

HERE = os.path.dirname(os.path.abspath(__file__))


def test_pair_arithmetic_rates_and_trajectories(tmp_path):
    """u = 2^-24, operands with |lo| <= u |hi|.  Product: four roundings of an error term of
    at most 3 u; sum: two roundings of low parts of at most 3 u; fused: both.  Reciprocal and
    root: a residual of a few u rounded a few times.  exp: the argument's own last bits
    (2^-48 of 8) and the sum's; sin/cos: absolute, a handful of u^2.  The rates are held to
    the renormalised double-float's (equal work on equal inputs, a factor of two for the
    sample), and where the multipole tails replace cancelling differences to FP64's own.
    Whole trajectories are held to FP64's: the three-float state has no rounding per step."""
    exe = str(tmp_path / "pair_arith")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I" + cuda_inc,
                    os.path.join(HERE, "pair_arith.cpp"), "-o", exe], check=True)
    res = json.loads(subprocess.run([exe], check=True, capture_output=True, text=True).stdout)
    u2 = 2.0 ** -48
    assert res["mul"] <= 12 * u2 and res["add"] <= 6 * u2 and res["fma"] <= 18 * u2, res
    assert res["rcp"] <= 8 * u2 and res["rsqrt"] <= 12 * u2, res
    assert res["exp"] <= 2.0 ** -44 and res["sincos"] <= 2.0 ** -46, res
    assert res["tf_add"] <= 2.0 ** -61, res
    assert res["rotate"] <= 2.0 ** -46, res  # absolute, as sincos: a handful of u^2
    for name, r in res["rates"].items():
        if name:
            assert r["n"] >= 5000, (name, r)
            assert r["pair"][0] <= 2 * r["df"][0] and r["pair"][1] <= 2 * r["df"][1], (name, r)
    assert res["rates"]["mn outside"]["pair"][0] <= res["rates"]["mn outside"]["f64"][0], res
    for name, r in res["frames"].items():
        if name:
            assert all(p <= f for p, f in zip(r["pair"], r["f64"])), (name, r)


# M, S, Q, r0, theta0, fov, nx, ny, steps, sp, options
FORMS = {
    "schwarzschild": (0.5, 0.0, 0.0, 10.0, math.pi / 2, 75.0, 33, 17, 2000, 1.5e-4, {}),
    "kerr to the end": (0.5, 0.225, 0.0, 15.0, 1.4, 40.0, 21, 15, 200000, 1e-3, {}),
    "retrograde, near extremal": (0.5, -0.2475, 0.0, 8.0, 0.6, 75.0, 9, 7, 20000, 1e-3, {}),
    "near the axis": (0.5, 0.2, 0.0, 10.0, 1e-3, 75.0, 9, 7, 1500, 1e-3, {}),
    "wide field": (0.5, 0.2, 0.0, 10.0, 1.2, 179.0, 9, 7, 2000, 1e-3, {}),
    "one pixel": (0.5, 0.24, 2.0, 15.0, 1.4, 75.0, 1, 1, 3000, 1.5e-4, {}),
    "one column, listing's weights and camera": (0.5, 0.24, 2.0, 15.0, 1.1, 75.0, 1, 7, 3000,
                                                1.5e-4, {"flags": 3}),
    "mn": (0.5, 0.24, 2.0, 15.0, 1.4, 75.0, 24, 16, 20000, 1.5e-4, {}),
    "mn oblate the other way, low spin": (0.5, 0.025, -2.0, 15.0, 1.4, 75.0, 13, 9, 5000, 1e-3, {}),
    "mn inside the zone": (0.5, 0.24, 2.0, 1.9, 1.4, 75.0, 13, 9, 2000, 1.5e-4, {}),
    "small unit of length": (1e-3, 0.45e-6, 0.0, 0.03, 1.4, 75.0, 9, 7, 3000, 1e-6, {}),
    "large unit of length": (500.0, 1.2e5, 0.0, 15000.0, 1.4, 75.0, 9, 7, 3000, 0.9, {}),
    "mn in large units": (500.0, 0.24e6, 2.0, 15000.0, 1.4, 75.0, 9, 7, 3000, 0.9, {}),
    "smallest step": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 5, 3, 300, 1e-9, {}),
    "coarse steps": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 9, 7, 200, 0.5, {}),
    "one ray per thread": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 33, 17, 2000, 1e-3,
                           {"flags": 4, "block_size": 64}),
    "graph": (0.5, 0.24, 2.0, 15.0, 1.2, 75.0, 33, 17, 1000, 1e-3, {"flags": 8}),
}
OUTSIDE = {
    "step above the range": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 9, 7, 100, 1.5, {}),
    "mass above the range": (2e3, 1e6, 0.0, 6e4, 1.2, 75.0, 9, 7, 300, 0.9, {}),
    "paper numerics": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 9, 7, 300, 1e-3, {"flags": 32}),
    "explicit Euler": (0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 9, 7, 300, 1e-3, {"flags": 128}),
}


@pytest.fixture(scope="module")
def tracer():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    from paper_2310_15183_gb300 import geotrace
    t = geotrace.Tracer(0)
    yield t
    t.close()


def _both_routes(tracer, form):
    """The frame through gt_trace, and through the FP64 kernel: gt_trace_disk with a ring
    that no ray meets."""
    M, S, Q, r0, th0, fov, nx, ny, steps, sp, opts = form
    tracer.set_spacetime(M, S, Q)
    tracer.set_camera(r0, th0, fov, nx, ny)
    tracer.set_options(**opts)
    got = to_numpy(tracer.trace(steps, sp, 0))
    ref = to_numpy(tracer.trace_disk(1e12, 2e12, 1e-9, steps, sp, 0))
    tracer.set_options()
    return got, ref


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(FORMS))
def test_fp64_route_against_the_fp64_kernel(tracer, name):
    """Every form the double-float route accepts: the same status and step count, the end
    position within the project's parity tolerance of 1e-9 (relative, per component) -- away
    from the shadow's edge and the axis, where the flow amplifies both routes' rounding."""
    form = FORMS[name]
    got, ref = _both_routes(tracer, form)
    keep = ~neighbour_band(ref["status"], form[6], form[7])
    assert keep.sum() > 0
    assert np.array_equal(got["status"][keep], ref["status"][keep])
    assert np.array_equal(got["nsteps"][keep], ref["nsteps"][keep])
    for k in ("t", "r", "th", "ph"):
        assert np.max(rel_err(got[k], ref[k])[keep]) <= 1e-9, k


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(OUTSIDE))
def test_other_fp64_calls_keep_the_fp64_kernel(tracer, name):
    got, ref = _both_routes(tracer, OUTSIDE[name])
    for k in ("t", "r", "th", "ph", "status", "nsteps"):
        assert np.array_equal(got[k], ref[k], equal_nan=k not in ("status", "nsteps")), k


@pytest.mark.gpu
def test_batch_of_both_kinds_and_pixel_lists(tracer):
    """A batch of Kerr and Manko-Novikov cameras (the per-camera kernel) and an all-Kerr one
    against single traces: 1e-9 and bit for bit; a pixel list and a range bit for bit."""
    torch = pytest.importorskip("torch")
    cams = [W.Camera(0.5, 0.1, 0.0, 12.0, 0.7, 75.0, 13, 9),
            W.Camera(0.5, 0.24, 2.0, 15.0, 1.3, 75.0, 7, 6),
            W.Camera(0.5, -0.2, 0.0, 9.0, 1.2, 75.0, 21, 3)]
    for group, exact in ((cams, False), (cams[::2], True), (cams[1:2], True)):
        out = to_numpy(tracer.trace_batch(group, 3000, 1e-3, 0))
        off = 0
        for c in group:
            tracer.set_spacetime(c.M, c.S, c.Q)
            tracer.set_camera(c.r0, c.theta0, c.fov_deg, c.res_x, c.res_y)
            one = to_numpy(tracer.trace(3000, 1e-3, 0))
            for k in one:
                part = out[k][off:off + c.n_rays]
                if exact or k in ("status", "nsteps"):
                    assert np.array_equal(part, one[k]), k
                else:
                    assert np.max(rel_err(part, one[k])) <= 1e-9, k
            off += c.n_rays
    pix = torch.tensor([0, 5, 17, 41], dtype=torch.int64, device="cuda")
    c = cams[1]
    tracer.set_spacetime(c.M, c.S, c.Q)
    tracer.set_camera(c.r0, c.theta0, c.fov_deg, c.res_x, c.res_y)
    full = to_numpy(tracer.trace(1000, 1e-3, 0))
    some = to_numpy(tracer.trace_pixels(pix, 1000, 1e-3, 0))
    part = to_numpy(tracer.trace_range(3, 20, 1000, 1e-3, 0))
    for k in full:
        assert np.array_equal(some[k], full[k][pix.cpu().numpy()]), k
        assert np.array_equal(part[k], full[k][3:23]), k
