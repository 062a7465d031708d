"""The double-float step at the limits of what it accepts (csrc/pair.cuh): on the host the
kernels' own step, on the GPU the routes that lead to it."""
import concurrent.futures
import json
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2310_15183_gb300 import build

from .parity import to_numpy

HERE = os.path.dirname(os.path.abspath(__file__))


# steps, step / M, r0 / M from and to, theta0 from and to, frames, whether pairs are taken
ACCURACY = {
    "a few steps": (10, 3e-4, 15, 50, 0.3, 1.5, 24, False),
    "hundreds of steps": (500, 3e-4, 15, 50, 0.3, 1.5, 24, False),
    "fewest steps": (1000, 3e-4, 8.5, 30, 0.3, 1.5, 24, True),
    "fewest steps, farthest camera": (1000, 3e-4, 30, 49, 0.3, 1.5, 24, True),
    "the workloads' step": (2000, 3e-4, 15, 60, 0.3, 1.5, 24, True),
    "shortest path": (2000, 7.6e-5, 8.5, 30, 0.3, 1.5, 24, True),
    "shortest path, far camera": (4000, 7.6e-5, 40, 60, 0.3, 1.5, 24, True),
    "too short a path": (2000, 1e-6, 8.5, 60, 0.3, 1.5, 24, False),
    "coarsest steps": (1000, 2e-3, 8.5, 30, 0.3, 1.5, 24, True),
    "coarse steps": (100, 0.2, 10, 30, 0.3, 1.5, 24, False),
    "coarse steps, long paths": (6000, 8e-3, 8.5, 25, 0.9, 1.5, 24, False),
    "far camera": (6000, 3e-4, 60, 180, 0.3, 1.5, 12, True),
    "too far a camera": (1000, 1e-4, 200, 2000, 0.3, 1.5, 24, False),
    "near the axis": (2000, 3e-4, 8.5, 60, 1e-3, 0.3, 24, True),
    "near the axis, coarsest": (1500, 2e-3, 5, 45, 1e-3, 0.3, 24, True),
}


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("pair") / "pair_route")
    cuda_inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I" + cuda_inc,
                    os.path.join(HERE, "pair_route.cpp"), "-o", exe], check=True)

    def run(*args):
        return json.loads(subprocess.run([exe, *map(str, args)], check=True, capture_output=True,
                                         text=True).stdout)
    return run


def test_a_step_whose_new_state_is_not_finite_is_refused(host):
    """NONFINITE keeps the last finite state: the step leaves the ray as it was and hands it to
    the FP64 step, also where every rate was finite and only the increments overflow."""
    r = host("new_state")
    assert r["n"] == 64 and r["refused"] == r["untouched"] == r["taken"] == r["n"], r


def test_operations_over_the_range_the_step_gives_them(host):
    """exp: the argument's low part, at most 2^-24 |x|, is rounded three times (3 |x| 2^-49), the
    series and the table cost 2^-45; sin/cos and the rotation as on their inner ranges, 2^-46."""
    r = host("operations")
    assert r["exp"] <= 1.0 and r["sincos"] <= 2.0 ** -46 and r["rotate"] <= 2.0 ** -46, r


WHOLE_PATHS = (22000, 2e-3, 8.5, 25, 0.9, 1.5, 12)


@pytest.fixture(scope="module")
def accuracy(host):
    rows = {**{k: v[:-1] for k, v in ACCURACY.items()}, "whole paths": WHOLE_PATHS}
    with concurrent.futures.ThreadPoolExecutor(os.cpu_count()) as ex:
        jobs = {k: ex.submit(host, "accuracy", *v) for k, v in rows.items()}
        return {k: j.result() for k, j in jobs.items()}


@pytest.mark.parametrize("name", sorted(ACCURACY))
def test_fp64_mode_is_as_accurate_as_fp64_arithmetic(accuracy, name):
    """GT_MODE_FP64's end positions against long double, by the step the kernels would take
    there, are no further off than FP64 steps', t, r, theta and phi each: both are random sums,
    so a quarter is left for the sample, and a ulp of the outputs for their own rounding."""
    r = accuracy[name]
    assert r["pairs"] == (ACCURACY[name][-2] if ACCURACY[name][-1] else 0), r
    for got, f64 in zip(r["route"], r["f64"]):
        assert got <= 1.25 * f64 + 2.0 ** -53, r


def test_fp64_mode_is_as_accurate_as_fp64_arithmetic_over_whole_paths(accuracy):
    """To the escape or the horizon some rays pass the photon orbits, which amplify either
    arithmetic's rounding a millionfold: the mean over frames is the geometric one, of the
    ratio of the two errors."""
    r = accuracy["whole paths"]
    assert r["pairs"] == WHOLE_PATHS[-1] and max(r["ratio"]) <= 1.25, r


def test_benchmark_names_the_kernel_that_runs(host):
    """bench.py's roofline is of the launched kernel: Manko-Novikov alone has its constants as
    kernel parameters, two rays a thread are a kernel of their own, and GT_MODE_FP64 takes pairs
    by the kernels' rule."""
    import bench
    from paper_2310_15183_gb300 import workloads as W
    mn = W.WORKLOADS["mn1000"]
    kerr = W.Camera(0.5, 0.2, 0.0, 15.0, 1.2, 75.0, 8, 8)
    assert bench.trace_kernel_name(mn.camera, mn, True, 1) == "trace_kernel<2,1,0,1>"
    assert bench.trace_kernel_name(kerr, mn, True, 1) == "trace_kernel<2,0,0,0>"
    assert bench.trace_kernel_name(kerr, mn, True, 2) == "trace2_kernel<0,0>"
    assert bench.trace_kernel_name(mn.camera, mn, False, 1) == "pair_kernel<5,1,1>"
    for M, r0, sp, n in ((0.5, 15, 1.5e-4, 1000), (0.5, 15, 1.5e-4, 999), (0.5, 25.1, 3e-4, 1000),
                         (0.5, 25, 3e-4, 1000), (0.5, 20, 9.9e-5, 1000), (0.5, 20, 1.01e-4, 1000),
                         (0.5, 15, 1.01e-3, 20000), (0.5, 15, 1e-5, 5000), (0.5, 501, 1e-4, 10 ** 6)):
        cam, wl = W.Camera(M, 0.0, 0.0, r0, 1.2, 75.0, 8, 8), W.Workload("x", None, n, sp)
        assert bench.fp64_takes_pairs(cam, wl) == bool(host("rule", M, r0, sp, n)), (M, r0, sp, n)


# ------------------------------------------------------------------ on the GPU
# M, S, Q, r0, theta0, nx, ny, steps, step: calls that take FP64 steps
FP64_CALLS = {
    "one step": (0.5, 0.2, 0.0, 10.0, 1.2, 9, 7, 1, 1.5e-4),
    "999 steps": (0.5, 0.24, 2.0, 15.0, 1.2, 9, 7, 999, 1.5e-4),
    "step above 2e-3 M": (0.5, 0.2, 0.0, 10.0, 1.2, 9, 7, 2000, 1.001e-3),
    "coarse steps": (0.5, 0.24, 2.0, 10.0, 1.2, 9, 7, 200, 0.3),
    "short path": (0.5, 0.2, 0.0, 10.0, 1.2, 9, 7, 1000, 7e-5),
    "far camera": (0.5, 0.2, 0.0, 25.1, 1.2, 9, 7, 1000, 3e-4),
    "short path for the distance": (0.5, 0.2, 0.0, 20.0, 1.2, 9, 7, 1000, 9.9e-5),
    "large unit of length": (500.0, 1e5, 0.0, 10000.0, 1.2, 9, 7, 1000, 1.01),
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


def _both(tracer, M, S, Q, r0, th0, nx, ny, steps, sp):
    """gt_trace, and the FP64 kernel: gt_trace_disk with a ring that no ray meets."""
    tracer.set_spacetime(M, S, Q)
    tracer.set_camera(r0, th0, 75.0, nx, ny)
    tracer.set_options()
    return (to_numpy(tracer.trace(steps, sp, 0)),
            to_numpy(tracer.trace_disk(1e12, 2e12, 1e-9, steps, sp, 0)))


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(FP64_CALLS))
def test_calls_outside_the_rule_take_fp64_steps(tracer, name):
    got, ref = _both(tracer, *FP64_CALLS[name])
    for k in ("t", "r", "th", "ph", "status", "nsteps"):
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.gpu
def test_calls_at_the_edge_of_the_rule_take_pairs(tracer):
    """1000 steps, of 2e-3 M: bits of their own, the end position within 1e-13 of FP64's."""
    got, ref = _both(tracer, 0.5, 0.2, 0.0, 10.0, 1.2, 9, 7, 1000, 1e-3)
    assert not np.array_equal(got["ph"], ref["ph"])
    for k in ("t", "r", "th", "ph"):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-13 * np.max(np.abs(ref[k])), k


@pytest.mark.gpu
@pytest.mark.parametrize("Q", [0.0, 2.0])
def test_steps_near_the_axis_are_fp64(tracer, Q):
    """A camera on the axis whose rays stay within 1000 step lengths of it (rho <= 0.01 + 0.8 in
    1000 steps of 1e-3): FP64's steps one for one, up to the rounding of two builds of one
    formula, 1e-15 a step, times what the axis amplifies (1 / theta of the closest, 1e2)."""
    got, ref = _both(tracer, 0.5, 0.2, Q, 10.0, 1e-3, 9, 7, 1000, 1e-3)
    assert np.array_equal(got["status"], ref["status"])
    for k in ("t", "r", "th"):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-12 * np.max(np.abs(ref[k])), k


def _cameras():
    from paper_2310_15183_gb300 import workloads as W
    near = W.Camera(0.5, 0.2, 0.0, 10.0, 1.2, 75.0, 9, 7)
    return {"distant": [near, W.Camera(0.5, 0.1, 0.0, 2e5, 1.2, 1.0, 5, 3), near],
            "heavy first": [W.Camera(2e3, 1e6, 0.0, 6e4, 1.2, 75.0, 5, 3), near],
            "both kinds": [near, W.Camera(0.5, 0.24, 2.0, 15.0, 1.3, 75.0, 7, 6),
                           W.Camera(0.5, 0.24, 2.0, 2e5, 1.3, 1.0, 3, 3),
                           W.Camera(0.5, 0.1, 0.0, 2e5, 1.2, 1.0, 5, 3)]}


@pytest.mark.gpu
@pytest.mark.parametrize("mode,flags", [(0, 0), (0, 4), (0, 8), (1, 0), (1, 4), (1, 8)])
@pytest.mark.parametrize("name", sorted(_cameras()))
def test_a_cameras_bits_do_not_depend_on_its_batch_mates(tracer, name, mode, flags):
    """Cameras of a batch that take different kernels -- one beyond the double-float and
    flush-to-zero ranges among others inside -- give the bits of a batch of their own route,
    through the direct launch, one ray per thread, and a graph replayed twice."""
    cams = _cameras()[name]
    steps, sp = 1500, 1e-3
    inside = [c.M <= 1e3 and c.r0 <= 1e5 for c in cams]
    tracer.set_options(flags=flags)
    out = tracer.alloc_outputs(sum(c.n_rays for c in cams))
    for _ in range(2):
        for v in out.values():
            v.fill_(77)
        tracer.trace_batch(cams, steps, sp, mode, out)
    got = to_numpy(out)
    off = np.cumsum([0] + [c.n_rays for c in cams])
    for part in (True, False):
        mine = [i for i, v in enumerate(inside) if v == part]
        # a camera of each kind in the group, so that it runs the same per-camera kernel
        alone = to_numpy(tracer.trace_batch([cams[i] for i in mine], steps, sp, mode))
        at = np.concatenate([np.arange(off[i], off[i + 1]) for i in mine])
        for k in ("t", "r", "th", "ph", "status", "nsteps"):
            assert np.array_equal(got[k][at], alone[k], equal_nan=k in ("t", "r", "th", "ph")), (part, k)
    tracer.set_options()


@pytest.mark.gpu
def test_watchdog_reaches_every_ray_of_a_split_batch(tracer):
    """A batch traced in two launches under a limit that runs out in the first: the timeout code,
    every ray's status written once, the context usable."""
    from paper_2310_15183_gb300 import geotrace as g
    from paper_2310_15183_gb300 import workloads as W
    cams = [W.Camera(0.5, 0.2, 0.0, 1e4, 1.2, 75.0, 64, 48),
            W.Camera(0.5, 0.2, 0.0, 2e5, 1.2, 1.0, 64, 48)]
    out = tracer.alloc_outputs(sum(c.n_rays for c in cams))
    for mode in (0, 1):
        out["status"].fill_(77)
        tracer.set_options(timeout_seconds=0.2)
        with pytest.raises(g.GeotraceError) as e:
            tracer.trace_batch(cams, 1 << 31, 1e-5, mode, out)
        assert e.value.code == -5
        assert np.all(to_numpy(out)["status"] == g.TIMEOUT)
    tracer.set_options()
    assert np.all(to_numpy(tracer.trace_batch(cams, 100, 1e-3, 0))["nsteps"] == 100)


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(_cameras()))
def test_noalloc_takes_each_cameras_route(tracer, name):
    """gt_trace_batch_noalloc in GT_MODE_FP64 gives gt_trace_batch's bits, split or not."""
    import ctypes
    torch = pytest.importorskip("torch")
    from paper_2310_15183_gb300 import geotrace as g
    cams = _cameras()[name]
    descs = (g.CameraDesc * len(cams))(*[g.CameraDesc(c.M, c.S, c.Q, c.r0, c.theta0, c.fov_deg, c.res_x,
                                                      c.res_y) for c in cams])
    out = tracer.alloc_outputs(sum(c.n_rays for c in cams))
    rc = g.load_library().gt_trace_batch_noalloc(
        0, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), descs, len(cams), 1500, 1e-3, 0,
        *[ctypes.c_void_p(out[k].data_ptr()) for k in ("t", "r", "th", "ph", "status", "nsteps")])
    assert rc == 0
    tracer.set_options()
    got, want = to_numpy(out), to_numpy(tracer.trace_batch(cams, 1500, 1e-3, 0))
    for k in got:
        assert np.array_equal(got[k], want[k], equal_nan=k in ("t", "r", "th", "ph")), k


@pytest.mark.gpu
@pytest.mark.parametrize("sp", [1e-9, 1e-10, 1e-30, 2e-38])
def test_mixed_mode_takes_steps_down_to_the_smallest_floats(tracer, sp):
    """Ten steps of any length make ten of them in -t, to the precision of FP32 (and of the
    denormals of 1e-38: 2^-149): a build that flushes them would leave t at zero."""
    tracer.set_spacetime(0.5, 0.2, 0.0)
    tracer.set_camera(10.0, 1.2, 75.0, 9, 7)
    tracer.set_options()
    got = to_numpy(tracer.trace(10, sp, 1))
    assert np.all(got["status"] == 2)
    assert np.max(np.abs(got["t"] + 10 * sp)) <= 1e-5 * 10 * sp + 100 * 2.0 ** -149


@pytest.mark.gpu
@pytest.mark.parametrize("kinds", ["kerr", "mn", "both"])
def test_noalloc_mixed_steps_are_the_rounds_kernels_bits(tracer, kinds):
    """The FP32 steps of gt_trace_batch_noalloc (a branch between stages, denormals kept) and of
    gt_trace_batch (straight-line steps, denormals flushed, for cameras of both kinds the form
    with the kind as the ray's own): one arithmetic, the same bits -- up to escape and horizon for
    Kerr, outside the zone for Manko-Novikov (2000 steps of 1.5e-4 from r0 = 15)."""
    import ctypes
    torch = pytest.importorskip("torch")
    from paper_2310_15183_gb300 import geotrace as g
    from paper_2310_15183_gb300 import workloads as W
    mn = [W.Camera(0.5, 0.24, 2.0, 15.0, 1.3, 75.0, 17, 9), W.Camera(0.5, 0.1, -1.0, 12.0, 0.8, 60.0, 8, 9)]
    kerr = [W.Camera(0.5, 0.2, 0.0, 8.0, 1.2, 60.0, 17, 11), W.Camera(0.5, -0.24, 0.0, 12.0, 0.5, 75.0, 9, 8)]
    cams = {"kerr": kerr, "mn": mn, "both": kerr + mn}[kinds]
    steps, sp = (20000, 2e-3) if kinds == "kerr" else (2000, 1.5e-4)
    descs = (g.CameraDesc * len(cams))(*[g.CameraDesc(c.M, c.S, c.Q, c.r0, c.theta0, c.fov_deg, c.res_x,
                                                      c.res_y) for c in cams])
    out = tracer.alloc_outputs(sum(c.n_rays for c in cams))
    rc = g.load_library().gt_trace_batch_noalloc(
        0, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), descs, len(cams), steps, sp, 1,
        *[ctypes.c_void_p(out[k].data_ptr()) for k in ("t", "r", "th", "ph", "status", "nsteps")])
    assert rc == 0
    tracer.set_options()
    got, want = to_numpy(out), to_numpy(tracer.trace_batch(cams, steps, sp, 1))
    if kinds == "kerr":
        assert set(got["status"]) >= {0, 1}
    for k in got:
        assert np.array_equal(got[k], want[k], equal_nan=k in ("t", "r", "th", "ph")), k


@pytest.mark.gpu
@pytest.mark.parametrize("mode", [0, 1])
def test_autotuner_tunes_the_kernel_of_long_calls_and_compares_the_default(tracer, tmp_path, mode):
    """Trials of few steps time the kernel that calls of many steps take, the cache's key names
    it, and the line says whether the candidate beats the default shape; a shape cached for
    another kernel is not taken; the tuned context is no slower than the default one."""
    import time
    torch = pytest.importorskip("torch")
    tracer.set_options()
    tracer.set_spacetime(0.5, 0.2, 0.0)
    tracer.set_camera(10.0, 1.2, 75.0, 64, 64)

    def pass_ms():
        tracer.trace(2000, 1.5e-4, mode)
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            tracer.trace(2000, 1.5e-4, mode)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best

    plain = pass_ms()
    name = torch.cuda.get_device_name(0)
    path = tmp_path / "tune.txt"
    path.write_text("mode=%d kind=0 sms=%d dev=%s|256 1 1 1e30\n" % (mode, tracer.sm_count(), name))
    shape = tracer.autotune(mode, trial_rays=4096, trial_steps=300, cache_path=str(path))
    assert shape[3] < 1e20
    lines = path.read_text().splitlines()
    assert len(lines) == 2 and "kernel=%d" % (2 if mode else 5) in lines[1]
    assert lines[1].split("|")[1].split()[4] in ("0", "1")
    assert tracer.autotune(mode, trial_rays=4096, trial_steps=300, cache_path=str(path))[:3] == shape[:3]
    assert pass_ms() <= 1.1 * plain
    tracer.set_options()


@pytest.mark.gpu
@pytest.mark.parametrize("Q,r0,th0", [(2.0, 1.9, 1.2), (2.0, 10.0, 0.01), (0.0, 10.0, 0.01)])
def test_a_ray_stopped_among_fp64_steps_reports_where_it_is(tracer, Q, r0, th0):
    """Rays below 4M and at the axis keep an FP64 state between steps: stopped there by the
    watchdog they report it.  A step makes -step of t, to the order of step^2."""
    from paper_2310_15183_gb300 import geotrace as g
    tracer.set_spacetime(0.5, 0.24, Q)
    tracer.set_camera(r0, th0, 60.0, 32, 24)
    out = tracer.alloc_outputs(32 * 24)
    tracer.set_options(timeout_seconds=0.1)
    with pytest.raises(g.GeotraceError) as e:
        tracer.trace(1 << 31, 1.5e-4, 0, out)
    assert e.value.code == -5
    tracer.set_options()
    got = to_numpy(out)
    live = got["nsteps"].view(np.uint32) > 0
    assert np.all(got["status"] == g.TIMEOUT) and live.sum() > 100
    t = -1.5e-4 * got["nsteps"].view(np.uint32)
    assert np.max(np.abs(got["t"][live] / t[live] - 1.0)) <= 1e-3
    assert np.all((got["r"][live] > 1.0) & (got["r"][live] < 1.5 * r0))


@pytest.mark.gpu
@pytest.mark.parametrize("steps", [1000, 3000])
@pytest.mark.parametrize("Q,r0,th0", [(2.0, 1.9, 1.2), (2.0, 2.05, 1.2), (2.0, 10.0, 0.05)])
def test_rays_that_change_between_pairs_and_fp64(tracer, Q, r0, th0, steps):
    """Rays below 4M, across it, and across the axis's line: the FP64 kernel's status, step count
    and end position (1e-9, the project's parity tolerance), and the same bits for a ray in a
    warp of its own."""
    got, ref = _both(tracer, 0.5, 0.24, Q, r0, th0, 9, 7, steps, 3e-4 if r0 < 3 else 1e-3)
    assert np.array_equal(got["status"], ref["status"]) and np.array_equal(got["nsteps"], ref["nsteps"])
    for k in ("t", "r", "th"):
        assert np.max(np.abs(got[k] - ref[k])) <= 1e-9 * np.max(np.abs(ref[k])), k
    for i in (0, 31, 40):
        one = to_numpy(tracer.trace_range(i, 1, steps, 3e-4 if r0 < 3 else 1e-3, 0))
        for k in got:
            assert np.array_equal(one[k], got[k][i:i + 1]), (k, i)
