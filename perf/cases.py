"""The calls this framework is used for, as timing cases.

A case is a dict of plain values.  `listed()` gives the named ones, `draw(rng)` one more of
the same ranges, `prepare(case, seed)` what a user's program holds before the call (a
configured Tracer or Surrogate, device inputs, output buffers), `run(state)` one pass through
the public entry points, `work(case)` the arithmetic and the bytes that pass cannot do
without, and `exact(case, seed)` the same outputs from plain numpy in 64 bits.

Spacetimes, cameras, step precision and step caps are those of the benchmark's workloads
(M = 0.5, the listing's S = 0.24 and q = 2, step precision 1.5e-4, caps of 2,000, 20,000 and
500,000 steps); the seed moves the viewpoint, the samples and the weights.
"""
import math

import numpy as np
import torch

from paper_2310_15183_gb300 import geotrace as g
from paper_2310_15183_gb300 import workloads as W

M = 0.5
SP = W.WORKLOADS["mn1000"].step_precision
DEG = math.pi / 180.0
# flops of one RK4 step (four fields and the combination; 24 more adds with the compensated
# state of the FP32-mixed mode), counted from the field formulas
STEP_FLOPS = {("kerr", "fp64"): 385, ("mn", "fp64"): 1281, ("kerr", "mixed"): 409,
              ("mn", "mixed"): 1305}
RAY_BYTES = 4 * 8 + 1 + 4  # t, r, theta, phi, status, steps
DIMS = ((16, 256), (256, 256), (256, 256), (256, 256), (256, 16))
N_PARAMS = sum(i * o + o for i, o in DIMS)
NET_FLOPS = 2 * sum(i * o for i, o in DIMS)  # one row forward


def listed():
    return [
        # the first thing a user runs: a small Schwarzschild frame, every ray at the step cap
        {"name": "fp64_schwarzschild_frame", "do": "trace", "mode": "fp64", "kind": "kerr",
         "spin": 0.0, "r0": 10.0, "nx": 64, "ny": 64, "steps": 2000},
        # an ordinary accuracy-reference frame of the Manko-Novikov hole
        {"name": "fp64_mn_frame", "do": "trace", "mode": "fp64", "kind": "mn", "spin": 0.96,
         "r0": 15.0, "nx": 240, "ny": 200, "steps": 2000},
        # the headline workload's kernel: a Manko-Novikov frame at 20,000 steps
        {"name": "mixed_mn_frame", "do": "trace", "mode": "mixed", "kind": "mn", "spin": 0.96,
         "r0": 15.0, "nx": 500, "ny": 400, "steps": 20000},
        # a Kerr shadow: every ray runs until it escapes or falls in; odd sides
        {"name": "mixed_kerr_shadow", "do": "trace", "mode": "mixed", "kind": "kerr",
         "spin": 0.9, "r0": 15.0, "nx": 301, "ny": 211, "steps": 500000},
        # near-horizon view: the camera inside the zone, where trapped Manko-Novikov rays live
        {"name": "mixed_mn_zone", "do": "trace", "mode": "mixed", "kind": "mn", "spin": 0.96,
         "r0": 1.9, "nx": 200, "ny": 200, "steps": 4000},
        # many cameras of uneven size in one launch: a parameter sweep of shadows
        {"name": "mixed_batch", "do": "batch", "cams": 24, "side_min": 13, "side_max": 96,
         "steps": 500000},
        # labelling random rays, each with a spacetime of its own, for the surrogate's training
        {"name": "mixed_labels", "do": "rays", "n": 32768, "steps": 500000},
        # surrogate: a handful of directions, a large set of them, a gradient, training
        # steps, a gated image with integrator probes and fallback
        {"name": "surrogate_eval_small", "do": "eval", "n": 300},
        {"name": "surrogate_eval_large", "do": "eval", "n": 1 << 20},
        {"name": "surrogate_grad", "do": "grad", "n": 16384},
        {"name": "surrogate_train", "do": "train", "n": 65536, "batch": 8192},
        {"name": "surrogate_image", "do": "infer", "spin": 0.1, "nx": 400, "ny": 300,
         "stride": 4, "steps": 500000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["trace64", "trace64", "trace32", "trace32", "shadow", "zone", "batch",
                     "rays", "eval", "eval", "grad", "train", "infer"])
    if do == "trace64":
        kind = rng.choice(["kerr", "mn"])
        return {"do": "trace", "mode": "fp64", "kind": kind,
                "spin": round(rng.uniform(0.1, 0.98), 3), "r0": round(rng.uniform(7.5, 25.0), 2),
                "nx": _log(rng, 16, 240), "ny": _log(rng, 16, 200),
                "steps": rng.randint(500, 2000)}
    if do == "trace32":
        kind = rng.choice(["kerr", "mn"])
        return {"do": "trace", "mode": "mixed", "kind": kind,
                "spin": round(rng.uniform(0.1, 0.98), 3), "r0": round(rng.uniform(12.0, 25.0), 2),
                "nx": _log(rng, 32, 500), "ny": _log(rng, 32, 400),
                "steps": rng.randint(2000, 20000)}
    if do == "shadow":
        return {"do": "trace", "mode": "mixed", "kind": "kerr",
                "spin": round(rng.uniform(0.0, 0.98), 3), "r0": round(rng.uniform(7.5, 20.0), 2),
                "nx": _log(rng, 48, 301), "ny": _log(rng, 48, 211), "steps": 500000}
    if do == "zone":
        return {"do": "trace", "mode": "mixed", "kind": "mn", "spin": 0.96,
                "r0": round(rng.uniform(1.8, 1.95), 3), "nx": _log(rng, 24, 200),
                "ny": _log(rng, 24, 200), "steps": rng.randint(500, 4000)}
    if do == "batch":
        return {"do": "batch", "cams": rng.randint(2, 24), "side_min": 13,
                "side_max": rng.randint(24, 96), "steps": 500000}
    if do == "rays":
        return {"do": "rays", "n": _log(rng, 2048, 32768), "steps": 500000}
    if do == "eval":
        return {"do": "eval", "n": _log(rng, 100, 1 << 20)}
    if do == "grad":
        return {"do": "grad", "n": _log(rng, 500, 16384)}
    if do == "train":
        batch = 1024 * rng.choice([1, 2, 4, 8])
        return {"do": "train", "n": batch * rng.randint(2, 8) + rng.randint(0, batch - 1),
                "batch": batch}
    return {"do": "infer", "spin": round(rng.uniform(0.0, 0.3), 3), "nx": _log(rng, 96, 400),
            "ny": _log(rng, 96, 300), "stride": rng.choice([4, 8]), "steps": 500000}


# ------------------------------------------------------------------ inputs
def _rng(case, seed):
    return np.random.Generator(np.random.PCG64([int(seed) & 0x7FFFFFFF, 15183]))


def _view(case, seed):
    """(S, Q, theta0, fov) of a camera case; the seed moves the viewpoint."""
    rng = _rng(case, seed)
    theta0 = rng.uniform(60.0, 85.0) * DEG
    q = 2.0 if case.get("kind") == "mn" else 0.0
    return case["spin"] * M * M, q, theta0, 75.0


def _samples(case, seed):
    """Surrogate inputs (alpha, beta, a/M, q, theta0) of the training ranges."""
    return W.surrogate_samples(case["n"], seed=int(seed) & 0x7FFFFFFF)


def _deflected(alpha, beta, spin, theta0, r0):
    """Impact parameter over its critical value, and end direction at 1.5 r0, of a ray: the
    Schwarzschild orbit integral (48 Gauss points) and the first-order term of the spin --
    labels and fits of the right shape without an integration."""
    f, b_c = 1.0 - 2.0 * M / r0, 3.0 * math.sqrt(3.0) * M
    w = np.hypot(alpha, beta) + 1e-15
    b = r0 * r0 * w / np.sqrt(1.0 + f * (r0 * w) ** 2)
    x = np.maximum(b, 1.02 * b_c)
    u_t = 0.5 * math.sqrt(3.0) / (x * np.cos(np.arccos(-b_c / x) / 3.0))  # 1 / turning radius
    node, weight = np.polynomial.legendre.leggauss(24)
    phi = -4.0 * spin * M * M * (alpha / w * np.sin(theta0)) / x ** 2
    for r in (r0, 1.5 * r0):  # u = u_t (1 - s^2) takes the root at u_t out of the integrand
        top = np.sqrt(1.0 - 1.0 / (r * u_t))
        s2 = (0.5 * top[:, None] * (node + 1.0)) ** 2
        u = u_t[:, None] * (1.0 - s2)
        rest = (1.0 / x[:, None] ** 2 - u * u + 2.0 * M * u ** 3) / (u_t[:, None] * s2)
        phi = phi + top * np.sqrt(u_t) * (weight / np.sqrt(rest)).sum(axis=1)
    st, ct, zero = np.sin(theta0), np.cos(theta0), np.zeros_like(alpha)
    radial = np.stack([st + zero, zero, ct + zero], axis=-1)
    along = np.stack([beta * ct, alpha, -beta * st], axis=-1) / w[:, None]
    return b / b_c, np.cos(phi)[:, None] * radial + np.sin(phi)[:, None] * along


def _labels(host):
    alpha, beta, spin, _, theta0 = host
    ratio, d = _deflected(alpha, beta, spin, theta0, 15.0)
    status = np.where(ratio > 1.0, g.ESCAPED, g.HORIZON).astype(np.uint8)
    return status, np.arccos(np.clip(d[:, 2], -1.0, 1.0)), np.arctan2(d[:, 1], d[:, 0])


def _weights(rng):
    """LeCun-normal layers [out, in] and zero biases, as training starts from."""
    ws = [rng.normal(0.0, 1.0 / math.sqrt(10 if k == 0 else i), (o, i)).astype(np.float32)
          for k, (i, o) in enumerate(DIMS)]
    return ws, [np.zeros(o, np.float32) for _, o in DIMS]


def _flat(ws, bs):
    return np.concatenate([x for w, b in zip(ws, bs) for x in (w.ravel(), b)]).astype(np.float32)


def _features(alpha, beta, spin, q, theta0, dtype=np.float64):
    """The network's 16 input columns for the default normalisation."""
    v = math.tan(0.5 * 75.0 * DEG) / 15.0
    h = math.atan(math.tan(v))
    lo, hi = 0.0872664626, 1.5707963268
    a, b = alpha / h, beta / v
    rho = np.sqrt(a * a + b * b)
    far = np.maximum(rho, 1e-3)
    x = np.zeros((len(alpha), 16), dtype)
    for k, col in enumerate((a, b, spin * (2.0 / 0.99) - 1.0, q / 2.0,
                             theta0 * (2.0 / (hi - lo)) - (hi + lo) / (hi - lo), rho, a / far,
                             b / far, np.cos(theta0), np.sin(theta0))):
        x[:, k] = col
    return x


def _silu(z):
    return z / (1.0 + np.exp(-z))


def _fitted(case, rng, theta0):
    """A network that holds one camera's image to a few 1e-3: ridge functions of the pixel
    direction and its radius in the first layer, a least-squares fit of the logit and the end
    direction on them, and the fit carried through the other layers (silu(z) - silu(-z) = z)."""
    n = 8192
    v = math.tan(0.5 * 75.0 * DEG) / 15.0
    alpha, beta = rng.uniform(-v, v, n), rng.uniform(-v, v, n)
    th, spin = np.full(n, theta0), np.full(n, case["spin"])
    ratio, d = _deflected(alpha, beta, spin, th, 15.0)
    x = _features(alpha, beta, spin, np.zeros(n), th)
    ws, bs = [np.zeros((o, i)) for i, o in DIMS], [np.zeros(o) for _, o in DIMS]
    ws[0][:, [0, 1, 5]] = rng.normal(0.0, 3.0, (256, 3))
    ws[0][:64, :2] = 0.0
    bs[0][:] = -np.sum(x[:256] * ws[0], axis=1)
    x1 = np.concatenate([_silu(x @ ws[0].T + bs[0]), np.ones((n, 1))], axis=1)

    def solve(rows, target):
        a = x1 * rows[:, None]
        return np.linalg.solve(a.T @ a + 1e-8 * n * np.eye(257), a.T @ (target * rows[:, None]))
    sol = np.concatenate([solve(np.ones(n), np.clip(16.0 * (ratio - 1.0), -6.0, 6.0)[:, None]),
                          solve(np.where(ratio > 1.15, 1.0, 0.002), d)], axis=1)
    ws[1][:4], ws[1][4:8], bs[1][:4], bs[1][4:8] = sol[:256].T, -sol[:256].T, sol[256], -sol[256]
    pair = np.concatenate([np.eye(4), -np.eye(4)], axis=1)
    for k in (2, 3):
        ws[k][:4, :8], ws[k][4:8, :8] = pair, -pair
    ws[4][:4, :8] = pair
    return _flat(ws, bs)


def _dev(arrays):
    return [torch.tensor(a, device="cuda") for a in arrays]


def prepare(case, seed):
    do = case["do"]
    rng = _rng(case, seed)
    s = {"case": case, "tracer": g.Tracer(0)}
    tr = s["tracer"]
    if do in ("trace", "infer"):
        spin_s, q, theta0, fov = _view(case, seed)
        tr.set_spacetime(M, spin_s, q)
        tr.set_camera(case.get("r0", 15.0), theta0, fov, case["nx"], case["ny"])
        s["mode"] = g.MODE_FP64 if case.get("mode") == "fp64" else g.MODE_FP32_MIXED
        s["out"] = tr.alloc_outputs(case["nx"] * case["ny"])
    if do == "infer":
        s["net"] = g.Surrogate(0, seed=1)
        s["net"].set_params(_fitted(case, rng, theta0))
    elif do == "batch":
        views = W.batch_cameras(case["cams"], seed=int(seed) & 0x7FFFFFFF)
        sides = W.batch_cameras(case["cams"], side_min=case["side_min"],
                                side_max=case["side_max"])  # the sizes belong to the case
        s["cams"] = [W.sub_camera(v, c.res_x, c.res_y) for v, c in zip(views, sides)]
        s["out"] = tr.alloc_outputs(sum(c.n_rays for c in s["cams"]))
    elif do == "rays":
        s["in"] = _dev(_samples(case, seed))
        s["out"] = tr.alloc_outputs(case["n"])
    elif do in ("eval", "grad", "train"):
        host = _samples(case, seed)
        s["in"] = _dev(host)
        s["net"] = g.Surrogate(0, seed=1)
        s["net"].set_params(_flat(*_weights(rng)))
        if do != "eval":
            s["labels"] = _dev(_labels(host))
    return s


def run(s):
    case, tr = s["case"], s["tracer"]
    do = case["do"]
    if do == "trace":
        return tr.trace(case["steps"], SP, s["mode"], s["out"])
    if do == "batch":
        return tr.trace_batch(s["cams"], case["steps"], SP, g.MODE_FP32_MIXED, s["out"])
    if do == "rays":
        return tr.trace_rays(*s["in"], M=M, r0=15.0, n_steps=case["steps"], step_precision=SP,
                             mode=g.MODE_FP32_MIXED, out=s["out"])
    if do == "eval":
        return {"net": s["net"].eval(tr, s["in"])}
    if do == "grad":
        grads, loss = s["net"].grad(tr, s["in"], s["labels"], 100.0)
        return {"grads": grads, "loss": np.float32(loss)}
    if do == "train":
        losses = s["net"].train(tr, s["in"], s["labels"], epochs=1, batch=case["batch"], lr=2e-3,
                                dir_weight=100.0)
        return {"losses": losses, "params": s["net"].get_params()}
    out, fallback, probes = s["net"].infer(
        tr, 2.0, 0.02, case["steps"], SP, g.MODE_FP32_MIXED, s["out"], probe_stride=case["stride"],
        probe_tol=2e-3, axis=0.02, with_probes=True)
    return {**out, "fallback": fallback, "probes": probes}


def _rays(case):
    if case["do"] == "batch":
        lo, hi = case["side_min"], case["side_max"]
        return case["cams"] * (hi * hi - lo * lo) / max(2.0 * math.log(hi / lo), 1e-9)
    return case["nx"] * case["ny"] if "nx" in case else case["n"]


def work(case):
    do = case["do"]
    n = _rays(case)
    if do in ("trace", "batch", "rays"):
        r0 = case.get("r0", 15.0)
        # a step takes about SP of coordinate time, and a ray leaves after about 2.5 r0 of it
        steps = min(case["steps"], 2.5 * r0 / SP)
        per = STEP_FLOPS[case.get("kind", "kerr"), case.get("mode", "mixed")]
        return {"bytes": n * (RAY_BYTES + (40 if do == "rays" else 0)), "flops": n * steps * per}
    if do == "eval":
        return {"bytes": n * (40 + 16) + 4 * N_PARAMS, "flops": n * NET_FLOPS}
    if do == "grad":
        return {"bytes": n * (40 + 17) + 8 * N_PARAMS, "flops": 3 * n * NET_FLOPS}
    if do == "train":
        k = n // case["batch"]
        return {"bytes": k * (case["batch"] * 57 + 28 * N_PARAMS),
                "flops": 3 * k * case["batch"] * NET_FLOPS}
    # the probes and some of the other pixels are integrated, the network sees all of them
    traced = n / case["stride"] ** 2 + 0.3 * n
    return {"bytes": n * RAY_BYTES, "flops": n * NET_FLOPS
            + traced * 2.5 * 15.0 / SP * STEP_FLOPS["kerr", "mixed"]}


# ------------------------------------------------------------------ 64-bit references
def _kerr_metric(a, r, th):
    """Inverse metric (tt, t phi, phi phi, rr, theta theta) of Kerr at complex arguments."""
    s2, c2 = np.sin(th) ** 2, np.cos(th) ** 2
    sig = r * r + a * a * c2
    dlt = r * r - 2.0 * M * r + a * a
    ra = r * r + a * a
    d = sig * dlt
    return (-(ra * ra - a * a * dlt * s2) / d, -2.0 * M * a * r / d,
            (dlt - a * a * s2) / (d * s2), dlt / sig, 1.0 / sig)


def _mn_metric(par, r, th):
    """The same for the Manko-Novikov spacetime of the line element
    -f (dt - w dphi)^2 + e^{2 gamma} rho^2 / (f Delta) dr^2 + ..., multipoles l <= 2."""
    al, k, be = par
    x, y, s2 = (r - M) / k, np.cos(th), np.sin(th) ** 2
    x2 = x * x - 1.0
    rr = np.sqrt(x2 + y * y)
    u = x * y / rr
    p = [1.0, u, 0.5 * (3.0 * u * u - 1.0), 0.5 * u * (5.0 * u * u - 3.0)]
    lo = [p[j] / rr ** (j + 1) for j in range(3)]
    plus, minus = lo[0] + lo[1] + lo[2], lo[0] - lo[1] + lo[2]
    fa = -al * np.exp(-2.0 * be * (-1.0 + (x - y) * plus))
    fb = al * np.exp(2.0 * be * (1.0 - (x + y) * minus))
    ab = fa * fb
    A = x2 * (1.0 + ab) ** 2 - s2 * (fb - fa) ** 2
    B = (x + 1.0 + (x - 1.0) * ab) ** 2 + ((1.0 + y) * fa + (1.0 - y) * fb) ** 2
    C = (x2 * (1.0 + ab) * (fb - fa - y * (fa + fb))
         + s2 * (fb - fa) * (1.0 + ab + x * (1.0 - ab)))
    e2psi = np.exp(2.0 * be * lo[2])
    g2 = (3.0 * be * be / rr ** 6 * (p[3] ** 2 - p[2] ** 2)
          + 2.0 * be * (-2.0 + (x - y) * plus + (x + y) * minus))
    f = e2psi * A / B
    w = 2.0 * k * C / (e2psi * A) - 4.0 * k * al / (1.0 - al * al)
    dlt = k * k * x2
    gth = (1.0 - al * al) ** 2 / (k * k) * np.exp(2.0 * be * lo[2] - g2) / B
    F = f / (dlt * s2)
    return -1.0 / f + w * w * F, w * F, F, gth * dlt, gth


def _frame_state(metric, theta0, r0, fov, nx, ny):
    """Initial state of every pixel of a pinhole camera at (r0, theta0)."""
    gu = [float(np.real(v)) for v in metric(np.array(r0), np.array(theta0))]
    det = gu[0] * gu[2] - gu[1] ** 2
    tt, tp, pp, rr, hh = gu[2] / det, -gu[1] / det, gu[0] / det, 1.0 / gu[3], 1.0 / gu[4]
    V = math.tan(0.5 * fov / 180.0 * math.pi) / r0
    H = math.atan(math.tan(V) * nx / ny)
    i, j = np.arange(nx), np.arange(ny)
    al = H * (2.0 * i - (nx - 1)) / (nx - 1)
    bt = V * (2.0 * j - (ny - 1)) / (ny - 1)
    vph, vth = np.tile(al / math.sin(theta0), ny), np.repeat(bt, nx)
    b2, c = tp * vph, rr + hh * vth ** 2 + pp * vph ** 2
    T = (-b2 + np.sqrt(b2 * b2 - tt * c)) / tt
    sc = 1.0 / np.abs(T)
    z = np.zeros(nx * ny)
    return (np.stack([z, z + r0, z + theta0, z, -rr * sc, hh * vth * sc]),
            (tt * T + tp * vph) * sc, (tp * T + pp * vph) * sc)


def _field(metric, x, pt, pph):
    """q' = g p and p' = -1/2 dg p p, the derivatives by the complex step."""
    _, r, th, _, pr, pth = x

    def h2(v):
        return (v[0] * pt ** 2 + 2.0 * v[1] * pt * pph + v[2] * pph ** 2 + v[3] * pr ** 2
                + v[4] * pth ** 2)
    vr, vt = metric(r + 1e-30j, th + 0j), metric(r + 0j, th + 1e-30j)
    v = [np.real(c) for c in vr]
    return np.stack([v[0] * pt + v[1] * pph, v[3] * pr, v[4] * pth, v[1] * pt + v[2] * pph,
                     -0.5e30 * np.imag(h2(vr)), -0.5e30 * np.imag(h2(vt))])


def _exact_frame(case, seed):
    spin_s, q, theta0, fov = _view(case, seed)
    n = case["nx"] * case["ny"]
    # every ray of these frames is still under way at the cap; the cost is the limit
    if case["mode"] != "fp64" or n * case["steps"] > (9e6 if q == 0.0 else 2.5e6):
        return None
    if q == 0.0:
        def metric(r, th):
            return _kerr_metric(spin_s / M, r, th)
    else:
        sm = spin_s / M
        al = (-M + math.sqrt(M * M - sm * sm)) / sm
        k = M * (1.0 - al * al) / (1.0 + al * al)

        def metric(r, th):
            return _mn_metric((al, k, q * M ** 3 / k ** 3), r, th)
    x, pt, pph = _frame_state(metric, theta0, case["r0"], fov, case["nx"], case["ny"])
    for _ in range(case["steps"]):
        k1 = _field(metric, x, pt, pph)
        h = np.abs(SP / k1[0])
        k2 = _field(metric, x + 0.5 * h * k1, pt, pph)
        k3 = _field(metric, x + 0.5 * h * k2, pt, pph)
        k4 = _field(metric, x + h * k3, pt, pph)
        x = x + h / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
    return {"t": x[0], "r": x[1], "th": x[2], "ph": x[3],
            "status": np.full(n, g.MAXSTEPS, np.uint8),
            "nsteps": np.full(n, case["steps"], np.int32)}


def _exact_net(case, seed):
    """Outputs, or the loss and its gradient, of the network in 64 bits."""
    host = _samples(case, seed)
    ws, bs = _weights(_rng(case, seed))
    ws = [w.astype(np.float64) for w in ws]
    a, z = [_features(*host)], []
    for k, w in enumerate(ws):
        z.append(a[k] @ w.T)
        if k < 4:
            a.append(_silu(z[k]))
    if case["do"] == "eval":
        return {"net": z[4][:, :4]}
    status, th, ph = _labels(host)
    y = (status == g.ESCAPED).astype(np.float64)
    d = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], axis=1)
    n, out = len(y), z[4]
    diff = (out[:, 1:4] - d) * y[:, None]
    loss = np.mean(np.logaddexp(0.0, out[:, 0]) - out[:, 0] * y
                   + 100.0 * np.sum(diff * diff, axis=1))
    dz = np.zeros_like(out)
    dz[:, 0] = (1.0 / (1.0 + np.exp(-out[:, 0])) - y) / n
    dz[:, 1:4] = 200.0 * diff / n
    gw, gb = [], []
    for k in range(4, -1, -1):
        gw.insert(0, dz.T @ a[k])
        gb.insert(0, dz.sum(axis=0))
        if k:
            sg = 1.0 / (1.0 + np.exp(-z[k - 1]))
            dz = (dz @ ws[k]) * sg * (1.0 + z[k - 1] * (1.0 - sg))
    return {"grads": np.concatenate([v for w, b in zip(gw, gb) for v in (w.ravel(), b)]),
            "loss": np.float64(loss)}


def exact(case, seed):
    if case["do"] == "trace":
        return _exact_frame(case, seed)
    if case["do"] == "grad" or (case["do"] == "eval" and case["n"] <= 1 << 17):
        return _exact_net(case, seed)
    return None
