"""The surrogate's single-kernel passes (csrc/mlp_fused.cu) at the edges of their tiles."""
import numpy as np
import pytest

from oracle import mlp
from paper_2310_15183_gb300 import workloads as W

from .test_gpu_surrogate import _abs_scales, _fake_labels

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def net():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_15183_gb300 import build, geotrace
    build.build()
    tracer, s = geotrace.Tracer(0), geotrace.Surrogate(0, seed=21)
    p = s.get_params()
    for b in mlp.split(p)[1]:  # a fresh network's biases are zero
        b[:] = np.random.Generator(np.random.PCG64(b.size)).normal(0, 0.3, b.size)
    s.set_params(p)
    yield tracer, s
    s.close()
    tracer.close()


@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 255, 152 * 128 - 1, 152 * 128, 152 * 128 + 1,
                               2 * 152 * 128 + 77])
def test_rows_at_tile_edges(net, n):
    """Every output within 2^-12 sum_k |a_k| |w_k| of the CPU reference's split-precision
    product (as for the layer-wise forward: split pairs to 2^-16, FP32 accumulation of 768
    terms 2^-14.4, earlier layers the same), and independent of the rows around it."""
    tracer, s = net
    host = W.surrogate_samples(n, seed=n)
    dev = [torch.tensor(x, device="cuda") for x in host]
    out = s.eval(tracer, dev).cpu().numpy()
    some = np.unique(np.concatenate([np.arange(min(n, 200)), np.arange(max(0, n - 200), n)]))
    X0 = mlp.features(*[x[some] for x in host])
    p = s.get_params().astype(np.float64)
    As, Zs = mlp.forward(p, X0, bf=True)
    scale = np.abs(As[4]) @ np.abs(mlp.split(p)[0][4]).T + np.abs(mlp.split(p)[1][4])
    err = np.abs(out[some] - Zs[4][:, :4])
    assert np.all(err <= 2.0 ** -12 * scale[:, :4]), float(np.max(err / scale[:, :4]))
    part = s.eval(tracer, [d[n // 2:].contiguous() for d in dev]).cpu().numpy()
    assert np.array_equal(part, out[n // 2:])


def test_unaligned_output(net):
    """The C entry takes any float pointer: rows of 16 bytes at a 4-byte offset."""
    tracer, s = net
    host = W.surrogate_samples(200, seed=3)
    dev = [torch.tensor(x, device="cuda") for x in host]
    buf = torch.zeros(4 * 200 + 2, dtype=torch.float32, device="cuda")
    rc = s.lib.gt_surrogate_eval(tracer.ctx, s.h, 200, *[d.data_ptr() for d in dev],
                                 buf.data_ptr() + 4)
    assert rc == 0
    torch.cuda.synchronize()
    assert torch.equal(buf[1:-1].view(200, 4), s.eval(tracer, dev))
    assert buf[0].item() == 0.0 and buf[-1].item() == 0.0


@pytest.mark.parametrize("sizes", [(1, 128, 127), (300, 129, 300), (152 * 128 + 5, 40)])
def test_gradients_at_tile_edges(net, sizes):
    """Loss and gradients (one kernel for forward, loss and input gradients, one for the weight
    gradients) on one network for batches of changing size: element-wise within the bounds of
    the layer-wise test (2^-7 of the running bound: one bf16 rounding decision per operand)."""
    tracer, s = net
    for n in sizes:
        host = W.surrogate_samples(n, seed=n + 1)
        lab_h, lab_d = _fake_labels(n, n + 2)
        grads, loss = s.grad(tracer, [torch.tensor(x, device="cuda") for x in host], lab_d, 10.0)
        p = s.get_params().astype(np.float64)
        X0 = mlp.features(*host)
        y, d = mlp.labels(*lab_h)
        ref_loss, ref_g, _ = mlp.loss_and_grad(p, X0, y, d, 10.0, bf=True)
        assert abs(loss - ref_loss) < 1e-4 * abs(ref_loss), (n, loss, ref_loss)
        scale_w, scale_b, _ = _abs_scales(p, X0, y, d, 10.0)
        ws, bs = mlp.split(grads.astype(np.float64))
        rws, rbs = mlp.split(ref_g)
        for l in range(5):
            assert np.all(np.abs(ws[l] - rws[l]) <= 2.0 ** -7 * scale_w[l] + 1e-12), (n, l)
            assert np.all(np.abs(bs[l] - rbs[l]) <= 2.0 ** -7 * scale_b[l] + 1e-12), (n, l)


def test_features_outside_the_pair_range(net):
    """Rows whose polar form or angle leaves the range of the double-float evaluation (the image
    centre, an angle of many turns) take FP64: the outputs match the reference like any row's."""
    tracer, s = net
    n = 8
    al = np.array([0.0, 1e-9, 1e-30, 0.05, 0.05, -0.02, 1e-7, 0.03])
    be = np.array([0.0, 0.0, 1e-30, 0.01, 0.0, 0.05, -1e-7, 0.0])
    th = np.array([1.0, 1.0, 0.5, 700.0, -129.0, 1.2, 1.3, 127.9])
    host = (al, be, np.full(n, 0.5), np.zeros(n), th)
    out = s.eval(tracer, [torch.tensor(x, device="cuda") for x in host]).cpu().numpy()
    p = s.get_params().astype(np.float64)
    As, Zs = mlp.forward(p, mlp.features(*host), bf=True)
    scale = np.abs(As[4]) @ np.abs(mlp.split(p)[0][4]).T + np.abs(mlp.split(p)[1][4])
    err = np.abs(out - Zs[4][:, :4])
    assert np.all(err <= 2.0 ** -12 * scale[:, :4]), float(np.max(err / scale[:, :4]))
