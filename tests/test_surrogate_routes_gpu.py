"""Networks and batches on both sides of the lines between the per-sample kernels and
the layer kernels, against the FP64 reference, from one workspace that was sized for
the largest batch; nothing is written behind it.  Tolerance as in the other surrogate
tests (1e-4 of each array's largest value)."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu
TOL = 1e-4


@pytest.mark.parametrize("sizes,batches", [
    ((64, 4, 8, 8, 2, 640, 6), [514, 513, 512, 3]),   # by layers, by layers, by samples, by samples
    ((64, 4, 8, 8, 2, 32, 6), [514, 512]),            # training by samples, forward from 513 on by layers
    ((100, 16, 32, 32, 3, 1280, 6), [17, 1]),         # wide: training by layers, forward by samples
    ((250, 16, 32, 32, 3, 1536, 6), [256, 255, 4]),   # wide behind long convolutions: training from 256
                                                      # samples on, forward from 64 on by samples
    ((29, 1, 1, 1, 1, 510, 3), [9]),                  # training by layers: rows of 4-byte reads
    ((64, 4, 8, 8, 2, 16, 1030), [5])])               # forward by layers: many outputs
def test_routes_match_fp64_reference(sizes, batches):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()
    from paper_1812_10375_gb300 import surrogate as sur
    L0, C1, C2, C3, NS, H, NOUT = sizes
    oc = S.Config(L0=L0, C1=C1, C2=C2, C3=C3, K=5, S=2, NS=NS, H=H, NOUT=NOUT)
    rng = np.random.default_rng(H + NOUT)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    theta = f32(S.init_params(oc, rng) + 0.02 * rng.normal(size=oc.n_params()))
    net = sur.Net(sur.hlb_sur_config(L0, C1, C2, C3, 5, 2, NS, H, NOUT), max_batch=max(batches))
    used = net.ws.value - net._ws.data_ptr() + net.ws_bytes
    net._ws[used:] = 0xA5
    t = lambda a, dt=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    net.params.copy_(t(theta))
    for B in batches:
        hist, scal, target = f32(rng.normal(size=(B, L0))), f32(rng.normal(size=(B, NS))), f32(rng.normal(size=B))
        label = rng.integers(0, NOUT - 1, size=B)
        y_o, _ = S.forward(oc, theta, hist, scal)
        y_g = net.forward(t(hist), t(scal)).cpu().numpy()
        assert np.abs(y_g - y_o).max() <= TOL * np.abs(y_o).max(), B
        loss, grad = net.loss_grad(t(hist), t(scal), t(target), t(label, torch.int32))
        mse, ce, g_o = S.loss_grad(oc, theta, hist, scal, target, label)
        np.testing.assert_allclose(loss.cpu().numpy(), [mse, ce], rtol=TOL, atol=1e-7)
        g_g, at = grad.cpu().numpy(), 0
        for name, shp in oc.shapes():
            n = int(np.prod(shp))
            a, b = g_g[at:at + n], g_o[at:at + n]
            assert np.abs(a - b).max() <= TOL * max(np.abs(b).max(), 1e-8), (B, name)
            at += n
        assert bool((net._ws[used:] == 0xA5).all()), B
