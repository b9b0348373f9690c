"""The one-CTA-per-sample surrogate kernels (K = 5, stride 2) against the FP64
reference at the sizes where their tiling can go wrong: one position or channel,
channel counts off the eight-channel blocks, rows of the linear layers that are
not whole 16-byte pieces, more neurons than threads, one sample.  Tolerance as in
the layer-by-layer test (1e-4 of each array's largest value): sums of up to a few
thousand FP32 terms, and units whose sign differs between FP32 and FP64."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu
TOL = 1e-4


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()


@pytest.mark.parametrize("L0,C1,C2,C3,NS,H,NOUT,B", [
    (29, 1, 1, 1, 1, 1, 2, 1), (100, 3, 9, 5, 2, 7, 3, 5), (64, 16, 32, 32, 2, 200, 6, 17),
    (500, 16, 32, 32, 3, 256, 6, 64), (512, 8, 16, 24, 3, 600, 9, 3)])
def test_sample_kernels_match_fp64_reference(L0, C1, C2, C3, NS, H, NOUT, B):
    import torch
    from paper_1812_10375_gb300 import surrogate as sur
    oc = S.Config(L0=L0, C1=C1, C2=C2, C3=C3, K=5, S=2, NS=NS, H=H, NOUT=NOUT)
    gc = sur.hlb_sur_config(L0, C1, C2, C3, 5, 2, NS, H, NOUT)
    rng = np.random.default_rng(L0 + H + B)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    theta = f32(S.init_params(oc, rng) + 0.05 * rng.normal(size=oc.n_params()))
    hist, scal, target = f32(rng.normal(size=(B, L0))), f32(rng.normal(size=(B, NS))), f32(rng.normal(size=B))
    label = rng.integers(0, NOUT - 1, size=B)
    net = sur.Net(gc, max_batch=B)
    t = lambda a, dt=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    net.params.copy_(t(theta))
    y_o, _ = S.forward(oc, theta, hist, scal)
    y_g = net.forward(t(hist), t(scal)).cpu().numpy()
    assert np.abs(y_g - y_o).max() <= TOL * np.abs(y_o).max()
    loss, grad = net.loss_grad(t(hist), t(scal), t(target), t(label, torch.int32))
    mse, ce, g_o = S.loss_grad(oc, theta, hist, scal, target, label)
    np.testing.assert_allclose(loss.cpu().numpy(), [mse, ce], rtol=TOL, atol=1e-7)
    g_g, at = grad.cpu().numpy(), 0
    for name, shp in oc.shapes():
        n = int(np.prod(shp))
        a, b = g_g[at:at + n], g_o[at:at + n]
        assert np.abs(a - b).max() <= TOL * max(np.abs(b).max(), 1e-8), name
        at += n
