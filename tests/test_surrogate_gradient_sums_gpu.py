"""The convolutions' gradients are sums over positions and samples; their rounding
errors stay at the last bit for large batches.  All parameters and inputs are positive
and every sample pulls the same way, so that no unit is cut off and no sum cancels:
what is left against the FP64 reference is the rounding of the sums.  A value's own
rounding is 2^-24 / sqrt(3) of it in the root mean square; with the values that go
into the sums rounded likewise and the sums' partial results, each of which rounds for
a part of the samples only, one unit in the last place (2^-23) bounds it.  One chain
of B additions comes to 2^-24 / sqrt(3) sqrt(B / 3): 6.4e-7 for 1,024 samples."""
import numpy as np
import pytest

from oracle import surrogate as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L0,B", [(100, 1024), (101, 1000), (500, 700)])
def test_convolution_gradients_keep_the_last_bit(L0, B):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()
    from paper_1812_10375_gb300 import surrogate as sur
    oc = S.Config(L0=L0, NS=3, H=64)
    rng = np.random.default_rng(L0)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)
    theta = f32(0.2 * np.abs(S.init_params(oc, rng)) + 0.01)
    hist, scal = f32(1.0 + 0.1 * rng.random((B, L0))), f32(1.0 + 0.1 * rng.random((B, 3)))
    target, label = np.full(B, -1.0), rng.integers(0, oc.NOUT - 1, size=B)
    net = sur.Net(sur.hlb_sur_config(L0, oc.C1, oc.C2, oc.C3, oc.K, oc.S, 3, oc.H, oc.NOUT), max_batch=B)
    t = lambda a, dt=torch.float32: torch.tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    net.params.copy_(t(theta))
    _, grad = net.loss_grad(t(hist), t(scal), t(target), t(label, torch.int32))
    _, _, want = S.loss_grad(oc, theta, hist, scal, target, label)
    got, at = grad.cpu().numpy().astype(np.float64), 0
    for name, shp in oc.shapes()[:6]:
        n = int(np.prod(shp))
        a, b = got[at:at + n], want[at:at + n]
        rms = float(np.sqrt(np.mean((a - b) ** 2) / np.mean(b ** 2)))
        print(name, rms)
        assert rms < 2.0 ** -23, name
        at += n
