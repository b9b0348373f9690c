"""The surrogate's calls from several host threads: networks of two sizes, each with
its own buffers and stream on one device, train and run side by side.  Every call
succeeds and the results are those of one thread alone, bit for bit (no kernel adds
in an order that depends on time).  The threads' loops are C, as in a program that
links the library: under Python's lock the calls hardly ever overlap."""
import ctypes as C
import os
import subprocess
import threading

import pytest

pytestmark = pytest.mark.gpu
LOOP = r"""
#include "hlb_surrogate.h"
typedef hlb_status (*loss_grad_fn)(const hlb_sur_config*, const float*, const float*, const float*, const float*,
                                   const int*, int, float*, float*, void*, size_t, void*);
typedef hlb_status (*adam_fn)(long long, float*, const float*, float*, float*, float, float, float, float, int, void*);
typedef hlb_status (*forward_fn)(const hlb_sur_config*, const float*, const float*, const float*, int, float*, void*,
                                 size_t, void*);
int train(loss_grad_fn loss_grad, adam_fn adam, forward_fn forward, const hlb_sur_config* c, long long n, float* p,
          float* g, float* m, float* v, const float* hist, const float* scal, const float* target, const int* label,
          int B, float* loss, float* y, void* ws, size_t ws_bytes, void* stream, int steps) {
  for (int k = 1; k <= steps; ++k) {
    hlb_status st = loss_grad(c, p, hist, scal, target, label, B, g, loss, ws, ws_bytes, stream);
    if (st == HLB_OK) st = adam(n, p, g, m, v, 1e-3f, 0.9f, 0.999f, 1e-8f, k, stream);
    if (st == HLB_OK) st = forward(c, p, hist, scal, B, y, ws, ws_bytes, stream);
    if (st != HLB_OK) return st;
  }
  return HLB_OK;
}
"""
B, STEPS = 8, 2000
SIZES = [(29, 1, 1, 1, 5, 2, 1, 8, 3), (500, 16, 32, 32, 5, 2, 3, 256, 6)]


def test_threads_with_networks_of_two_sizes(tmp_path):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()
    from paper_1812_10375_gb300 import surrogate as sur
    src, so = tmp_path / "loop.c", tmp_path / "loop.so"
    src.write_text(LOOP)
    subprocess.run([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", build.INCLUDE, "-o", str(so),
                    str(src)], check=True)
    loop, lib = C.CDLL(str(so)), sur._lib()

    def job(k):
        """(call, tensors the call writes)"""
        cfg = sur.hlb_sur_config(*SIZES[k])
        net = sur.Net(cfg, seed=k, max_batch=B)
        g = torch.Generator(device="cuda").manual_seed(k)
        r = lambda *shape: torch.randn(*shape, device="cuda", generator=g)
        hist, scal, target = r(B, cfg.L0), r(B, cfg.NS), r(B)
        label = torch.randint(0, cfg.NOUT - 1, (B,), device="cuda", generator=g).int()
        y, stream = torch.empty(B, cfg.NOUT, device="cuda"), torch.cuda.Stream()
        fns = [C.cast(getattr(lib, f), C.c_void_p) for f in ("hlb_sur_loss_grad", "hlb_sur_adam", "hlb_sur_forward")]
        p = lambda t: C.c_void_p(t.data_ptr())
        args = [*fns, C.byref(cfg), C.c_longlong(net.n), p(net.params), p(net.grad), p(net.m), p(net.v), p(hist),
                p(scal), p(target), p(label), B, p(net.loss), p(y), net.ws, C.c_size_t(net.ws_bytes),
                C.c_void_p(stream.cuda_stream), STEPS]
        out = dict(params=net.params, loss=net.loss, y=y)
        return lambda: loop.train(*args), out, (net, hist, scal, target, label, stream)

    alone, together = [[job(k) for k in range(2)] for _ in range(2)]
    torch.cuda.synchronize()
    for call, _, _ in alone:
        assert call() == 0
    torch.cuda.synchronize()
    status = {}
    threads = [threading.Thread(target=lambda k=k: status.__setitem__(k, together[k][0]())) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert status == {0: 0, 1: 0}
    for (_, a, _), (_, b, _) in zip(alone, together):
        for name in a:
            assert torch.equal(a[name], b[name]), name
