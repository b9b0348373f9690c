"""Destroying a handle gives back what the library holds on the host and waits for no
work of other streams: an application that closes one domain goes on launching for the
others.  Records read through handles that come and go stay right, also when more
handles live at once than the library keeps page-locked records for."""
import pytest

from helpers import coexistence, gpu_domain, ragged_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()


@pytest.mark.parametrize("kind", ["domain", "batch"])
def test_destroy_does_not_wait_for_other_streams(kind):
    import torch
    from paper_1812_10375_gb300 import hlb
    p = hlb.default_params(64, 48)
    h = hlb.Domain(p) if kind == "domain" else hlb.Batch([p, p])
    a = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
    b = torch.empty_like(a)
    torch.mm(a, a, out=b)
    torch.cuda.synchronize()
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    with torch.cuda.stream(side):
        for _ in range(400):  # about 0.2 s
            torch.mm(a, a, out=b)
        done.record()
    h.close()
    waited = done.query()
    torch.cuda.synchronize()
    assert not waited


def test_records_of_many_handles():
    from paper_1812_10375_gb300 import hlb
    coex, case = coexistence(), ragged_case()
    want = []
    d = gpu_domain(case, coex)
    for _ in range(4):
        d.step(1)
        want.append(d.diag())
    d.close()
    p = hlb.default_params(16, 16)
    for _ in range(2):
        crowd = [hlb.Batch([p] * 60) for _ in range(10)]
        ds = [gpu_domain(case, coex) for _ in range(3)]
        for k in range(4):
            for d in ds[k % 3:]:
                d.step(k + 1 - d.diag().step)
                assert d.diag() == want[k], k
        for b in crowd:
            b.close()
        late = gpu_domain(case, coex)
        late.step(4)
        assert late.diag() == want[3]
        for d in ds + [late]:
            d.close()
