"""The tuner times the steps that hlb_step runs: on a lattice whose steps are chained,
the timed steps of the variants that chain launch the chained flow kernel (all but the
first of them), and a reduction of their own after the last only.  Counted from a
kernel trace, in a process of its own so that tracing ends with it."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STEPS = 5
TRACE = """
import json, sys
sys.path[:0] = [%r, %r]
import torch
from torch.profiler import ProfilerActivity, profile
from helpers import coexistence, gpu_domain, ragged_case
d = gpu_domain(ragged_case(), coexistence())
def kernels(f):
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return [e.name.split("(")[0].replace("void ", "") for e in p.events() if "hlb::k_" in e.name]
kernels(lambda: d.step(1))
print(json.dumps([kernels(lambda: d.step(1)), kernels(lambda: d.autotune(%d))]))
"""


def test_tuner_times_chained_steps():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()
    out = subprocess.run([sys.executable, "-c", TRACE % (ROOT, os.path.join(ROOT, "tests"), STEPS)],
                         capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stderr
    one, tuned = json.loads(out.stdout.strip().splitlines()[-1])
    if len(one) != 3:
        pytest.skip("no kernel trace on this machine")
    count = lambda *parts: sum(all(p in k for p in parts) for k in tuned)
    assert count("k_flow_chain<4,") == STEPS - 1   # variant 0 on 45 x 37: tiles of 4 rows
    assert count("k_flow_chain<16,") == STEPS - 1  # variant 1
    # one reduction for the untimed and one for the last timed step of a chain, one a
    # step for the four split variants that never chain
    assert count("k_reduce_split") == 2 * 2 + 4 * (STEPS + 1)
