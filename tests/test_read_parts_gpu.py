"""Reading some of the fields: every subset of rho, u_x, u_y and T gives the values of a
full read bit for bit (rho without u is formed from a cell's own populations alone, T
is copied), leaves the other arrays as they were, and solid rows are zero; before the
first step and after, both storages, every top."""
import itertools

import numpy as np
import pytest

from paper_1812_10375_gb300 import workloads as wl

from helpers import coexistence

pytestmark = pytest.mark.gpu
NAMES = ("rho", "ux", "uy", "T")


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("top", ["convective", "const_rho", "wall"])
def test_every_subset_equals_the_full_read(storage, top):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build, hlb
    from paper_1812_10375_gb300.config import params_for
    build.build()
    coex, rng = coexistence(), np.random.default_rng(3)
    cases = [wl.Case("read", nx=nx, ny=ny, wall_rows=W, top_bc=top, T_bottom_over_Tc=wl.TS_OVER_TC + 0.05,
                     T_top_over_Tc=wl.TS_OVER_TC - 0.02, eos_T_fixed=False, g_y=-3e-5, Gw0=0.3, sites=[])
             for nx, ny, W in ((45, 37, 6), (640, 300, 9))]
    b = hlb.Batch([params_for(c, storage=storage, rho_l=coex["rho_l"], rho_v=coex["rho_v"])[0] for c in cases])
    dev = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    for i, c in enumerate(cases):
        rho0 = wl.tanh_film(c.ny, c.nx, coex["rho_l"], coex["rho_v"], c.wall_rows + 10.0)
        T0 = wl.layered_T(c.ny, c.nx, c.wall_rows, c.T_bottom(coex["Tc"]), coex["Ts"])
        b.set_fields(i, dev(rho0 * (1.0 + 0.01 * rng.standard_normal((c.ny, c.nx)))),
                     dev(T0 * (1.0 + 1e-3 * rng.standard_normal((c.ny, c.nx)))))
    for steps in (0, 1, 4):
        b.step(steps)
        for i, c in enumerate(cases):
            full = dict(zip(NAMES, b.read(i)))
            assert bool((full["rho"][:c.wall_rows] == 0).all()) and bool((full["rho"][c.wall_rows:-1] > 0).all())
            assert (float(full["rho"][-1].abs().max()) == 0.0) == (top == "wall")
            for n in (1, 2, 3):
                for names in itertools.combinations(NAMES, n):
                    got = {k: torch.full((c.ny, c.nx), 7.5, device="cuda") for k in NAMES}
                    torch.cuda.synchronize()
                    b.read_into(i, **{k: got[k] for k in names})
                    torch.cuda.synchronize()
                    for k in NAMES:
                        want = full[k] if k in names else torch.full_like(full[k], 7.5)
                        assert torch.equal(got[k], want), (steps, i, names, k)
