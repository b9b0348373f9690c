"""Steps of one call hand the lagged scalars on inside the flow kernel where the lattice
has few flow tiles.  Calls of several steps (a graph's, the launches around it) leave
the same checkpoint, flux history and record, bit for bit, as as many calls of
one step: from one tile to about the 608 that are chained, around the edges of the
sum's two forms (128 and 256 tiles), tiles of 4, 8, 16 and 24 rows, with and without
an outlet that lags, one energy sub-step and more.  The sums are added in one
order on both ways, so nothing may differ."""
import numpy as np
import pytest

from paper_1812_10375_gb300 import workloads as wl

from helpers import coexistence, gpu_domain

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()


@pytest.mark.parametrize("nx,ny,W,top,n_sub", [
    (40, 20, 16, "convective", 1), (64, 58, 3, "wall", 1), (65, 133, 5, "convective", 2),
    (128, 260, 4, "convective", 1), (129, 133, 3, "const_rho", 1), (64, 521, 5, "convective", 1),
    (256, 262, 5, "wall", 1), (385, 301, 5, "convective", 1), (640, 300, 5, "convective", 1),
    (1024, 340, 5, "const_rho", 1), (1217, 485, 4, "convective", 1), (1281, 520, 4, "convective", 1)])
def test_calls_of_several_steps_equal_single_ones(nx, ny, W, top, n_sub):
    coex = coexistence()
    rng = np.random.default_rng(nx + ny)
    case = wl.Case("chain", nx=nx, ny=ny, wall_rows=W, top_bc=top, T_bottom_over_Tc=wl.TS_OVER_TC + 0.05,
                   T_top_over_Tc=wl.TS_OVER_TC - 0.02, eos_T_fixed=False, g_y=-3e-5, Gw0=0.3,
                   sites=[(nx / 3.0, 8.0, -0.3)])
    rho0 = wl.tanh_film(ny, nx, coex["rho_l"], coex["rho_v"], W + 10.0) * (1.0 + 0.01 * rng.standard_normal((ny, nx)))
    T0 = wl.layered_T(ny, nx, W, case.T_bottom(coex["Tc"]), coex["Ts"]) * (1.0 + 1e-3 * rng.standard_normal((ny, nx)))
    many, single = [gpu_domain(case, coex, rho0=rho0, T0=T0, n_sub=n_sub) for _ in range(2)]
    for n in (3, 1, 37, 2, 18):
        many.step(n)
        for _ in range(n):
            single.step(1)
        assert many.checkpoint() == single.checkpoint(), n
    assert many.diag() == single.diag()
    assert np.array_equal(many.flux_history(), single.flux_history())
