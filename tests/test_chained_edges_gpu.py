"""The edges of the rule that chains the steps of a call: lattices of exactly 608 flow
tiles, the most that are chained, and of a row more, with tiles by size (4 rows at 608,
8 rows beyond) and with 16-row tiles (variant 1: chained at 608, not beyond), and 128
tiles of either height and a row more, where the longer form of the sums begins.
Calls of several steps leave what as many calls of one step leave, bit for bit."""
import numpy as np
import pytest

from paper_1812_10375_gb300 import workloads as wl

from helpers import coexistence, gpu_domain

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant,nx,fluid_rows,tiles", [
    (0, 512, 304, 608), (0, 512, 305, 312), (1, 512, 1216, 608), (1, 512, 1217, 616), (1, 64, 2048, 128),
    (1, 64, 2049, 129), (0, 128, 256, 128), (0, 128, 257, 130)])
def test_edges_of_the_chaining_rule(variant, nx, fluid_rows, tiles):
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()
    W, ny, coex, rng = 5, fluid_rows + 5, coexistence(), np.random.default_rng(fluid_rows)
    ty = 16 if variant else (8 if (nx // 64) * -(-fluid_rows // 4) > 608 else 4)
    assert (nx // 64) * -(-fluid_rows // ty) == tiles
    case = wl.Case("chain", nx=nx, ny=ny, wall_rows=W, top_bc="convective", T_bottom_over_Tc=wl.TS_OVER_TC + 0.05,
                   T_top_over_Tc=wl.TS_OVER_TC - 0.02, eos_T_fixed=False, g_y=-3e-5, Gw0=0.3,
                   sites=[(nx / 3.0, 8.0, -0.3)])
    rho0 = wl.tanh_film(ny, nx, coex["rho_l"], coex["rho_v"], W + 10.0) * (1.0 + 0.01 * rng.standard_normal((ny, nx)))
    T0 = wl.layered_T(ny, nx, W, case.T_bottom(coex["Tc"]), coex["Ts"]) * (1.0 + 1e-3 * rng.standard_normal((ny, nx)))
    many, single = [gpu_domain(case, coex, rho0=rho0, T0=T0) for _ in range(2)]
    for d in (many, single):
        d.set_tile_variant(variant)
    for n in (3, 1, 18):
        many.step(n)
        for _ in range(n):
            single.step(1)
        assert many.checkpoint() == single.checkpoint(), n
    assert many.diag() == single.diag()
    assert np.array_equal(many.flux_history(), single.flux_history())
