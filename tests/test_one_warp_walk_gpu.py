"""The one-warp energy walk and the rules that size it (segment rows, loop form, flow
tile) against the FP64 oracle, where they can go wrong: widths around the 56-column
strips and the 64-column flow tiles, with and without 16-byte rows; heater heights
on either side of a segment's and a flow tile's edge, so that each wall flux and
the vapour count come from the right row of blocks; both tops; a lattice tall and
wide enough for taller segments and the three-row loop.  Tolerances are those of the
other parity tests: 1e-5 of the largest value, u in sound speeds, and a face flux
within 2 lambda 1e-5 max|T|."""
import numpy as np
import pytest

from paper_1812_10375_gb300 import workloads as wl

from helpers import coexistence, gpu_domain, oracle_domain, rel_linf

pytestmark = pytest.mark.gpu
TOL = 1e-5
CS = 1.0 / np.sqrt(3.0)


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1812_10375_gb300 import build
    build.build()


@pytest.mark.parametrize("nx,ny,W,top,n_sub,steps", [
    (56, 30, 3, "convective", 1, 30), (57, 31, 4, "wall", 1, 30), (64, 41, 5, "convective", 2, 20),
    (65, 26, 8, "wall", 3, 20), (112, 33, 7, "const_rho", 1, 30), (58, 29, 12, "convective", 1, 30),
    (1500, 300, 13, "convective", 1, 8), (1198, 420, 17, "wall", 1, 6)])
def test_walk_matches_oracle(nx, ny, W, top, n_sub, steps):
    coex = coexistence()
    rng = np.random.default_rng(nx + ny)
    case = wl.Case("walk", nx=nx, ny=ny, wall_rows=W, top_bc=top, T_bottom_over_Tc=wl.TS_OVER_TC + 0.05,
                   T_top_over_Tc=wl.TS_OVER_TC - 0.02, eos_T_fixed=False, g_y=-3e-5, Gw0=0.3,
                   sites=[(nx / 3.0, 8.0, -0.3)])
    rho0 = wl.tanh_film(ny, nx, coex["rho_l"], coex["rho_v"], W + 10.0) * (1.0 + 0.01 * rng.standard_normal((ny, nx)))
    T0 = wl.layered_T(ny, nx, W, case.T_bottom(coex["Tc"]), coex["Ts"]) * (1.0 + 1e-3 * rng.standard_normal((ny, nx)))
    kw = dict(n_sub=n_sub)
    od = oracle_domain(case, coex, rho0=rho0, T0=T0, **kw).step(steps)
    gd = gpu_domain(case, coex, rho0=rho0, T0=T0, **kw)
    gd.step(steps)
    rho, ux, uy, T = [t.cpu().numpy() for t in gd.read()]
    rho_o, ux_o, uy_o, T_o = od.fields()
    fl = od.fluid
    err = dict(rho=rel_linf(rho, rho_o, fl), T=rel_linf(T, T_o),
               u=float(max(np.abs(ux - ux_o)[fl].max(), np.abs(uy - uy_o)[fl].max()) / CS))
    dg, do = gd.diag(), od.diag()
    print(nx, ny, err)
    assert max(err.values()) < TOL, err
    tol = 2.0 * 3.0 * coex["rho_l"] * 6.0 * 0.1 * TOL * float(np.abs(od.T).max())
    for k in ("q_bottom", "q_interface", "q_top"):
        assert getattr(dg, k) == pytest.approx(do[k], abs=tol), k
    for k in ("mass", "energy", "rho_ave"):
        assert getattr(dg, k) == pytest.approx(do[k], rel=TOL), k
    assert dg.vapour_coverage == pytest.approx(do["vapour_coverage"], abs=1e-12)
    assert dg.u_top == pytest.approx(do["u_top"], abs=TOL * CS)
