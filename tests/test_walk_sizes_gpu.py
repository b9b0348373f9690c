"""The energy walks where the other parity tests have no lattice: the one-warp walk's
three-row loop on a single lattice (segments of 13 rows and more: large lattices, with
and without 16-byte rows, the heater's edge in a later segment), and every split
variant with the heater's height, and the top wall's last fluid row, within the halo of
a neighbouring segment of 64 or 96 rows, where a wall flux could be counted twice.
Against the FP64 oracle; tolerances are those of the other parity tests."""
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


def segment_rows(nx, ny):
    """The one-warp walk's: the fewest, from 4 on, with at most 8 segments of 56 columns per SM."""
    L = 4
    while -(-nx // 56) * -(-ny // L) > 152 * 8:
        L += 1
    return L


def start(nx, ny, W, top):
    coex = coexistence()
    rng = np.random.default_rng(nx + ny + W)
    case = wl.Case("walk", nx=nx, ny=ny, wall_rows=W, top_bc=top, T_bottom_over_Tc=wl.TS_OVER_TC + 0.05,
                   T_top_over_Tc=wl.TS_OVER_TC - 0.02, eos_T_fixed=False, g_y=-3e-5, Gw0=0.3,
                   sites=[(nx / 3.0, 8.0, -0.3)])
    rho0 = wl.tanh_film(ny, nx, coex["rho_l"], coex["rho_v"], W + 10.0) * (1.0 + 0.01 * rng.standard_normal((ny, nx)))
    T0 = wl.layered_T(ny, nx, W, case.T_bottom(coex["Tc"]), coex["Ts"]) * (1.0 + 1e-3 * rng.standard_normal((ny, nx)))
    return coex, case, rho0, T0


def compare(gd, od, coex):
    rho, ux, uy, T = [t.cpu().numpy() for t in gd.read()]
    rho_o, ux_o, uy_o, T_o = od.fields()
    fl = od.fluid
    err = dict(rho=rel_linf(rho, rho_o, fl), T=rel_linf(T, T_o),
               u=float(max(np.abs(ux - ux_o)[fl].max(), np.abs(uy - uy_o)[fl].max()) / CS))
    print(err)
    assert max(err.values()) < TOL, err
    dg, do = gd.diag(), od.diag()
    tol = 2.0 * 3.0 * coex["rho_l"] * 6.0 * 0.1 * TOL * float(np.abs(od.T).max())
    for k in ("q_bottom", "q_interface", "q_top"):
        assert getattr(dg, k) == pytest.approx(do[k], abs=tol), k
    for k in ("mass", "energy", "rho_ave"):
        assert getattr(dg, k) == pytest.approx(do[k], rel=TOL), k
    assert dg.vapour_coverage == pytest.approx(do["vapour_coverage"], abs=1e-12)


@pytest.mark.parametrize("nx,ny,W,top,n_sub,steps", [
    (1100, 1000, 20, "convective", 1, 3), (1101, 1000, 35, "wall", 1, 3), (1062, 900, 16, "const_rho", 2, 2)])
def test_three_row_loop_on_one_lattice(nx, ny, W, top, n_sub, steps):
    L = segment_rows(nx, ny)
    assert L > 12 and W > L - 4
    coex, case, rho0, T0 = start(nx, ny, W, top)
    od = oracle_domain(case, coex, rho0=rho0, T0=T0, n_sub=n_sub).step(steps)
    gd = gpu_domain(case, coex, rho0=rho0, T0=T0, n_sub=n_sub)
    gd.step(steps)
    compare(gd, od, coex)


@pytest.mark.parametrize("nx,ny,W", [(70, 130, 61), (57, 131, 62), (64, 132, 64), (70, 133, 66), (70, 194, 93),
                                     (60, 196, 98)])
def test_wall_fluxes_near_the_edges_of_segments(nx, ny, W):
    from paper_1812_10375_gb300 import hlb
    coex, case, rho0, T0 = start(nx, ny, W, "wall")
    od = oracle_domain(case, coex, rho0=rho0, T0=T0).step(4)
    for v, kind in enumerate(hlb.variant_kinds()):
        if kind != hlb.HLB_KIND_SPLIT:
            continue
        gd = gpu_domain(case, coex, rho0=rho0, T0=T0)
        gd.set_tile_variant(v)
        gd.step(4)
        compare(gd, od, coex)
