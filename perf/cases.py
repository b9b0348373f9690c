"""Performance cases of the framework: what a program that uses it has it do.

Two kinds of work carry the framework: coupled steps of the thermal lattice
Boltzmann model (single domains and batches of domains, advanced some steps and
then read back), and the sweep surrogate (a training step, a forward call).

A lattice case starts from a boiling pool in full swing, made from the seed: liquid
with a few vapour bubbles, a heater with the temperature drop of its heat
flux, a thermal boundary layer above it, and a little noise on density and
temperature; or from a liquid film, or a liquid slab between two walls.  One
pass advances every domain by ``steps`` steps and reads the fields and the
diagnostics back, as a program does at each of its sampling points; the next
pass goes on from there.

``exact`` evaluates the same steps with plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1812_10375_gb300 import hlb, surrogate

TC, RHO_L, RHO_V = 0.10938300611120137, 6.498945763287885, 0.379678999399721
TS = 0.86 * TC
CV, K = 6.0, 0.1
RHO_W, LAM_W = 3.0 * RHO_L, 3.0 * RHO_L * CV * K
GRAVITY, GW0 = -3e-5, 0.3


# ---------------------------------------------------------------- the cases
def _domain(name, nx, ny, steps, **kw):
    c = dict(kind="domain", nx=nx, ny=ny, steps=steps, start="pool", wall_rows=25, top="convective", superheat=0.1,
             sites=5, q_in=0.0, n_sub=1, heater=1.0, storage="deviation", scheme="fv")
    c.update(kw)
    return dict(c, name=name) if name else c


def _batch(name, points, lo, hi, stride, aspect, steps, **kw):
    c = dict(kind="batch", points=points, lo=lo, hi=hi, stride=stride, aspect=aspect, steps=steps, wall_rows=25,
             superheat_lo=0.02, superheat_hi=0.30, sites=5)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one step of a small ragged box, its fields and diagnostics read after it
        _domain("box_45x37_each_step", 45, 37, 1, wall_rows=6, superheat=0.12, sites=2),
        # a bubble-departure run samples a narrow column every 20 steps
        _domain("departure_64x200", 64, 200, 20, wall_rows=10, superheat=0.11, sites=1),
        # film evaporation on a heater with an imposed flux, constant-density top
        _domain("film_flux_200x100", 200, 100, 48, start="film", wall_rows=20, top="const_rho", superheat=0.0,
                sites=0, q_in=2e-4),
        # pool boiling on the benchmark's single lattice
        _domain("pool_400x400", 400, 400, 64),
        # a heater that conducts too well for one energy sub-step (N = 3), odd sizes, plain population storage
        _domain("substeps_385x301", 385, 301, 32, superheat=0.08, sites=4, n_sub=3, heater=5.0, storage="plain"),
        # the isotropic diffusion scheme the method is compared against: slab between two walls
        _domain("iso_slab_120x200", 120, 200, 32, start="slab", wall_rows=1, top="wall", superheat=0.0, sites=0,
                scheme="iso"),
        # the largest single lattice of the benchmark
        _domain("pool_2048x2048", 2048, 2048, 24),
        # runs that train the surrogate: many small domains at once
        _batch("training_runs_48", 48, 64, 96, 32, 1.25, 50, wall_rows=10, sites=2),
        # the paper's boiling curve: 14 superheats on one geometry
        _batch("curve_14_400x600", 14, 400, 400, 64, 1.5, 32, sites=3),
        # the boiling-curve sweep, the benchmark's headline workload
        _batch("sweep_32", 32, 256, 512, 64, 1.0, 48),
        # one training step of the surrogate at its training batch
        dict(name="surrogate_train_64", kind="train", batch=64, L0=500, H=256, NS=3),
        # the early-stop policy asks the network about a calibration set
        dict(name="surrogate_forward_96", kind="forward", batch=96, L0=500, H=256, NS=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.40:
        nx, ny = _log_int(rng, 32, 2048), _log_int(rng, 48, 2048)
        wall = rng.randint(2, min(25, ny // 4))
        top = rng.choice(["convective", "convective", "wall"])
        steps = rng.choice([1, 4, 16, 20, 33, 48])
        steps = max(1, min(steps, int(1e8 // (nx * ny))))
        n_sub, heater = rng.choice([(1, 1.0), (1, 1.0), (1, 1.0), (2, 3.0), (3, 5.0)])
        return _domain(None, nx, ny, steps, wall_rows=wall, top=top, superheat=round(rng.uniform(0.02, 0.05 if top == "wall" else 0.2), 3),
                       sites=rng.randint(0, max(1, nx // 64)), n_sub=n_sub, heater=heater,
                       storage=rng.choice(["deviation", "deviation", "plain"]))
    if what < 0.50:
        nx, ny = _log_int(rng, 20, 800), _log_int(rng, 90, 400)
        return _domain(None, nx, ny, rng.choice([10, 20, 48]), start="film", wall_rows=20, top="const_rho",
                       superheat=0.0, sites=0, q_in=2e-4, scheme=rng.choice(["fv", "fv", "iso"]))
    if what < 0.56:
        return _domain(None, _log_int(rng, 4, 400), _log_int(rng, 100, 400), rng.choice([16, 32]), start="slab",
                       wall_rows=1, top="wall", superheat=0.0, sites=0, scheme=rng.choice(["iso", "fv"]))
    if what < 0.80:
        lo = _log_int(rng, 48, 400)
        hi = rng.randint(lo, min(2 * lo, 512))
        points = _log_int(rng, 2, 40)
        aspect = rng.choice([1.0, 1.0, 1.25, 1.5])
        steps = max(4, min(rng.choice([16, 20, 48, 64]), int(2e8 // (points * hi * hi * aspect))))
        return _batch(None, points, lo, hi, rng.choice([1, 7, 32, 64]), aspect, steps,
                      wall_rows=rng.randint(5, min(25, lo // 4)), sites=rng.randint(1, max(1, lo // 64)))
    return dict(kind=rng.choice(["train", "forward"]), batch=_log_int(rng, 4, 256), L0=rng.choice([100, 250, 500, 512]),
                H=rng.choice([64, 200, 256]), NS=rng.choice([2, 3]))


# ------------------------------------------------------------------- inputs
def _points(case):
    """The domains of a lattice case as single-domain cases."""
    if case["kind"] == "domain":
        return [case]
    n = case["points"]
    sides = list(range(case["lo"], case["hi"] + 1, case["stride"]))
    out = []
    for i in range(n):
        side = sides[(7 * i) % len(sides)]
        heat = case["superheat_lo"] + (case["superheat_hi"] - case["superheat_lo"]) * ((5 * i) % n) / max(1, n - 1)
        out.append(_domain(None, side, int(round(side * case["aspect"])), case["steps"], wall_rows=case["wall_rows"],
                           superheat=heat, sites=case["sites"] + i % 3))
    return out


def _T_walls(c):
    """(T_bottom, T_top) of a domain."""
    if c["start"] == "slab":
        return 1.0, 0.0
    return TS + c["superheat"] * TC, TS


def _lam_w(c):
    return RHO_V * CV * K if c["start"] == "slab" else LAM_W * c["heater"]


def _sites(c, seed):
    """Nucleation sites (centre, width, minimum) spread over the width."""
    r = np.random.default_rng([seed, 1])
    n = c["sites"]
    return [(float(int((k + r.uniform(0.2, 0.8)) * c["nx"] / n)), 10.0, (0.0, -0.3, -0.6)[k % 3]) for k in range(n)]


def _fields(c, seed):
    """Initial density and temperature of a domain, FP32 on the GPU."""
    nx, ny, W = c["nx"], c["ny"], c["wall_rows"]
    r = np.random.default_rng([seed, 2])
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(r.integers(1 << 40)))
    y = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]
    T_bottom, _ = _T_walls(c)
    span = RHO_L - RHO_V
    # interfaces carry a wave of a few cells, as evaporating ones do
    wave = min(4.0, nx / 12.0) * torch.cos(2.0 * math.pi * (x / nx * max(1, nx // 60) + r.uniform()))
    if c["start"] == "slab":
        rho = RHO_V + 0.5 * span * (torch.tanh(2.0 * (y - ny / 4.0 - wave) / 5.0)
                                    - torch.tanh(2.0 * (y - 0.75 * ny + wave) / 5.0))
        T = 1.0 - y / (ny - 1.0) + 0.0 * x
    elif c["start"] == "film":
        rho = 0.5 * (RHO_L + RHO_V) - 0.5 * span * torch.tanh(2.0 * (y - W - 30.0 - wave) / 5.0)
        T = torch.where(y < W, TS + c["q_in"] * (W - y) / _lam_w(c), torch.full_like(y, TS)) + 0.0 * x
    else:
        liquid = torch.ones((ny, nx), dtype=torch.float64, device=dev)
        for _ in range(1 + min(400, nx * ny // 8000)):
            rad = min(r.uniform(6.0, 18.0), nx / 6.0, (ny - W) / 6.0)
            xc, yc = int(r.integers(nx)), W + r.uniform(0.0, 0.7) * (ny - W)
            half = min(int(rad) + 16, (nx - 1) // 2)
            y0, y1 = max(0, int(yc - rad - 16)), min(ny, int(yc + rad + 17))
            at = torch.arange(-half, half + 1, device=dev)
            cols, rows = (xc + at) % nx, torch.arange(y0, y1, device=dev)[:, None]
            d = torch.sqrt((at * at)[None, :] + (rows - yc) ** 2)
            liquid[rows, cols] = liquid[rows, cols] * 0.5 * (1.0 + torch.tanh(2.0 * (d - rad) / 5.0))
        rho = RHO_V + span * liquid
        drop = 0.3 * c["superheat"] * TC
        T_face = T_bottom - drop
        T = torch.where(y < W, T_bottom - drop * y / W, TS + (T_face - TS) * torch.exp(-(y - W) / 15.0)) + 0.0 * x
    rho = rho * (1.0 + 1e-3 * torch.randn((ny, nx), dtype=torch.float64, device=dev, generator=gen))
    T = T * (1.0 + 1e-4 * torch.randn((ny, nx), dtype=torch.float64, device=dev, generator=gen))
    return rho.float().contiguous(), T.float().contiguous()


def _params(c):
    p = hlb.default_params(c["nx"], c["ny"])
    p.wall_rows = c["wall_rows"]
    p.top_bc = hlb.TOP_KIND[c["top"]]
    p.eos_T_fixed = 1 if c["start"] == "slab" else 0
    p.storage = hlb.HLB_STORE_PLAIN if c["storage"] == "plain" else hlb.HLB_STORE_DEVIATION
    p.g_y = 0.0 if c["start"] == "slab" else GRAVITY
    p.Gw0 = GW0
    p.T_bottom, p.T_top = _T_walls(c)
    p.rho_l, p.rho_v = RHO_L, RHO_V
    p.n_sub = c["n_sub"]
    p.lambda_w = _lam_w(c)
    if c["scheme"] == "iso":
        p.diffusion = hlb.HLB_DIFF_ISO
    if c["q_in"]:
        p.bottom_bc = hlb.HLB_BOTTOM_FLUX
        p.q_in = c["q_in"]
    return p


def _surrogate_arrays(case, seed):
    """Network input, targets, parameters and Adam state, mid-training."""
    r = np.random.default_rng([seed, 3])
    B, L0, NS = case["batch"], case["L0"], case["NS"]
    t = np.linspace(0.0, 4.0, L0)[None, :]
    hist = np.exp(-r.uniform(0.2, 1.0, (B, 1)) * t) - 0.4 + 0.1 * r.standard_normal((B, L0))
    a = dict(hist=hist, scal=r.standard_normal((B, NS)), target=r.standard_normal(B))
    a = {k: torch.tensor(v, dtype=torch.float32, device="cuda") for k, v in a.items()}
    a["label"] = torch.tensor(r.integers(0, 5, B), dtype=torch.int32, device="cuda")
    return a, r


def _shapes(case):
    C1, C2, C3, ks, H, W0 = 16, 32, 32, 5, case["H"], 32 + case["NS"]
    return [(C1, 1, ks), (C1,), (C2, C1, ks), (C2,), (C3, C2, ks), (C3,), (H, W0), (H,), (H, H), (H,), (6, H), (6,)]


def _net_state(case, r):
    parts = [0.02 * r.standard_normal(s) if len(s) == 1 else r.uniform(-1, 1, s) * math.sqrt(6.0 / np.prod(s[1:]))
             for s in _shapes(case)]
    p = np.concatenate([v.ravel() for v in parts])
    m, v = 5e-4 * r.standard_normal(p.size), 1e-6 * r.uniform(0.5, 1.5, p.size)
    return [torch.tensor(q, dtype=torch.float32, device="cuda") for q in (p, m, v)]


def prepare(case, seed):
    if case["kind"] in ("train", "forward"):
        a, r = _surrogate_arrays(case, seed)
        cfg = surrogate.default_config()
        cfg.L0, cfg.H, cfg.NS = case["L0"], case["H"], case["NS"]
        net = surrogate.Net(cfg, max_batch=case["batch"])
        for own, made in zip((net.params, net.m, net.v), _net_state(case, r)):
            own.copy_(made)
        net.t = 200
        return dict(case=case, net=net, **a)
    points = _points(case)
    if case["kind"] == "domain":
        d = hlb.Domain(_params(case))
        d.set_fields(*_fields(case, seed))
        if case["sites"]:
            d.set_nucleation_sites(_sites(case, seed))
        return dict(case=case, domain=d)
    b = hlb.Batch([_params(c) for c in points])
    for i, c in enumerate(points):
        b.set_fields(i, *_fields(c, seed + 1000 * i))
        b.set_nucleation_sites(i, _sites(c, seed + 1000 * i))
    # the program's own result arrays, one stretch per point
    cells = sum(c["nx"] * c["ny"] for c in points)
    flat = {k: torch.empty(cells, dtype=torch.float32, device="cuda") for k in ("rho", "T")}
    views, at = [], 0
    for c in points:
        n = c["nx"] * c["ny"]
        views.append({k: v[at:at + n] for k, v in flat.items()})
        at += n
    return dict(case=case, batch=b, flat=flat, views=views)


def _numbers(dg):
    return dict(mass=dg.mass, energy=dg.energy, rho_ave=dg.rho_ave, q_interface=dg.q_interface)


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        net = state["net"]
        loss, grad = net.loss_grad(state["hist"], state["scal"], state["target"], state["label"])
        net.adam(lr=2e-3)
        return dict(loss=loss, grad=grad, params=net.params, m=net.m, v=net.v)
    if case["kind"] == "forward":
        return state["net"].forward(state["hist"], state["scal"])
    if case["kind"] == "domain":
        d = state["domain"]
        d.step(case["steps"])
        rho, ux, uy, T = d.read()
        return dict(rho=rho, ux=ux, uy=uy, T=T, **_numbers(d.diag()))
    b = state["batch"]
    b.step(case["steps"])
    for i, v in enumerate(state["views"]):
        b.read_into(i, rho=v["rho"], T=v["T"])
    torch.cuda.current_stream().wait_stream(b.stream)
    return dict(rho=state["flat"]["rho"], T=state["flat"]["T"],
                q_interface=[b.diag(i).q_interface for i in range(b.n)])


# --------------------------------------------------------------------- work
def work(case):
    if case["kind"] in ("train", "forward"):
        B, L0, H, W0 = case["batch"], case["L0"], case["H"], 32 + case["NS"]
        L1 = (L0 - 5) // 2 + 1
        L2 = (L1 - 5) // 2 + 1
        L3 = (L2 - 5) // 2 + 1
        conv1 = 16 * L1 * 5
        rest = 32 * L2 * 80 + 32 * L3 * 160 + H * W0 + H * H + 6 * H
        n = sum(int(np.prod(s)) for s in _shapes(case))
        if case["kind"] == "forward":
            return dict(bytes=4 * (n + B * (L0 + case["NS"] + 6)), flops=2 * B * (conv1 + rest))
        # weight gradients as much again as the forward pass, data gradients too but for the first layer
        return dict(bytes=4 * (7 * n + B * (L0 + case["NS"] + 2)), flops=2 * B * (2 * conv1 + 3 * rest) + 12 * n)
    total = flops = 0
    for c in _points(case):
        solid = c["nx"] * (c["wall_rows"] + (1 if c["top"] == "wall" else 0))
        fluid = c["nx"] * c["ny"] - solid
        # a step: nine populations and T in and out of a fluid cell, T of a solid cell
        total += c["steps"] * (80 * fluid + 8 * solid)
        total += 4 * c["nx"] * c["ny"] * (4 if case["kind"] == "domain" else 2)
        # streaming, EOS, forces and collision; four RK4 stages a sub-step and their coefficients
        flops += c["steps"] * (fluid * (260 + 180 * c["n_sub"]) + solid * 60 * c["n_sub"])
    return dict(bytes=total, flops=flops)


# -------------------------------------------------------------------- exact
EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
PA, PB, PR_ = 3.0 / 49.0, 2.0 / 21.0, 1.0
KAPPA = 0.37464 + 1.54226 * 0.344 - 0.26992 * 0.344 * 0.344


def _x(a, d):
    """b[..., x] = a[..., x + d], periodic."""
    return torch.roll(a, -d, -1) if d else a


def _rows(a):
    """a with a copy of its first and last row below and above it."""
    return torch.cat([a[:1], a, a[-1:]])


def _nb(P, dx, dy):
    """From P = _rows(a): b[y, x] = a[y + dy, x + dx]."""
    return _x(P[1 + dy:P.shape[0] - 1 + dy], dx)


def _grad(a):
    P = _rows(a)
    ne, nw, se, sw = _nb(P, 1, 1), _nb(P, -1, 1), _nb(P, 1, -1), _nb(P, -1, -1)
    gx = (_nb(P, 1, 0) - _nb(P, -1, 0)) / 3.0 + (ne - sw) / 12.0 + (se - nw) / 12.0
    gy = (_nb(P, 0, 1) - _nb(P, 0, -1)) / 3.0 + (ne - sw) / 12.0 + (nw - se) / 12.0
    return gx, gy


class _Exact:
    """The coupled step of one domain in 64 bits, one plain array expression after the other."""

    def __init__(self, c, seed):
        self.c = c
        self.T_bottom, self.T_top = _T_walls(c)
        rho, T = (v.double() for v in _fields(c, seed))
        nx, ny, W = c["nx"], c["ny"], c["wall_rows"]
        self.top_wall = c["top"] == "wall"
        self.lo, self.hi = W, ny - 1 if self.top_wall else ny
        self.flux = c["q_in"] != 0.0
        if not self.flux:
            T[0] = self.T_bottom
        if self.top_wall:
            T[-1] = self.T_top
        self.T = T
        rho = rho[self.lo:self.hi]
        self.w = torch.tensor(WT, dtype=torch.float64, device=rho.device)
        self.f = self.w[:, None, None] * rho
        self.entering = self.f[[4, 7, 8], -1].clone()
        self.rho_ave, self.U = rho.mean(), rho.new_zeros(())
        g = np.full(nx, GW0)
        at = np.arange(nx, dtype=np.float64)
        for xc, width, low in _sites(c, seed):
            d = np.abs(at - xc)
            d = np.minimum(d, nx - d)
            g = np.where(d <= width / 2, np.minimum(g, low + (GW0 - low) * d / (width / 2)), g)
        self.Gw = torch.tensor(g, dtype=torch.float64, device=rho.device)
        rows = torch.full((ny, 1), RHO_W * CV, dtype=torch.float64, device=rho.device)
        self.rcv_w = rows
        self.lam_w = torch.full_like(rows, _lam_w(c))

    def full(self, a):
        """A fluid field on the whole lattice, 0 in the walls."""
        out = a.new_zeros((self.c["ny"], self.c["nx"]))
        out[self.lo:self.hi] = a
        return out

    def pulled(self):
        f = self.f
        new = torch.empty_like(f)
        for i in range(9):
            s = _x(f[i], -EX[i])
            if EY[i] == 0:
                new[i] = s
            elif EY[i] > 0:
                new[i, 1:] = s[:-1]
                new[i, 0] = f[OPP[i], 0]
            else:
                new[i, :-1] = s[1:]
                if self.top_wall:
                    new[i, -1] = f[OPP[i], -1]
        if not self.top_wall:
            for j, i in enumerate((4, 7, 8)):
                if self.c["top"] == "const_rho":
                    new[i, -1] = WT[i] * RHO_V
                else:
                    new[i, -1] = (self.entering[j] + self.U * new[i, -2]) / (1.0 + self.U)
                    self.entering[j] = new[i, -1]
        return new

    def flow(self):
        c = self.c
        f = self.pulled()
        rho = f.sum(0)
        T = torch.full_like(rho, TS) if c["start"] == "slab" else self.T[self.lo:self.hi]
        al = 1.0 + KAPPA * (1.0 - torch.sqrt(T.clamp(min=0.0) / TC))
        p = rho * PR_ * T / (1.0 - PB * rho) - PA * al * al * rho * rho / (1.0 + 2.0 * PB * rho - (PB * rho) ** 2)
        psi = torch.sqrt((2.0 * (rho / 3.0 - p)).clamp(min=0.0))
        P = _rows(psi)
        sx, sy = torch.zeros_like(psi), torch.zeros_like(psi)
        for i in range(1, 9):
            n = _nb(P, EX[i], EY[i]).clone()
            if EY[i] < 0:
                n[0] = psi[0]  # a solid neighbour carries the node's own psi
            if EY[i] > 0 and self.top_wall:
                n[-1] = psi[-1]
            om = 1.0 / 3.0 if i < 5 else 1.0 / 12.0
            sx += om * EX[i] * n
            sy += om * EY[i] * n
        Fx, Fmy = psi * sx, psi * sy  # G = -1
        Fy = Fmy + (rho - self.rho_ave) * (0.0 if c["start"] == "slab" else GRAVITY)
        Fy[0] -= self.Gw * psi[0] ** 2 / 6.0
        if self.top_wall:
            Fy[-1] += self.Gw * psi[-1] ** 2 / 6.0
        jx = sum(EX[i] * f[i] for i in range(9) if EX[i])
        jy = sum(EY[i] * f[i] for i in range(9) if EY[i])
        ux, uy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        # moments rho, e, zeta, jx, qx, jy, qy, pxx, pxy and their relaxation
        rows, norm = [], []
        for i in range(9):
            e2 = EX[i] ** 2 + EY[i] ** 2
            rows.append([1.0, -4.0 + 3.0 * e2, 4.0 - 10.5 * e2 + 4.5 * e2 * e2, EX[i], (-5.0 + 3.0 * e2) * EX[i],
                         EY[i], (-5.0 + 3.0 * e2) * EY[i], EX[i] ** 2 - EY[i] ** 2, EX[i] * EY[i]])
        M = torch.tensor(rows, dtype=torch.float64, device=rho.device).T
        u2, uF = ux * ux + uy * uy, ux * Fx + uy * Fy
        tau = (1.0 + (rho - RHO_V) / (RHO_L - RHO_V) * (0.8 - 1.0)).clamp(0.8, 1.0)
        psi2 = psi * psi
        fm = torch.where(psi2 > 0, (Fx * Fx + Fmy * Fmy) / torch.where(psi2 > 0, psi2, torch.ones_like(psi2)), 0.0 * psi2)
        extra = 12.0 * 0.107 * fm / (1.0 / 0.8 - 0.5)
        one = torch.ones_like(rho)
        meq = (rho, rho * (-2.0 + 3.0 * u2), rho * (1.0 - 3.0 * u2), rho * ux, -rho * ux, rho * uy, -rho * uy,
               rho * (ux * ux - uy * uy), rho * ux * uy)
        S = (0.0 * rho, 6.0 * uF + extra, -6.0 * uF - extra, Fx, -Fx, Fy, -Fy, 2.0 * (ux * Fx - uy * Fy),
             ux * Fy + uy * Fx)
        s = (one, 0.8 * one, 0.8 * one, one, 1.1 * one, one, 1.1 * one, 1.0 / tau, 1.0 / tau)
        out = torch.zeros_like(f)
        for q in range(9):
            m = sum(float(M[q, i]) * f[i] for i in range(9) if float(M[q, i]))
            star = (m - s[q] * (m - meq[q]) + (1.0 - 0.5 * s[q]) * S[q]) / float((M[q] ** 2).sum())
            for i in range(9):
                if float(M[q, i]):
                    out[i] += float(M[q, i]) * star
        self.f = out
        return rho, ux, uy

    def energy(self, rho, ux, uy):
        c, ny, W = self.c, self.c["ny"], self.c["wall_rows"]
        wall = torch.ones((ny, 1), dtype=torch.bool, device=rho.device)
        wall[self.lo:self.hi] = False
        held = torch.zeros_like(wall)
        held[0] = not self.flux
        held[-1] = self.top_wall
        rf, ux, uy = self.full(rho), self.full(ux), self.full(uy)
        lam = torch.where(wall, self.lam_w, rf * CV * K)
        rcv = torch.where(wall, self.rcv_w, rf * CV)
        safe = torch.where(wall, torch.ones_like(rf), rf)
        divu = _grad(ux)[0] + _grad(uy)[1]
        P = _rows(lam)
        faces = [(dx, dy, 2.0 / (1.0 / lam + 1.0 / _nb(P, dx, dy))) for dx, dy in ((1, 0), (-1, 0), (0, 1), (0, -1))]
        glx, gly = _grad(lam)

        def rhs(T):
            P = _rows(T)
            gx, gy = _grad(T)
            if c["scheme"] == "iso":
                lap = (_nb(P, 1, 1) + _nb(P, -1, 1) + _nb(P, 1, -1) + _nb(P, -1, -1) + 4.0 * (
                    _nb(P, 1, 0) + _nb(P, -1, 0) + _nb(P, 0, 1) + _nb(P, 0, -1)) - 20.0 * T) / 6.0
                k = (lam * lap + glx * gx + gly * gy) / rcv
            else:
                k = sum(l * (_nb(P, dx, dy) - T) for dx, dy, l in faces) / rcv
            if self.flux:
                k[0] += c["q_in"] / rcv[0]
            s = torch.sqrt(T.clamp(min=0.0) / TC)
            heat = safe * PR_ * T / (1.0 - PB * safe) + PA * KAPPA * s * (1.0 + KAPPA * (1.0 - s)) * safe ** 2 / (
                1.0 + 2.0 * PB * safe - (PB * safe) ** 2)
            k = torch.where(wall, k, k - ux * gx - uy * gy - heat / rcv * divu)
            return torch.where(held, 0.0 * k, k)

        def fluxes(T):
            return (faces[3][2][W] * (T[W - 1] - T[W])).sum()

        T, dt, q = self.T, 1.0 / c["n_sub"], 0.0
        for _ in range(c["n_sub"]):
            h1 = rhs(T)
            T2 = T + 0.5 * dt * h1
            h2 = rhs(T2)
            T3 = T + 0.5 * dt * h2
            h3 = rhs(T3)
            T4 = T + dt * h3
            q = q + dt / 6.0 * (fluxes(T) + 2.0 * fluxes(T2) + 2.0 * fluxes(T3) + fluxes(T4))
            T = T + dt / 6.0 * (h1 + 2.0 * h2 + 2.0 * h3 + rhs(T4))
        self.T = T
        return q / c["nx"], rcv

    def go(self):
        for _ in range(self.c["steps"]):
            rho, ux, uy = self.flow()
            q, rcv = self.energy(rho, ux, uy)
            self.rho_ave = rho.mean()
            self.U = self.full(uy)[-2].mean().clamp(min=0.0)
        return dict(rho=self.full(rho), ux=self.full(ux), uy=self.full(uy), T=self.T, mass=float(rho.sum()),
                    energy=float((rcv * self.T).sum()), rho_ave=float(self.rho_ave), q_interface=float(q))


def _exact_net(case, seed):
    a, r = _surrogate_arrays(case, seed)
    p, m, v = (t.double() for t in _net_state(case, r))
    p.requires_grad_(case["kind"] == "train")
    parts, at = [], 0
    for s in _shapes(case):
        n = int(np.prod(s))
        parts.append(p[at:at + n].reshape(s))
        at += n
    h = a["hist"].double()[:, None, :]
    for k in (0, 2, 4):
        cols = h.unfold(2, 5, 2)
        h = torch.relu(torch.einsum("bctk,ock->bot", cols, parts[k]) + parts[k + 1][None, :, None])
    h = torch.cat([h.mean(2), a["scal"].double()], 1)
    h = torch.relu(h @ parts[6].T + parts[7])
    h = torch.relu(h @ parts[8].T + parts[9])
    y = h @ parts[10].T + parts[11]
    if case["kind"] == "forward":
        return y
    mse = ((y[:, 0] - a["target"].double()) ** 2).mean()
    ce = (torch.logsumexp(y[:, 1:], 1) - y[:, 1:].gather(1, a["label"].long()[:, None])[:, 0]).mean()
    (g,) = torch.autograd.grad(mse + ce, p)
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    new = p.detach() - 2e-3 * (m / (1 - 0.9 ** 201)) / (torch.sqrt(v / (1 - 0.999 ** 201)) + 1e-8)
    return dict(loss=torch.stack([mse, ce]).detach(), grad=g, params=new, m=m, v=v)


def exact(case, seed):
    with torch.no_grad() if case["kind"] != "train" else torch.enable_grad():
        if case["kind"] in ("train", "forward"):
            return _exact_net(case, seed)
        points = _points(case)
        if sum(c["nx"] * c["ny"] * c["steps"] * c["n_sub"] for c in points) > 4e8:
            return None
        if case["kind"] == "domain":
            return _Exact(case, seed).go()
        got = [_Exact(c, seed + 1000 * i).go() for i, c in enumerate(points)]
        return dict(rho=torch.cat([g["rho"].reshape(-1) for g in got]), T=torch.cat([g["T"].reshape(-1) for g in got]),
                    q_interface=[g["q_interface"] for g in got])
