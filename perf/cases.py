"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is a plain dict; ``prepare`` makes what a program holds before its call (initial
fields, the simulation handle), ``run`` is one pass through the public entry points, ``work``
the bytes and operations the pass cannot do without, and ``exact`` the same outputs from a
plain FP64 torch restatement of the equations (arXiv 2505.10899, Eqs. 20-37), which shares no
code with the library.  The set-ups are those of the paper's Sec. 4 and of ``workloads``:
droplets at rest, the sheared cavity, the liquid film between walls, the single vortex, the
batch of uneven cases, one large grid, liquid threads and balls in three dimensions, and the
reverse mode.  Centres, radii and speeds come from the seed; droplet centres lie off the nodes.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2505_10899_gb300 import adjoint, lbm, lbm3

EDGES = (64, 96, 128, 192, 256, 384, 512)  # square edges of the batched droplet cases


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # droplet volume against time (Sec. 4.1): a short call and a labelled volume per sample;
        # launches and the read-back count
        dict(name="droplets_128x64_f32", kind="droplets", nx=128, ny=64, precision="f32", steps=10),
        # film between resting walls (Sec. 4.3) on the 200 x 100 grid class, odd sizes: a long
        # run of a small grid, phi read back at its end
        dict(name="film_201x101_f32", kind="film", nx=201, ny=101, precision="f32", steps=500),
        # droplet in the sheared cavity (Sec. 4.4, 512 x 256): L2-resident long run
        dict(name="cavity_512x256_f32", kind="cavity", nx=512, ny=256, precision="f32", steps=256),
        # single vortex (Sec. 4.2): the phase field alone
        dict(name="vortex_256_f32", kind="vortex", nx=256, ny=256, precision="f32", steps=256),
        # parameter study: 512 uneven cases in one batch, volumes of every step
        dict(name="batch_512_f32", kind="batch", ncases=512, precision="f32", steps=32),
        # one grid far larger than L2
        dict(name="lattice_8192x4096_f32", kind="lattice", mx=32, my=16, cell_x=256, cell_y=256,
             precision="f32", steps=32),
        # the precise run of a part of the study
        dict(name="batch_64_f64", kind="batch", ncases=64, precision="f64", steps=8),
        # the liquid thread of Eq. 45 in three dimensions, as the experiments run it (autotuned,
        # phi read back after a run of steps), in both storage precisions
        dict(name="column_256_f32", kind="column", nx=256, ny=256, nz=256, precision="f32",
             steps=200),
        dict(name="column_256_f16", kind="column", nx=256, ny=256, nz=256, precision="f16",
             steps=200),
        # a translating ball in a small uneven box, untuned, all fields read back
        dict(name="ball_90x75x66_f32", kind="ball", nx=90, ny=75, nz=66, precision="f32",
             steps=100),
        # gradient of the Taylor deformation in the sheared cavity (walls), FP32
        dict(name="gradient_512x256_f32", kind="gradient", nx=512, ny=256, walls=True,
             precision="f32", steps=200),
        # the same objective on a periodic grid in the default precision
        dict(name="gradient_384x192_f64", kind="gradient", nx=384, ny=192, walls=False,
             precision="f64", steps=32),
    ]


def _spread(rng, lo, hi):
    """An integer, spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(("droplets", "film", "cavity", "vortex", "batch", "lattice", "column",
                       "ball", "gradient"))
    prec = "f64" if rng.random() < 0.25 else "f32"
    few = 4 if prec == "f64" else 1  # FP64 steps take longer
    if kind in ("droplets", "film", "cavity", "vortex"):
        nx, ny = _spread(rng, 64, 768), _spread(rng, 48, 512)
        if rng.random() < 0.5:  # widths that the bulk copies can take
            nx = (nx + 3) // 4 * 4
        if kind == "vortex":
            ny = nx = min(nx, 512)
        steps = _spread(rng, 2, 20) if kind == "droplets" else _spread(rng, 60, 500) // few
        return dict(kind=kind, nx=nx, ny=ny, precision=prec, steps=steps)
    if kind == "batch":
        n = _spread(rng, 4, 400) if prec == "f32" else _spread(rng, 2, 48)
        return dict(kind=kind, ncases=n, precision=prec, steps=_spread(rng, 4, 32) // few + 1)
    if kind == "lattice":
        return dict(kind=kind, mx=_spread(rng, 4, 30), my=_spread(rng, 4, 16),
                    cell_x=rng.randint(150, 256), cell_y=rng.randint(150, 256),
                    precision="f32", steps=_spread(rng, 8, 32))
    if kind == "column":
        p = rng.choice(("f32", "f16", "f64"))
        side = rng.choice((64, 96, 100, 128, 160, 192, 256)) if p != "f64" else rng.choice((48, 64, 80))
        return dict(kind=kind, nx=side, ny=side, nz=_spread(rng, 64, 256) if p != "f64" else 64,
                    precision=p, steps=_spread(rng, 20, 160) // (4 if p == "f64" else 1))
    if kind == "ball":
        p = rng.choice(("f32", "f32", "f16", "f64"))
        s = [_spread(rng, 24, 150 if p != "f64" else 64) for _ in range(3)]
        return dict(kind=kind, nx=s[0], ny=s[1], nz=s[2], precision=p, steps=_spread(rng, 10, 100))
    return dict(kind="gradient", nx=_spread(rng, 96, 512), ny=_spread(rng, 64, 256),
                walls=rng.random() < 0.5, precision=prec, steps=_spread(rng, 16, 150) // few)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _params2(nx, ny, **kw):
    """The case dictionary of one 2-D grid (Sec. 4.1 physics unless said otherwise)."""
    c = dict(nx=int(nx), ny=int(ny), flow="coupled", W=4.0, sigma=1e-3, xi=1e-10, tau_g=0.8,
             rho_l=1.0, rho_g=1.0, tau_f_l=1.0, tau_f_g=1.0)
    c["lambda"] = 0.5
    c.update(kw)
    return c


def _profile(dist, W):
    return 0.5 * (1.0 + torch.tanh(2.0 * dist / W))


def _axis(n, c, periodic=True):
    d = torch.arange(n, dtype=torch.float64, device="cuda") - c
    return d - n * torch.round(d / n) if periodic else d


def _disc(nx, ny, cx, cy, R, W, periodic=True):
    dx, dy = _axis(nx, cx, periodic)[None, :], _axis(ny, cy, periodic)[:, None]
    return _profile(R - torch.sqrt(dx * dx + dy * dy), W)


def _inputs2(case, seed):
    """(case dictionaries, phi0 tensors, u0 tensors or None), FP64 on the GPU."""
    rng = random.Random(1000003 * int(seed) + 17)
    kind = case["kind"]
    if kind == "batch":
        ps, phis, us = [], [], []
        sizes = random.Random(case["ncases"])  # the grids of a study are fixed, the droplets vary
        for _ in range(case["ncases"]):
            n = sizes.choice(EDGES)
            R = rng.uniform(0.05, 0.3) * n
            v, ang = rng.uniform(0.0, 0.02), rng.uniform(0.0, 2.0 * math.pi)
            ps.append(_params2(n, n, rho_l=math.exp(rng.uniform(0.0, math.log(10.0)))))
            phis.append(_disc(n, n, 0.5 * n + rng.uniform(0.1, 0.4), 0.5 * n + rng.uniform(0.1, 0.4),
                              R, 4.0))
            u = torch.empty((2, n, n), dtype=torch.float64, device="cuda")
            u[0], u[1] = v * math.cos(ang), v * math.sin(ang)
            us.append(u)
        return ps, phis, us
    if kind == "lattice":
        cx, cy = case["cell_x"], case["cell_y"]
        cell = _disc(cx, cy, 0.5 * cx + rng.uniform(0.1, 0.4), 0.5 * cy + rng.uniform(0.1, 0.4),
                     rng.uniform(20.0, 28.0), 4.0)
        return [_params2(cx * case["mx"], cy * case["my"])], [cell.repeat(case["my"], case["mx"])], None
    nx, ny = case["nx"], case["ny"]
    jx, jy = rng.uniform(0.1, 0.4), rng.uniform(0.1, 0.4)
    side = min(nx, ny)
    if kind == "droplets":  # a large and a small droplet
        W = 4.0
        phi = _disc(nx, ny, 0.31 * nx + jx, 0.5 * ny + jy, rng.uniform(0.17, 0.2) * side, W)
        phi = phi + _disc(nx, ny, 0.75 * nx + jx, 0.5 * ny + jy, rng.uniform(0.09, 0.11) * side, W)
        return [_params2(nx, ny)], [phi], None
    if kind == "film":
        h = rng.uniform(0.1, 0.2) * ny
        x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :] * (2.0 * math.pi / nx)
        y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None] + 0.5
        phi = _profile(h * (1.0 + 0.33 * torch.cos(x + jx)) - y, 4.0)
        return [_params2(nx, ny, tau_f_l=0.6, tau_f_g=0.6, walls=1)], [phi], None
    if kind == "vortex":
        p = _params2(nx, ny, flow="vortex", W=3.0, sigma=0.01, vortex_U=rng.uniform(0.015, 0.02),
                     vortex_T=64.0 * nx)
        return [p], [_disc(nx, ny, 0.5 * nx + jx, 0.75 * ny + jy, 0.15 * nx, 3.0)], None
    # a droplet in shear between moving walls (also the reverse mode's cavity), or translating
    # in a periodic box
    R = rng.uniform(0.13, 0.15) * side
    if kind == "cavity" or case["walls"]:
        U, Ca, Re = 0.01, 0.1, 0.1
        G = 2.0 * U / ny
        nu = min(G * R * R / Re, 1.1)  # larger viscosities are unstable in this model
        p = _params2(nx, ny, tau_f_l=3.0 * nu + 0.5, tau_f_g=3.0 * nu + 0.5,
                     sigma=nu * G * R / Ca, walls=1, u_top=U, u_bot=-U)
        u = torch.zeros((2, ny, nx), dtype=torch.float64, device="cuda")
        u[0] = (-U + 2.0 * U * (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny)[:, None]
    else:
        p = _params2(nx, ny, sigma=5e-3, tau_f_l=0.9, tau_f_g=0.9)
        u = torch.empty((2, ny, nx), dtype=torch.float64, device="cuda")
        u[0], u[1] = rng.uniform(0.005, 0.01), rng.uniform(-0.005, 0.005)
    if kind == "cavity":
        return [p], [_disc(nx, ny, 0.5 * nx + jx, 0.5 * ny - 0.5 + jy, R, 4.0)], [u]
    # reverse mode: a droplet already deformed (Taylor D of 0.1 to 0.15), as it is later in a run;
    # of a circle D is 0, where it has no derivative
    s, ang = rng.uniform(1.1, 1.15), rng.uniform(0.6, 0.9)
    dx, dy = _axis(nx, 0.5 * nx + jx)[None, :], _axis(ny, 0.5 * ny - 0.5 + jy, False)[:, None]
    a = (math.cos(ang) * dx + math.sin(ang) * dy) / s
    b = (math.cos(ang) * dy - math.sin(ang) * dx) * s
    return [p], [_profile(R - torch.sqrt(a * a + b * b), 4.0)], [u]


def _inputs3(case, seed):
    rng = random.Random(1000003 * int(seed) + 29)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    p = dict(nx=nx, ny=ny, nz=nz, W=4.0, sigma=1e-3, xi=1e-10, tau_g=0.8, rho_l=1.0, rho_g=1.0)
    p["lambda"] = 0.5
    jx, jy = rng.uniform(0.1, 0.4), rng.uniform(0.1, 0.4)
    if case["kind"] == "column":  # Eq. 45 as a thread along z, at rest
        p.update(tau_f_l=0.6, tau_f_g=0.6)
        h = 2.0 * math.pi / 256.0
        z = torch.arange(nz, dtype=torch.float64, device="cuda") * (2.0 * math.pi / nz)
        R = ((0.15 + 0.05 * torch.cos(z + rng.uniform(0.0, 6.0))) / h)[:, None, None]
        dx, dy = _axis(nx, 0.5 * nx + jx)[None, None, :], _axis(ny, 0.5 * ny + jy)[None, :, None]
        return p, _profile(R - torch.sqrt(dx * dx + dy * dy), 4.0), None
    p.update(rho_l=3.0, tau_f_l=1.0, tau_f_g=1.0)
    dx = _axis(nx, 0.5 * nx + jx)[None, None, :]
    dy = _axis(ny, 0.5 * ny + jy)[None, :, None]
    dz = _axis(nz, 0.5 * nz + 0.23)[:, None, None]
    R = rng.uniform(0.22, 0.3) * min(nx, ny, nz)
    phi = _profile(R - torch.sqrt(dx * dx + dy * dy + dz * dz), 4.0)
    u = torch.empty((3, nz, ny, nx), dtype=torch.float64, device="cuda")
    u[0], u[1], u[2] = rng.uniform(0.008, 0.012), rng.uniform(0.004, 0.008), rng.uniform(-0.01, -0.006)
    return p, phi, u


def _host(t):
    return None if t is None else t.cpu().numpy()


class _Run2:
    """A 2-D simulation and the buffers a program keeps beside it."""

    def __init__(self, case, seed):
        ps, phis, us = _inputs2(case, seed)
        self.case, prec = case, case["precision"]
        us = None if us is None else [_host(u) for u in us]
        self.sim = lbm.Sim(ps, [_host(p) for p in phis], us, precision=prec)
        h = self.sim.h
        self.sizes = [lbm.lbm_snapshot_bytes(h, c) for c in range(len(ps))]
        dtype = torch.float32 if prec == "f32" else torch.float64
        self.states = torch.empty(sum(self.sizes) // dtype.itemsize, dtype=dtype, device="cuda")
        self.volumes = None
        if case["kind"] == "batch":
            self.volumes = self.sim.track_volume_history(case["steps"], host=False)
        if case["kind"] == "droplets":  # left and right half of the box
            lab = np.zeros((case["ny"], case["nx"]), dtype=np.int8)
            lab[:, int(0.55 * case["nx"]):] = 1
            self.sim.set_regions(0, lab, 2)


class _Run3:
    def __init__(self, case, seed):
        p, phi, u = _inputs3(case, seed)
        self.case = case
        self.sim = lbm3.Sim3(p, _host(phi), _host(u), precision=case["precision"])
        if case["kind"] == "column":
            self.sim.autotune(1)
            shape = (case["nz"], case["ny"], case["nx"])
            self.host = torch.empty(shape, dtype=torch.float64, pin_memory=True)
            self.phi = torch.empty(shape, dtype=getattr(torch, "float" + case["precision"][1:]))


class _RunGrad:
    def __init__(self, case, seed):
        (p,), (phi,), (u,) = _inputs2(case, seed)
        dtype = torch.float32 if case["precision"] == "f32" else torch.float64
        theta = [p["sigma"], p["tau_g"], p["lambda"], p["tau_f_l"]]
        if case["walls"]:
            theta += [p["u_top"], p["u_bot"]]
        self.case, self.p, self.u0 = case, p, _host(u)
        self.phi0 = phi.to(dtype).requires_grad_(True)
        self.theta = torch.tensor(theta, dtype=dtype, requires_grad=True)


def prepare(case, seed):
    if case["kind"] == "gradient":
        return _RunGrad(case, seed)
    return (_Run3 if case["kind"] in ("column", "ball") else _Run2)(case, seed)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    case = state.case
    if case["kind"] == "gradient":
        phi = adjoint.coupled_run(state.phi0, state.theta, state.p, case["steps"], u0=state.u0,
                                  precision=case["precision"])
        D = adjoint.taylor_deformation(phi)
        dphi0, dtheta = torch.autograd.grad(D, (state.phi0, state.theta))
        dtype = state.phi0.dtype
        return dict(phi=phi.detach().to(dtype), D=D.detach().to(dtype), dphi0=dphi0, dtheta=dtheta)
    sim = state.sim
    sim.step(case["steps"])
    if case["kind"] == "column":  # phi after a run of steps, into the program's own buffer
        lbm.lib().lbm3_fields(sim.h, lbm._dp(state.host.numpy()), None, None)
        return dict(phi=state.phi.copy_(state.host))
    if case["kind"] == "ball":
        phi, u, p = sim.fields()
        t = _HOST[case["precision"]]
        return dict(phi=phi.astype(t), u=u.astype(t), p=p.astype(t))
    out = dict(states=state.states)
    ptr = state.states.data_ptr()
    for c, nbytes in enumerate(state.sizes):
        lbm.lbm_snapshot(sim.h, c, ptr)
        ptr += nbytes
    if state.volumes is not None:
        out["volumes"] = state.volumes
    if case["kind"] == "droplets":
        out["volumes"] = sim.volume()
    if case["kind"] == "film":  # experiments.film: phi after a run of steps
        out["phi"] = sim.fields(0)[0].astype(_HOST[case["precision"]])
    return out


# fields are FP64 on the host whatever the precision of the run: kept in the run's own
_HOST = {"f64": np.float64, "f32": np.float32, "f16": np.float16}


def work(case):
    """State read and written once per step (2-D: 18 populations, or 9 in the vortex, and phi*u;
    3-D: 19 + 7 populations and phi*u), and the outputs; the reverse mode reads every state and
    reads and writes an adjoint state per step.  Operations per node: counted from the equations."""
    n, e = case["steps"], {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
    if case["kind"] in ("column", "ball"):
        nodes = case["nx"] * case["ny"] * case["nz"]
        per = 2 * (26 * e + 3 * max(e, 4))
        out = nodes * 8 * (1 if case["kind"] == "column" else 5)
        return dict(bytes=float(n * nodes * per + out), flops=float(n * nodes * 420))
    if case["kind"] == "batch":
        nodes = case["ncases"] * sum(k * k for k in EDGES) / len(EDGES)
    elif case["kind"] == "lattice":
        nodes = case["mx"] * case["cell_x"] * case["my"] * case["cell_y"]
    else:
        nodes = case["nx"] * case["ny"]
    planes = 11 if case["kind"] == "vortex" else 20
    if case["kind"] == "gradient":
        return dict(bytes=float(n * nodes * e * planes * 5), flops=float(n * nodes * 900))
    return dict(bytes=float(n * nodes * 2 * planes * e + 2 * nodes * planes * e),
                flops=float(n * nodes * (150 if planes == 11 else 260)))


# ---------------------------------------------------------------------------
# The same in plain FP64 torch
# ---------------------------------------------------------------------------

_C2 = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
_OPP2 = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_W2 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
_RIDGE = 0.1  # |grad psi| below which the interface normal has no direction


def _relax2(rates):
    """M^-1 diag(rates) M with the moment matrix of Eq. 24."""
    rows = [[1.0] * 9, [-4.0] + [-1.0] * 4 + [2.0] * 4, [4.0] + [-2.0] * 4 + [1.0] * 4]
    cx, cy = [float(c[0]) for c in _C2], [float(c[1]) for c in _C2]
    rows += [cx, [-2.0 * v if 0 < i < 5 else v for i, v in enumerate(cx)],
             cy, [-2.0 * v if 0 < i < 5 else v for i, v in enumerate(cy)],
             [x * x - y * y for x, y in zip(cx, cy)], [x * y for x, y in zip(cx, cy)]]
    M = torch.tensor(rows, dtype=torch.float64, device="cuda")
    rates = torch.stack([torch.as_tensor(r, dtype=torch.float64, device="cuda") for r in rates])
    return torch.linalg.inv(M) @ (rates[:, None] * M)


def _shift(a, dx, dy, walls):
    """a(x + dx, y + dy): periodic, or with the wall rows mirrored beyond the walls."""
    if dx:
        a = torch.roll(a, -dx, -1)
    if not dy:
        return a
    if not walls:
        return torch.roll(a, -dy, -2)
    return torch.cat((a[..., 1:, :], a[..., -1:, :]) if dy > 0 else (a[..., :1, :], a[..., :-1, :]), -2)


def _grad2(a, walls):
    n = [_shift(a, c[0], c[1], walls) for c in _C2]
    gx = sum(3.0 * w * c[0] * v for w, c, v in zip(_W2, _C2, n) if c[0])
    gy = sum(3.0 * w * c[1] * v for w, c, v in zip(_W2, _C2, n) if c[1])
    lap = sum(6.0 * w * (v - a) for w, v in zip(_W2[1:], n[1:]))
    return gx, gy, lap


class _Exact2:
    """One grid, or a stack of equal grids [B][ny][nx], stepped in FP64."""

    def __init__(self, p, phi0, u0, theta=None, rho_l=None):
        self.p, self.walls, self.vortex = p, p.get("walls", 0), p["flow"] == "vortex"
        th = theta if theta is not None else (p["sigma"], p["tau_g"], p["lambda"], p["tau_f_l"],
                                              p.get("u_top", 0.0), p.get("u_bot", 0.0))
        sigma, tau_g, self.lam, tau_f = th[:4]
        self.top, self.bot = (th[4], th[5]) if self.walls else (0.0, 0.0)
        self.beta, self.kappa = 12.0 * sigma / p["W"], 1.5 * sigma * p["W"]
        self.rho_l = p["rho_l"] if rho_l is None else rho_l
        one, sg, sf = torch.tensor(1.0, dtype=torch.float64, device="cuda"), 1.0 / tau_g, 1.0 / tau_f
        self.Ag = _relax2([one, one, one, sg, one, sg, one, one, one])
        self.Af = _relax2([one] * 7 + [sf, sf])
        self.t = 0
        u = torch.zeros((2,) + phi0.shape, dtype=torch.float64, device="cuda") if u0 is None else u0
        if self.vortex:
            u = self._vortex(phi0, 0)
        gx, gy, lap = _grad2(phi0, self.walls)
        J = phi0 * u
        self.J = J
        self.g = self._geq(phi0, self._mu(phi0, lap), J)
        self.f = None if self.vortex else self._feq(0.0, self._rho(phi0), u)
        self.post = None  # post-collision populations of the last step

    def _rho(self, phi):
        return self.p["rho_g"] + phi * (self.rho_l - self.p["rho_g"])

    def _mu(self, phi, lap):
        return 4.0 * self.beta * phi * (phi - 1.0) * (phi - 0.5) - self.kappa * lap

    def _geq(self, phi, mu, J):
        L = mu + self.lam * phi
        rest = phi - (1.0 - _W2[0]) * L
        return torch.stack([rest] + [w * (L + 3.0 * (c[0] * J[0] + c[1] * J[1]))
                                     for w, c in zip(_W2[1:], _C2[1:])])

    @staticmethod
    def _feq(p, rho, u):
        u2 = u[0] * u[0] + u[1] * u[1]
        out = []
        for i, (w, c) in enumerate(zip(_W2, _C2)):
            cu = c[0] * u[0] + c[1] * u[1]
            s = w * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2)
            out.append((3.0 * p * (w - 1.0) if i == 0 else 3.0 * p * w) + rho * s)
        return torch.stack(out)

    def _vortex(self, phi, t):
        ny, nx = phi.shape[-2:]
        X = ((torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx * math.pi)[None, :]
        Y = ((torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny * math.pi)[:, None]
        a = self.p["vortex_U"] * math.cos(math.pi * t / self.p["vortex_T"])
        return torch.stack((-a * torch.sin(X) ** 2 * torch.sin(2 * Y) + 0.0 * phi,
                            a * torch.sin(Y) ** 2 * torch.sin(2 * X) + 0.0 * phi))

    def _stream(self, v):
        """Values delivered to each node: v_i(x - c_i), bounced back at walls."""
        out = []
        for i, c in enumerate(_C2):
            a = torch.roll(v[i], (c[1], c[0]), (-2, -1))
            if self.walls and c[1]:
                own = v[_OPP2[i]]
                a = (torch.cat((own[..., :1, :], a[..., 1:, :]), -2) if c[1] > 0 else
                     torch.cat((a[..., :-1, :], own[..., -1:, :]), -2))
            out.append(a)
        return torch.stack(out)

    def macro(self):
        """phi, u and what the collision needs, of the current time."""
        if self.post is not None:
            self.g = self._stream(self.post[1])
        phi = self.g.sum(0)
        rho = self._rho(phi)
        if self.post is not None and not self.vortex:
            f = self._stream(self.post[0])
            if self.walls:
                add = torch.zeros_like(f)
                for i, c in enumerate(_C2):
                    if c[0] and c[1]:
                        r, uw = (0, self.bot) if c[1] > 0 else (-1, self.top)
                        add[i, ..., r, :] = rho[..., r, :] * c[0] * uw / 6.0
                f = f + add
            self.f = f
        return phi, rho

    def step(self):
        p, walls = self.p, self.walls
        phi, rho = self.macro()
        gx, gy, lap = _grad2(phi, walls)
        mu = self._mu(phi, lap)
        inside = (phi > 0.0) & (phi < 1.0)
        pc = torch.where(inside, phi, (phi >= 1.0).double())
        a, b = pc + p["xi"], 1.0 - pc + p["xi"]
        qx, qy, _ = _grad2(0.25 * p["W"] * torch.log(a / b), walls)
        q2 = qx * qx + qy * qy
        far = q2 >= _RIDGE ** 2
        inv = torch.where(far, 1.0 / torch.sqrt(torch.where(far, q2, torch.ones_like(q2))),
                          torch.zeros_like(q2))
        sharp = self.lam / p["W"] * 4.0 * a * b / (a + b) ** 2 * inv
        F = torch.stack((mu * gx, mu * gy))
        if self.vortex:
            u, fs = self._vortex(phi, self.t), None
        else:
            f = self.f
            m = torch.stack((sum(c[0] * f[i] for i, c in enumerate(_C2) if c[0]),
                             sum(c[1] * f[i] for i, c in enumerate(_C2) if c[1])))
            u = (m + 0.5 * F) / rho
            R = (self.rho_l - p["rho_g"]) * torch.stack((gx, gy))
            pr = 0.6 * (f[1:].sum(0) + 0.5 * (u * R).sum(0) - 2.0 / 3.0 * rho * (u * u).sum(0))
            Fi = torch.stack([3.0 * w * (c[0] * F[0] + c[1] * F[1] + (c[0] * u[0] + c[1] * u[1]) *
                                         (c[0] * R[0] + c[1] * R[1])) for w, c in zip(_W2, _C2)])
            fs = (f - torch.tensordot(self.Af, f - self._feq(pr, rho, u), 1) + Fi -
                  0.5 * torch.tensordot(self.Af, Fi, 1))
        J = phi * u
        V = 3.0 * (J - self.J) + sharp * torch.stack((qx, qy))
        Gi = torch.stack([w * (c[0] * V[0] + c[1] * V[1]) for w, c in zip(_W2, _C2)])
        g = self.g
        gs = (g - torch.tensordot(self.Ag, g - self._geq(phi, mu, J), 1) + Gi -
              0.5 * torch.tensordot(self.Ag, Gi, 1))
        self.post, self.J = (fs, gs), J
        self.t += 1
        return phi

    def snapshot(self, f32):
        """Planes of lbm_snapshot: f*, g*, phi u (and the rest population's low part)."""
        fs, gs = self.post
        parts = [torch.zeros_like(gs) if fs is None else fs, gs, self.J]
        if f32:
            parts.append(torch.zeros_like(gs[:1]))
        return torch.cat(parts, 0)


def _taylor(phi):
    ny, nx = phi.shape
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    m = phi.sum()
    dx, dy = x - (phi * x).sum() / m, y - (phi * y).sum() / m
    a, b, c = ((phi * v).sum() / m for v in (dx * dx, dy * dy, dx * dy))
    r = torch.sqrt(0.25 * (a - b) ** 2 + c * c)
    L, B = torch.sqrt(0.5 * (a + b) + r), torch.sqrt(0.5 * (a + b) - r)
    return (L - B) / (L + B)


def _exact_gradient(case, seed):
    s = _RunGrad(case, seed)
    phi0 = s.phi0.detach().double().requires_grad_(True)
    theta = s.theta.detach().double().cuda().requires_grad_(True)
    e = _Exact2(s.p, phi0, torch.as_tensor(s.u0, device="cuda"), theta=tuple(theta))
    for _ in range(case["steps"]):
        e.step()
    phi, _ = e.macro()
    D = _taylor(phi)
    dphi0, dtheta = torch.autograd.grad(D, (phi0, theta))
    return dict(phi=phi.detach(), D=D.detach(), dphi0=dphi0, dtheta=dtheta.cpu())


def _exact_batch(case, seed):
    ps, phis, us = _inputs2(case, seed)
    f32, steps = case["precision"] == "f32", case["steps"]
    states, vols = [None] * len(ps), torch.empty((steps, len(ps)), dtype=torch.float64)
    for n in EDGES:
        ids = [k for k, p in enumerate(ps) if p["nx"] == n]
        for k0 in range(0, len(ids), max(1, (1 << 22) // (n * n))):
            some = ids[k0:k0 + max(1, (1 << 22) // (n * n))]
            rho_l = torch.tensor([ps[k]["rho_l"] for k in some], dtype=torch.float64,
                                 device="cuda")[:, None, None]
            e = _Exact2(ps[some[0]], torch.stack([phis[k] for k in some]),
                        torch.stack([us[k] for k in some], 1), rho_l=rho_l)
            for t in range(steps):
                vols[t, some] = e.step().sum((-2, -1)).cpu()
            snap = e.snapshot(f32)
            for q, k in enumerate(some):
                states[k] = snap[:, q].reshape(-1)
    return dict(states=torch.cat(states), volumes=vols)


_C3 = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0),
       (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
       (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1))
_W3 = (1 / 3,) + (1 / 18,) * 6 + (1 / 36,) * 12


def _roll3(a, c, sign=1):
    return torch.roll(a, (sign * c[2], sign * c[1], sign * c[0]), (0, 1, 2)) if any(c) else a


def _grad3(a):
    n = [_roll3(a, c, -1) for c in _C3]
    g = [sum(3.0 * w * c[k] * v for w, c, v in zip(_W3, _C3, n) if c[k]) for k in range(3)]
    return g, sum(6.0 * w * (v - a) for w, v in zip(_W3[1:], n[1:]))


def _exact3(case, seed):
    """The single-relaxation-time limit on D3Q19 and D3Q7, in FP64."""
    p, phi, u0 = _inputs3(case, seed)
    beta, kappa, lam, W, xi = 12.0 * p["sigma"] / p["W"], 1.5 * p["sigma"] * p["W"], p["lambda"], p["W"], p["xi"]
    drho, wf, wg = p["rho_l"] - p["rho_g"], 1.0 / p["tau_f_l"], 1.0 / p["tau_g"]
    u = [torch.zeros_like(phi) for _ in range(3)] if u0 is None else list(u0)
    dot = lambda c, v: sum(k * x for k, x in zip(c, v) if k)  # noqa: E731

    def mu_of(phi, lap):
        return 4.0 * beta * phi * (phi - 1.0) * (phi - 0.5) - kappa * lap

    def feq(i, pr, rho, u, u2):
        c, w = _C3[i], _W3[i]
        if i == 0:
            return 3.0 * pr * (w - 1.0) - 1.5 * w * rho * u2
        cu = dot(c, u)
        return w * (3.0 * pr + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * u2))

    def geq(i, phi, L, J):
        return phi - 0.75 * L if i == 0 else 0.125 * L + 0.5 * dot(_C3[i], J)

    def macro(f, g):
        phi = sum(g[1:], g[0])
        gp, lap = _grad3(phi)
        mu = mu_of(phi, lap)
        rho = p["rho_g"] + phi * drho
        F = [mu * v for v in gp]
        u = [(sum(c[k] * f[i] for i, c in enumerate(_C3) if c[k]) + 0.5 * F[k]) / rho for k in range(3)]
        R = [drho * v for v in gp]
        u2 = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        pr = 0.5 * (sum(f[2:], f[1]) + 0.5 * sum(a * b for a, b in zip(u, R)) - 0.5 * rho * u2)
        return phi, mu, rho, F, u, R, u2, pr

    _, lap = _grad3(phi)
    L0 = mu_of(phi, lap) + lam * phi
    Jp = [phi * v for v in u]
    rho0, u20 = p["rho_g"] + phi * drho, u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    f = [feq(i, 0.0, rho0, u, u20) for i in range(19)]
    g = [geq(i, phi, L0, Jp) for i in range(7)]
    for _ in range(case["steps"]):
        phi, mu, rho, F, u, R, u2, pr = macro(f, g)
        pc = phi.clamp(0.0, 1.0)
        a, b = pc + xi, 1.0 - pc + xi
        q, _ = _grad3(0.25 * W * torch.log(a / b))
        q2 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2]
        sharp = torch.where(q2 >= _RIDGE ** 2, lam / W * 4.0 * a * b / (a + b) ** 2 *
                            torch.rsqrt(q2.clamp_min(_RIDGE ** 2)), torch.zeros_like(q2))
        J = [phi * v for v in u]
        V = [(x - y) + 0.25 * sharp * n for x, y, n in zip(J, Jp, q)]
        L = mu + lam * phi
        for i in range(19):
            c, w = _C3[i], _W3[i]
            Fi = 3.0 * w * (dot(c, F) + dot(c, u) * dot(c, R)) if i else 0.0
            f[i] = _roll3(f[i] + wf * (feq(i, pr, rho, u, u2) - f[i]) + (1.0 - 0.5 * wf) * Fi, c)
        for i in range(7):
            Gi = 0.5 * dot(_C3[i], V) if i else 0.0
            g[i] = _roll3(g[i] + wg * (geq(i, phi, L, J) - g[i]) + (1.0 - 0.5 * wg) * Gi, _C3[i])
        Jp = J
    phi, _, _, _, u, _, _, pr = macro(f, g)
    if case["kind"] == "column":
        return dict(phi=phi.cpu().numpy())
    return dict(phi=phi.cpu().numpy(), u=torch.stack(u).cpu().numpy(), p=pr.cpu().numpy())


def exact(case, seed):
    if case["kind"] == "gradient":
        return _exact_gradient(case, seed)
    if case["kind"] in ("column", "ball"):
        return _exact3(case, seed)
    if case["kind"] == "batch":
        return _exact_batch(case, seed)
    (p,), (phi0,), us = _inputs2(case, seed)
    if case["kind"] == "lattice":  # every cell of the periodic lattice is the same
        cx, cy = case["cell_x"], case["cell_y"]
        e = _Exact2(p, phi0[:cy, :cx].contiguous(), None)
        for _ in range(case["steps"]):
            e.step()
        return dict(states=e.snapshot(True).repeat(1, case["my"], case["mx"]).reshape(-1))
    e = _Exact2(p, phi0, None if us is None else us[0])
    for _ in range(case["steps"]):
        e.step()
    out = dict(states=e.snapshot(case["precision"] == "f32").reshape(-1))
    if case["kind"] == "droplets":
        phi, _ = e.macro()
        k = int(0.55 * case["nx"])
        out["volumes"] = np.array([float(phi[:, :k].sum()), float(phi[:, k:].sum())])
    if case["kind"] == "film":
        out["phi"] = e.macro()[0].cpu().numpy()
    return out
