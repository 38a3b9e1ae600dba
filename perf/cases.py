"""Performance cases: what users of this package have it do, called as their programs call it.

A pass advances a lattice (or many, or a lattice and its adjoint) through the public entry points and reads
back what such a program reads: the macroscopic fields, the wall-load report or the gradients. Sizes come from
the package's workloads (the 128 x 128 droplet, the 2048 x 256 and 16384 x 2048 airway channels, the 64-channel
sweep, the 512 x 128 adjoint channel, the 1500 x 202 trend lattice) or are generic.

`exact` restates the method in plain float64 torch: the D2Q9 step with the equation-of-state force, walls,
pressure columns and masks, differentiated by autograd for the adjoint cases.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2103_08301_gb300 as lbm
from paper_2103_08301_gb300.adjoint import Adjoint, WallLoads

# The method's own coexistence at 0.85 Tc (tau = 1, kappa = 0.5): vapour and liquid density, saturation pressure.
RHO_G, RHO_L, P_STAR = 0.02185, 0.2759, 1.4362e-3
DEVICE = "cuda"


def _case(name, form, nx, ny, steps, **more):
    c = {"form": form, "nx": nx, "ny": ny, "steps": steps, "walls": True, "precision": 32, "eos": "cs",
         "collision": "bgk", "dp": 0.0, "gx": 0.0, "readout": "device", "report": False}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the static droplet of the verification section: a small periodic box in double precision
        _case("droplet 128x128 fp64", "lattice", 128, 128, 64, walls=False, precision=64),
        # a monitored run: one step, its wall-load report and the fields after each (the smallest call)
        _case("monitored 512x128 fp32", "lattice", 512, 128, 1, dp=1e-4, report=True),
        # the airway-reopening channel: many steps between two read-backs
        _case("airway 2048x256 fp32", "lattice", 2048, 256, 128, dp=1e-3),
        # the trend study: body force, ends at one pressure, fields to host arrays every 250 steps
        _case("trend 1500x202 fp32", "lattice", 1500, 202, 250, gx=5e-8, readout="host", report=True),
        # the largest channel of the workloads
        _case("airway 16384x2048 fp32", "lattice", 16384, 2048, 16, dp=1e-3),
        # the variants on a periodic box of odd sizes: Peng-Robinson water, multiple relaxation times; the whole
        # state (populations) is read back for a restart on the device, besides the fields
        _case("pr mrt box 1999x1501 fp32", "lattice", 1999, 1501, 16, walls=False, eos="pr", collision="mrt",
              readout="state"),
        # the double-precision build on a channel of ordinary size
        _case("airway 4096x512 fp64", "lattice", 4096, 512, 8, precision=64, dp=2e-4),
        # general wall geometry: constrictions on both walls
        _case("masked 4096x1024 fp32", "masked", 4096, 1024, 16, dp=2e-4),
        # one population array: grids that would not fit otherwise
        _case("in-place 16384x2048 fp32", "inplace", 16384, 2048, 16, dp=1e-3),
        # the parameter sweep: channels of uneven size stepped together, every channel read back at the end
        _case("sweep of 64 channels fp32", "sweep", 4096, 512, 64, channels=64, dp=1e-3),
        # gradients of the wall loads, single-precision forward and double-precision reverse sweep
        _case("adjoint 512x128 fp32 fp64", "adjoint", 512, 128, 200, reverse=64, dp=1e-3),
        # gradients for an optimiser that keeps single-precision parameters, through autograd
        _case("adjoint 1024x256 fp32 fp32", "adjoint", 1024, 256, 100, reverse=32, dp=1e-3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _gentle(nx, ny):
    """A pressure drop whose vapour core stays slow in a channel run for long."""
    return min(1e-3, 6e-4 * nx / (ny * ny))


def draw(rng):
    form = rng.choice(["lattice", "lattice", "lattice", "lattice", "masked", "inplace", "sweep", "adjoint", "adjoint"])
    if form == "sweep":
        return _case("", form, 2048, 512, _log(rng, 16, 64), channels=rng.randint(4, 48), dp=1e-3)
    if form == "adjoint":
        nx, ny = _log(rng, 96, 1024), _log(rng, 32, 256)
        precision, reverse = rng.choice([(32, 64), (32, 32), (64, 64)])
        steps = max(8, min(200, int(1.3e7 / (nx * ny))))
        return _case("", form, nx, ny, rng.randint(8, steps), precision=precision, reverse=reverse, dp=_gentle(nx, ny))
    if form == "masked":
        nx, ny, precision = _log(rng, 256, 4096), _log(rng, 96, 1024), rng.choice([32, 32, 64])
    elif form == "inplace":
        nx, ny, precision = _log(rng, 256, 16384), _log(rng, 64, 2048), rng.choice([32, 32, 64])
    else:
        nx, ny, precision = _log(rng, 96, 16384), _log(rng, 48, 2048), rng.choice([32, 32, 32, 64])
    most = int((3e8 if precision == 32 else 1.5e7) / (nx * ny))
    if most < 4:  # double precision: the ordinary sizes
        nx, ny = nx % 4096 + 96, ny % 512 + 48
        most = int(1.5e7 / (nx * ny))
    steps = rng.randint(1, max(1, min(250, most)))
    report = rng.random() < 0.3
    readout = "host" if nx * ny < 500000 and rng.random() < 0.3 else "device"
    if form == "lattice" and rng.random() < 0.4:
        eos = rng.choice(["cs", "cs", "pr"])
        collision = "mrt" if eos == "pr" and rng.random() < 0.5 else "bgk"
        return _case("", form, nx, ny, steps, walls=False, precision=precision, eos=eos, collision=collision,
                     readout="state" if rng.random() < 0.3 else readout)
    if form == "lattice" and rng.random() < 0.25:
        return _case("", form, nx, ny, steps, precision=precision, gx=min(5e-8, _gentle(nx, ny) / nx), readout=readout,
                     report=report)
    return _case("", form, nx, ny, steps, precision=precision, dp=_gentle(nx, ny), readout=readout, report=report)


# ---- inputs ----------------------------------------------------------------

def _model(case):
    """Keyword arguments of the package's classes: equation of state, relaxation, collision."""
    if case["eos"] == "pr":
        kw = dict(eos="pr", a=2 / 49, b=2 / 21, T_over_Tc=0.8, k=1.0, kappa=0.01, tau=1.2)
        if case["collision"] == "mrt":
            kw.update(collision="mrt", s_e=1.64, s_eps=1.54, s_q=1 / 1.2, s_j=1 / 1.2)
        return kw
    return dict(T_over_Tc=0.85 if case["walls"] else 0.8, k=1.0, kappa=0.5, tau=1.0)


def _densities(case):
    """(vapour, liquid) of the initial profile."""
    if case["walls"]:
        return RHO_G, RHO_L
    return (0.19708, 7.20405) if case["eos"] == "pr" else (0.021723, 0.307196)  # the equations of state at 0.8 Tc


def _noise(shape, seed, amp):
    g = torch.Generator(device=DEVICE).manual_seed(int(seed) * 7919 + 17)
    return amp * (2.0 * torch.rand(shape, generator=g, dtype=torch.float64, device=DEVICE) - 1.0)


def _channel_rho0(nx, ny, film, plug_x, plug_len, seed):
    y = torch.arange(ny, dtype=torch.float64, device=DEVICE)[:, None]
    x = torch.arange(nx, dtype=torch.float64, device=DEVICE)[None, :]
    wall = torch.minimum(y - 0.5, (ny - 1.5) - y)
    s_film = 0.5 * (1.0 - torch.tanh(0.5 * (wall - film)))
    s_plug = 0.5 * (torch.tanh(0.5 * (x - plug_x)) - torch.tanh(0.5 * (x - plug_x - plug_len)))
    rho = RHO_G + (RHO_L - RHO_G) * torch.maximum(s_film, s_plug)
    return rho * (1.0 + _noise((ny, nx), seed, 1e-3))


def _rho0(case, seed):
    """Initial density (float64, on the GPU): films and a plug, or a disk, with seeded noise of 0.1%."""
    nx, ny = case["nx"], case["ny"]
    if case["walls"]:
        return _channel_rho0(nx, ny, max(3, ny // 32), nx // 4, max(6, nx // 16), seed)
    g, l = _densities(case)
    y = torch.arange(ny, dtype=torch.float64, device=DEVICE)[:, None]
    x = torch.arange(nx, dtype=torch.float64, device=DEVICE)[None, :]
    r = torch.sqrt((x - nx / 2) ** 2 + (y - ny / 2) ** 2)
    s = 0.5 * (1.0 - torch.tanh(0.5 * (r - 0.23 * min(nx, ny))))
    return (g + (l - g) * s) * (1.0 + _noise((ny, nx), seed, 1e-3))


def _p_ref(case):
    return P_STAR - 0.5 * case["dp"] if case["walls"] else None


def _mask(case):
    """Constrictions on both walls: blocks a quarter of the height tall, one per 512 columns or so."""
    nx, ny = case["nx"], case["ny"]
    m = np.zeros((ny, nx), np.uint8)
    for x0 in range(nx // 8, nx - 64, max(128, min(512, nx // 3))):
        m[1:ny // 4, x0:x0 + 32] = 1
        m[ny - ny // 4:ny - 1, x0:x0 + 32] = 1
    return m


def _sweep_specs(case):
    """Sizes, pressure drops, plugs and films of the sweep's channels."""
    rng = np.random.RandomState(3)
    out = []
    for _ in range(case["channels"]):
        u = rng.random_sample(5)
        nx, ny = 1024 + int(u[0] * 3073), 128 + int(u[1] * 385)
        out.append(dict(nx=nx, ny=ny, dp=(0.25 + 0.75 * u[2]) * case["dp"], plug=64 + int(u[3] * 193),
                        film=4 + int(u[4] * 21)))
    return out


REPORT = ("mass", "wall_shear_sum", "tau_wall_min", "tau_wall_max", "p_wall_min", "p_wall_max")


class _Lattice:
    def __init__(self, case, seed):
        self.case = case
        self.steps = case["steps"]
        rho0 = _rho0(case, seed).cpu().numpy()
        self.stream = torch.cuda.Stream()
        self.lat = lbm.Lattice(case["nx"], case["ny"], rho0, walls=case["walls"], bc_x=case["walls"],
                               precision=case["precision"], dp=case["dp"], p_ref=_p_ref(case), gx=case["gx"],
                               stream=self.stream, mask=_mask(case) if case["form"] == "masked" else None,
                               inplace=case["form"] == "inplace", **_model(case))
        self.out = None
        if case["readout"] != "host":
            dt = torch.float32 if case["precision"] == 32 else torch.float64
            z = lambda *s: torch.zeros(s, dtype=dt, device=DEVICE)  # noqa: E731
            ny, nx = case["ny"], case["nx"]
            self.out = dict(rho=z(ny, nx), vx=z(ny, nx), vy=z(ny, nx), tau_wall=z(2, nx), p_wall=z(2, nx))
            self.f = z(9, ny, nx) if case["readout"] == "state" else None

    def run(self):
        self.lat.step(self.steps)
        if self.out is None:
            fields = self.lat.fields()
        else:
            self.lat.fields_into(**self.out)
            fields = self.out
        if self.case["readout"] == "state":
            # the C entry point, for a device destination (Lattice.populations returns a host array)
            st = lbm.lib().lbm_populations(self.lat.ctx, self.f.data_ptr())
            assert st == lbm.LBM_OK
            return {"fields": fields, "populations": self.f}
        if not self.case["report"]:
            return fields
        d = self.lat.diag()
        return {"fields": fields, "report": {k: d[k] for k in REPORT}}


class _Sweep:
    def __init__(self, case, seed):
        self.steps = case["steps"]
        specs = _sweep_specs(case)
        chans = [dict(nx=s["nx"], ny=s["ny"], dp=s["dp"], p_ref=P_STAR - 0.5 * s["dp"],
                      rho0=_channel_rho0(s["nx"], s["ny"], s["film"], s["nx"] // 4, s["plug"],
                                         seed * 101 + k).cpu().numpy()) for k, s in enumerate(specs)]
        self.batch = lbm.Batch(chans, walls=True, bc_x=True, precision=case["precision"], T_over_Tc=0.85, k=1.0,
                               kappa=0.5, tau=1.0)
        dt = torch.float32 if case["precision"] == 32 else torch.float64
        self.out = [torch.zeros((3, s["ny"], s["nx"]), dtype=dt, device=DEVICE) for s in specs]

    def run(self):
        self.batch.step(self.steps)
        # the C entry point, for device destinations (Batch.fields returns host arrays)
        for c, o in enumerate(self.out):
            st = lbm.lib().lbm_batch_fields(self.batch.h, c, o[0].data_ptr(), o[1].data_ptr(), o[2].data_ptr(), None,
                                            None)
            assert st == lbm.LBM_OK
        return self.out


class _Adjoint:
    """The gradient of J_tau + 0.3 J_p with respect to the initial density and the drive."""

    def __init__(self, case, seed):
        self.case = case
        rho0 = _rho0(case, seed)
        self.adj = Adjoint(case["nx"], case["ny"], case["steps"], T_over_Tc=0.85, k=1.0, kappa=0.5, tau=1.0,
                           p_ref=_p_ref(case), precision=case["precision"], reverse_precision=case["reverse"])
        if case["reverse"] == 32:
            self.rho0 = rho0.to(torch.float32).requires_grad_(True)
            self.dp = torch.tensor(case["dp"], dtype=torch.float64, requires_grad=True)
        else:
            self.rho0 = rho0

    def run(self):
        if self.case["reverse"] == 32:
            self.rho0.grad = self.dp.grad = None
            j_tau, j_p = WallLoads.apply(self.adj, self.rho0, self.dp)
            (j_tau + 0.3 * j_p).backward()
            return {"J": [float(j_tau), float(j_p)], "rho0": self.rho0.grad, "dp": float(self.dp.grad)}
        j_tau, j_p = self.adj.forward(self.rho0, dp=self.case["dp"])
        g, drive = self.adj.backward(1.0, 0.3)
        return {"J": [j_tau, j_p], "rho0": g, "dp": drive["dp"]}


def prepare(case, seed):
    return {"sweep": _Sweep, "adjoint": _Adjoint}.get(case["form"], _Lattice)(case, seed)


def run(state):
    return state.run()


def work(case):
    """Populations read and written once per step (9 values each way); the read-back reads them once more and
    writes its fields; a reverse step recomputes a state and reads it, and reads and writes the adjoint."""
    v = case["precision"] // 8
    n = case["nx"] * case["ny"]
    if case["form"] == "sweep":
        n = sum(s["nx"] * s["ny"] for s in _sweep_specs(case))
    if case["form"] == "adjoint":
        r = case["reverse"] // 8
        per = 18 * v + 18 * v + 9 * v + 18 * r
        return {"bytes": per * n * case["steps"] + 24 * n, "flops": 1000 * n * case["steps"]}
    back = 12 + (9 if case["readout"] == "state" else 0)
    return {"bytes": 18 * v * n * case["steps"] + back * v * n, "flops": 200 * n * case["steps"]}


# ---- the method in 64 bits ---------------------------------------------------

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
# Lallemand-Luo moments: rho, e, eps, j_x, q_x, j_y, q_y, p_xx, p_xy
MOMENTS = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
                    [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
                    [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
                    [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=np.float64)


def _extremum(f, lo, hi):
    """Maximum of a unimodal f on [lo, hi]."""
    for _ in range(300):
        a, b = lo + (hi - lo) / 3, hi - (hi - lo) / 3
        lo, hi = (a, hi) if f(a) < f(b) else (lo, b)
    return f(0.5 * (lo + hi))


def _cs(eta):  # compressibility factor of Carnahan-Starling and d(eta Z)/d eta
    z = (1 + eta + eta ** 2 - eta ** 3) / (1 - eta) ** 3
    h = (1 + 4 * eta + 4 * eta ** 2 - 4 * eta ** 3 + eta ** 4) / (1 - eta) ** 4
    return z, h


class _CS:
    """Carnahan-Starling, a = 1, b = 4, R = 1 (eta = rho)."""

    def __init__(self, T_over_Tc):
        self.T = T_over_Tc * _extremum(lambda e: 2 * e / _cs(e)[1], 1e-3, 0.6)

    def p(self, r):
        return r * self.T * _cs(r)[0] - r * r

    def dp(self, r):
        return self.T * _cs(r)[1] - 2 * r

    def mu(self, r):
        return self.T * (math.log(r) - 1 + r * (4 - 3 * r) / (1 - r) ** 2) - r + self.p(r) / r

    def root(self, p, r):
        for _ in range(100):
            r -= (self.p(r) - p) / self.dp(r)
        return r

    @functools.lru_cache(None)
    def maxwell(self):
        g, l = 0.03, 0.26
        for _ in range(100):  # Newton on equal pressure and chemical potential (d mu = d p / rho)
            f1, f2 = self.p(g) - self.p(l), self.mu(g) - self.mu(l)
            a, b, c, d = self.dp(g), -self.dp(l), self.dp(g) / g, -self.dp(l) / l
            det = a * d - b * c
            g, l = g - (f1 * d - b * f2) / det, l - (a * f2 - c * f1) / det
        return g, l


@functools.lru_cache(None)
def _pr_T(b, a, omega, tr):
    """(R T, a alpha(T)) of Peng-Robinson with R = 1; Tc where dp/drho first vanishes at its inflection."""
    def spinodal_T(x):
        return 2 * x * (1 + x) * (1 - x) ** 2 / (1 + 2 * x - x * x) ** 2
    tc = a / b * _extremum(spinodal_T, 1e-3, 0.6)
    m = 0.37464 + 1.54226 * omega - 0.26992 * omega ** 2
    return tr * tc, a * (1 + m * (1 - math.sqrt(tr))) ** 2


class _Exact:
    """The method on one lattice in float64 torch."""

    def __init__(self, nx, ny, walls, dp, gx, model, mask=None):
        self.nx, self.ny, self.walls, self.gx = nx, ny, walls, gx
        self.kappa, self.tau = model["kappa"], model["tau"]
        self.pr = model.get("eos") == "pr"
        if self.pr:
            self.b = model["b"]
            self.RT, self.aalpha = _pr_T(model["b"], model["a"], 0.344, model["T_over_Tc"])
        else:
            self.cs = _CS(model["T_over_Tc"])
        self.relax = None
        self.shift = self.tau
        if model.get("collision") == "mrt":
            s = np.array([0, model["s_e"], model["s_eps"], model["s_j"], model["s_q"], model["s_j"], model["s_q"],
                          1 / self.tau, 1 / self.tau])
            k = np.linalg.inv(MOMENTS) @ np.diag(s) @ MOMENTS
            self.relax, self.shift = torch.tensor(k, device=DEVICE), 1 / model["s_j"]
        if walls:
            g, l = self.cs.maxwell()
            self.ph_g, self.dph = g, l - g
            p_ref = P_STAR - 0.5 * dp
            self.cols = torch.tensor([self.cs.root(p, r) for p in (p_ref + dp / 2, p_ref - dp / 2) for r in (g, l)],
                                     dtype=torch.float64, device=DEVICE)
            self.rates = [s * 0.5 / self.cs.dp(float(r)) for s, r in zip((1, 1, -1, -1), self.cols)]
        solid = np.zeros((ny, nx), bool)
        if walls:
            solid[0] = solid[-1] = True
        if mask is not None:
            solid |= mask != 0
        y, x = np.arange(-2, ny + 2), np.arange(-2, nx + 2)
        self.xmap = torch.tensor(np.clip(x, 0, nx - 1) if walls else x % nx, device=DEVICE)
        ym = np.where(y <= 0, 1 - y, np.where(y >= ny - 1, 2 * ny - 3 - y, y)) if walls else y % ny
        self.ymap = torch.tensor(ym, device=DEVICE)
        self.ghost = _ghosts(solid, walls) if mask is not None else None
        self.solid = torch.tensor(solid, device=DEVICE) if walls else None
        self.bounce = [None] * 9
        if walls:
            self.bounce = [torch.roll(self.solid, (EY[i], EX[i]), (0, 1)) if i else None for i in range(9)]
            open_ = ~solid
            o = np.stack([open_[1] & open_[2], open_[-2] & open_[-3]])
            o[:, 0] = o[:, -1] = False
            self.open = torch.tensor(o, device=DEVICE)

    def k2p0(self, r):
        if self.pr:
            x = self.b * r
            return r * self.RT / (1 - x) - self.aalpha * r * r / (1 + x * (2 - x))
        om = 1 - r
        return self.cs.T * r * (1 + r * (1 + r * om)) / (om * om * om) - r * r

    def start(self, rho0):
        return torch.stack([w * rho0 for w in WT])

    def density(self, f):
        """(rho with column densities, rho on the lattice extended by two nodes)"""
        rho = f.sum(0)
        if self.walls:
            def col(r, g, l):
                return g + torch.clamp((r - self.ph_g) / self.dph, 0, 1) * (l - g)
            rho = torch.cat([col(rho[:, 1:2], self.cols[0], self.cols[1]), rho[:, 1:-1],
                             col(rho[:, -2:-1], self.cols[2], self.cols[3])], 1)
        if self.ghost is None:
            return rho, rho[self.ymap][:, self.xmap]
        dst, src, w = self.ghost
        E = rho[self.ymap.clamp(0, self.ny - 1)][:, self.xmap].reshape(-1)
        E = E.index_copy(0, dst, (rho.reshape(-1)[src] * w).sum(1))
        return rho, E.reshape(self.ny + 4, self.nx + 4)

    @staticmethod
    def grad(A):
        a, b, c = A[:-2], A[1:-1], A[2:]
        gx = (4 * (b[:, 2:] - b[:, :-2]) + (c[:, 2:] - c[:, :-2]) + (a[:, 2:] - a[:, :-2])) / 12
        gy = (4 * (c[:, 1:-1] - a[:, 1:-1]) + (c[:, 2:] - a[:, 2:]) + (c[:, :-2] - a[:, :-2])) / 12
        return gx, gy

    @staticmethod
    def lap(A):
        a, b, c = A[:-2], A[1:-1], A[2:]
        return (4 * (b[:, 2:] + b[:, :-2] + a[:, 1:-1] + c[:, 1:-1]) + a[:, 2:] + a[:, :-2] + c[:, 2:] + c[:, :-2]
                - 20 * b[:, 1:-1]) / 6

    def forces(self, f):
        rho, E = self.density(f)
        L = self.lap(E)
        phx, phy = self.grad((self.k2p0(E) - E / 3)[1:-1, 1:-1])
        lx, ly = self.grad(L)
        Fx = -phx + self.kappa * rho * lx + self.gx
        Fy = -phy + self.kappa * rho * ly
        jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
        jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        return rho, E, L, Fx, Fy, jx, jy

    def loads(self, rho, E, L, Fx, jx):
        """Wall shear and wall pressure, 2 x nx (bottom, top)."""
        v = lambda y: (jx[y] + 0.5 * Fx[y]) / rho[y]  # noqa: E731
        nu = (self.tau - 0.5) / 3
        ny = self.ny
        tw = torch.stack([rho[a] * nu * (9 * v(a) - v(b)) / 3 for a, b in ((1, 2), (ny - 2, ny - 3))])
        pw = []
        for y in (1, ny - 2):
            gx, gy = self.grad(E[y + 1:y + 4, 1:-1])
            pw.append((self.k2p0(rho[y]) - self.kappa * rho[y] * L[y + 1, 1:-1]
                       - 0.5 * self.kappa * (gx * gx + gy * gy))[0])
        zero = torch.zeros((), dtype=torch.float64, device=DEVICE)
        return torch.where(self.open, tw, zero), torch.where(self.open, torch.stack(pw), zero)

    @staticmethod
    def feq(rho, ux, uy):
        usq = 1.5 * (ux * ux + uy * uy)
        out = []
        for i in range(9):
            eu = EX[i] * ux + EY[i] * uy
            out.append(WT[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - usq))
        return torch.stack(out)

    def step(self, f, s=None):
        rho, E, L, Fx, Fy, jx, jy = s or self.forces(f)
        fe = self.feq(rho, (jx + self.shift * Fx) / rho, (jy + self.shift * Fy) / rho)
        if self.relax is None:
            fs = f + (fe - f) / self.tau
        else:
            fs = f - torch.tensordot(self.relax, f - fe, 1)
        if self.walls:
            ends = []
            for b, n in ((0, 1), (-1, -2)):
                vx, vy = (jx[:, n] + 0.5 * Fx[:, n]) / rho[:, n], (jy[:, n] + 0.5 * Fy[:, n]) / rho[:, n]
                neq = f[:, :, n] - self.feq(rho[:, n], vx, vy)
                ends.append((self.feq(rho[:, b], vx, vy) + (1 - 1 / self.tau) * neq)[:, :, None])
            fs = torch.cat([ends[0], fs[:, :, 1:-1], ends[1]], 2)
        new = []
        for i in range(9):
            g = torch.roll(fs[i], (EY[i], EX[i]), (0, 1))
            new.append(g if self.bounce[i] is None else torch.where(self.bounce[i], fs[OPP[i]], g))
        new = torch.stack(new)
        return new if self.solid is None else torch.where(self.solid, f, new)

    def fields(self, f):
        rho, E, L, Fx, Fy, jx, jy = self.forces(f)
        vx, vy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        out = {}
        zero = torch.zeros((), dtype=torch.float64, device=DEVICE)
        if self.walls:
            out["tau_wall"], out["p_wall"] = self.loads(rho, E, L, Fx, jx)
            vx, vy = (torch.cat([v[:, 1:2], v[:, 1:-1], v[:, -2:-1]], 1) for v in (vx, vy))
            rho, vx, vy = (torch.where(self.solid, zero, v) for v in (rho, vx, vy))
        else:
            out["tau_wall"] = out["p_wall"] = torch.zeros((2, self.nx), dtype=torch.float64, device=DEVICE)
        out.update(rho=rho, vx=vx, vy=vy)
        return out


def _ghosts(solid, clamp):
    """Ghost densities of solid points on the lattice extended by two nodes: (points, their sources, weights).
    Sources of a point: along the axis directions of least depth d <= 2 to fluid, the node 2d - 1 out (or d out
    where that is solid); else the diagonals likewise; else the fluid nodes at knight offsets; their mean."""
    ny, nx = solid.shape

    def at(x, y):
        xm = np.clip(x, 0, nx - 1) if clamp else x % nx
        ym = y if clamp else y % ny
        inside = (ym >= 0) & (ym < ny)
        return xm, np.clip(ym, 0, ny - 1), inside

    def fluid(x, y):
        xm, ym, inside = at(x, y)
        return inside & ~solid[ym, xm]

    Y, X = np.meshgrid(np.arange(-2, ny + 2), np.arange(-2, nx + 2), indexing="ij")
    todo = ~fluid(X, Y)
    X, Y = X[todo], Y[todo]
    src = np.zeros((X.size, 8), np.int64)
    has = np.zeros((X.size, 8), bool)

    def take(slot, sel, x, y):
        xm, ym, _ = at(x, y)
        src[sel, slot] = (ym * nx + xm)[sel]
        has[sel, slot] = True

    for dirs in (((1, 0), (-1, 0), (0, 1), (0, -1)), ((1, 1), (-1, 1), (-1, -1), (1, -1))):
        for d in (1, 2):
            free = ~has.any(1)
            for k, (dx, dy) in enumerate(dirs):
                sel = free & fluid(X + d * dx, Y + d * dy)
                if d == 2:
                    sel &= ~fluid(X + dx, Y + dy)
                far = fluid(X + (2 * d - 1) * dx, Y + (2 * d - 1) * dy)
                m = np.where(far, 2 * d - 1, d)
                take(k, sel, X + m * dx, Y + m * dy)
    free = ~has.any(1)
    for k, (dx, dy) in enumerate(((1, 2), (2, 1), (-1, 2), (-2, 1), (-1, -2), (-2, -1), (1, -2), (2, -1))):
        take(k, free & fluid(X + dx, Y + dy), X + dx, Y + dy)
    w = has / np.maximum(1, has.sum(1, keepdims=True))
    # a point with no source keeps density zero; none of its neighbours is fluid
    return tuple(torch.tensor(a, device=DEVICE) for a in ((Y + 2) * (nx + 4) + (X + 2), src, w))


def _exact_lattice(case, seed):
    E = _Exact(case["nx"], case["ny"], case["walls"], case["dp"], case["gx"], _model(case),
               _mask(case) if case["form"] == "masked" else None)
    f = E.start(_rho0(case, seed))
    total = dict(wall_shear_sum=0.0, tau_wall_min=[], tau_wall_max=[], p_wall_min=[], p_wall_max=[])
    for _ in range(case["steps"]):
        s = None
        if case["report"]:
            s = E.forces(f)
            tw, pw = E.loads(s[0], s[1], s[2], s[3], s[5])
            total["wall_shear_sum"] += tw.sum()
            for k, v in (("tau", tw), ("p", pw)):
                total[k + "_wall_min"].append(v[E.open].min())
                total[k + "_wall_max"].append(v[E.open].max())
            mass = torch.where(E.solid, torch.zeros_like(s[0]), s[0]).sum()
        f = E.step(f, s)
    fields = E.fields(f)
    if case["readout"] == "state":
        return {"fields": fields, "populations": f}
    if not case["report"]:
        return fields
    rep = {"mass": float(mass), "wall_shear_sum": float(total["wall_shear_sum"])}
    for k in ("tau_wall", "p_wall"):
        rep[k + "_min"] = float(torch.stack(total[k + "_min"]).min())
        rep[k + "_max"] = float(torch.stack(total[k + "_max"]).max())
    return {"fields": fields, "report": rep}


def _exact_sweep(case, seed):
    out = []
    for k, s in enumerate(_sweep_specs(case)):
        E = _Exact(s["nx"], s["ny"], True, s["dp"], 0.0, _model(case))
        f = E.start(_channel_rho0(s["nx"], s["ny"], s["film"], s["nx"] // 4, s["plug"], seed * 101 + k))
        for _ in range(case["steps"]):
            f = E.step(f)
        fields = E.fields(f)
        out.append(torch.stack([fields["rho"], fields["vx"], fields["vy"]]))
    return out


def _exact_adjoint(case, seed):
    E = _Exact(case["nx"], case["ny"], True, case["dp"], 0.0, _model(case))
    rho0 = _rho0(case, seed)
    if case["reverse"] == 32:
        rho0 = rho0.to(torch.float32).to(torch.float64)
    states = [E.start(rho0)]
    J = torch.zeros(2, dtype=torch.float64, device=DEVICE)
    with torch.no_grad():
        for n in range(case["steps"]):
            s = E.forces(states[-1])
            tw, pw = E.loads(s[0], s[1], s[2], s[3], s[5])
            J += torch.stack([tw.sum(), pw.sum()])
            if n + 1 < case["steps"]:
                states.append(E.step(states[-1], s))
    E.cols.requires_grad_(True)
    lam = torch.zeros_like(states[0])
    gcol = torch.zeros_like(E.cols)
    for f in reversed(states):
        f = f.requires_grad_(True)
        s = E.forces(f)
        tw, pw = E.loads(s[0], s[1], s[2], s[3], s[5])
        total = tw.sum() + 0.3 * pw.sum() + (E.step(f, s) * lam).sum()
        lam, gc = torch.autograd.grad(total, (f, E.cols))
        gcol += gc
    grad = sum(w * lam[i] for i, w in enumerate(WT))
    return {"J": [float(J[0]), float(J[1])], "rho0": grad,
            "dp": float(sum(float(g) * r for g, r in zip(gcol, E.rates)))}


def exact(case, seed):
    return {"sweep": _exact_sweep, "adjoint": _exact_adjoint}.get(case["form"], _exact_lattice)(case, seed)
