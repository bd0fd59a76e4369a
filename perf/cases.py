"""The work that a user of this framework has it do, as timed cases.

Most cases are one job through the context API: initial fields that lie on
the GPU (density, order parameter, velocity), `steps` time steps, and the
fields read back into device tensors -- tlb_init_fields_device, tlb_step,
tlb_get_fields_device, what a driver script does between two outputs.  One
case advances a contact-angle sweep through a resident batch, one takes
requests on host arrays through the server.  The geometries are those of the
package's workloads module (drops on walls, capillary channels, bi-slugs,
periodic drops, lubricated substrates) at its sizes and at odd ones.

A case: `kind` (geometry), `lattice` ("d2q9" or "d3q27"), `nx`, `ny`, `nz`,
`steps`, `wetting` ("force", "extrap", "interp"), `angle` (theta_21 of the
geometric schemes, in degrees; the interpolation's sample point jumps where
the sign of a gradient changes, so rounding shows at single nodes and most
cases take the extrapolation), `kw` (strength of the force scheme), `fp16`
(reduced-precision storage of g), `eos` ("cs", "pr"), `nu` (per-component
viscosities instead of one).  The seed moves and resizes the liquid bodies
and sets the phases of a smooth initial velocity of about 1e-2.
"""
import math
import random

import numpy as np
import torch

from paper_1904_06881_gb300 import tlb
from paper_1904_06881_gb300 import workloads as W

WETTING = {"force": 0, "extrap": 1, "interp": 2}
EOS = {"cs": 0, "pr": 2}
NU = (0.12, 1.0 / 6.0, 0.25)


def _case(name, kind, lattice, nx, ny, nz, steps, wetting="force", angle=90.0, kw=0.0, fp16=False, eos="cs", nu=False):
    return dict(name=name, kind=kind, lattice=lattice, nx=nx, ny=ny, nz=nz, steps=steps, wetting=wetting, angle=angle,
                kw=kw, fp16=fp16, eos=eos, nu=nu)


def listed():
    return [
        # the smallest drop that is run: one wave of few blocks, all latency
        _case("drop2d_64", "drop", "d2q9", 64, 64, 1, 40),
        # the capillary-filling channel: walls with corners, menisci, geometric interpolation
        _case("channel2d_1024x64", "channel", "d2q9", 1024, 64, 1, 30, "interp", 30.0),
        # a self-propelled bi-slug, at its odd channel height and length: ragged tiles
        _case("bislug2d_1001x41", "bislug", "d2q9", 1001, 41, 1, 40, "extrap", 60.0),
        # one lattice of an equation-of-state and viscosity study, an odd size
        _case("drop2d_pr_nu_515x387", "drop", "d2q9", 515, 387, 1, 30, "extrap", 70.0, eos="pr", nu=True),
        # the large two-dimensional lattice, far larger than the L2 cache
        _case("bubble2d_2048", "bubble", "d2q9", 2048, 2048, 1, 20),
        # the smallest three-dimensional substrate that is run
        _case("lubricated3d_32x32x20", "lubricated", "d3q27", 32, 32, 20, 50, kw=0.02),
        # a spherical cap on a wall, geometric extrapolation, odd in every axis
        _case("cap3d_75x61x47", "drop", "d3q27", 75, 61, 47, 30, "extrap", 70.0),
        # the mid-sized substrate of a served mix with reduced-precision g
        _case("lubricated3d_fp16_128", "lubricated", "d3q27", 128, 128, 128, 20, kw=0.02, fp16=True),
        # the headline lattice: a drop over a lubricated substrate
        _case("lubricated3d_192x192x128", "lubricated", "d3q27", 192, 192, 128, 20, kw=0.02),
        # a three-dimensional drop in a periodic box (a surface-tension measurement), no walls at all
        _case("bubble3d_101x100x100", "bubble", "d3q27", 101, 100, 100, 20),
        # a contact-angle sweep: drops of four sizes, two wetting schemes, one resident batch
        dict(name="sweep2d_16", kind="sweep", lattices=16, largest=512, steps=30),
        # requests on host arrays through the server: create, run, read back
        dict(name="served_12", kind="served", requests=12, largest=256, steps=160),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    pick = rng.random()
    if pick < 0.08:
        return dict(kind="sweep", lattices=rng.randint(4, 16), largest=rng.choice([128, 256, 512]),
                    steps=rng.randint(20, 30))
    if pick < 0.14:
        return dict(kind="served", requests=rng.randint(3, 10), largest=rng.choice([128, 256]),
                    steps=rng.randint(50, 160))
    wetting = rng.choice(["force", "extrap"])
    angle = round(rng.uniform(50.0, 115.0), 1)
    kw = round(rng.uniform(0.0, 0.1), 3) if wetting == "force" else 0.0
    fp16 = rng.random() < 0.2
    eos = "pr" if rng.random() < 0.12 else "cs"
    nu = rng.random() < 0.15
    if pick < 0.55:
        kind = rng.choice(["drop", "drop", "channel", "bislug", "bubble"])
        n = math.exp(rng.uniform(math.log(64 * 64), math.log(2048 * 2048)))   # nodes
        if kind in ("drop", "channel") and rng.random() < 0.4:
            wetting, kw = "interp", 0.0
        if kind in ("channel", "bislug"):
            ny = rng.randint(41, 96)
            nx = min(4096, max(256, int(n / ny)))
        else:
            nx = max(56, int(math.sqrt(n) * rng.uniform(0.8, 1.25)))
            ny = max(56, int(n / nx))
        steps = max(15, min(30, int(40 * 2.0e6 / (nx * ny))))
        return _case(None, kind, "d2q9", nx, ny, 1, steps, wetting, angle, kw, fp16, eos, nu) | {"name": "drawn"}
    kind = rng.choice(["drop", "lubricated", "lubricated", "bubble"])
    n = log_int(24, 150)
    nx, ny, nz = (max(20, int(n * rng.uniform(0.8, 1.25))) for _ in range(3))
    if rng.random() < 0.5:
        nx += -nx % 8              # most are whole numbers of 32-byte segments long
    steps = max(10, min(40, int(20 * 4.0e6 / (nx * ny * nz))))
    return _case(None, kind, "d3q27", nx, ny, nz, steps, wetting, angle, kw, fp16, eos, nu) | {"name": "drawn"}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _params(case):
    """Keyword parameters of a lattice (names of the package's make_params)."""
    p = W.base_params(wetting=WETTING[case["wetting"]])
    a = case["angle"]
    if case["wetting"] == "force":
        p.update(kw_rho=case["kw"])
    elif case["kind"] == "channel":
        p.update(theta_deg=(a, a, 120.0))
    elif case["kind"] == "bislug":
        p.update(theta_deg=(a, a, a))
    else:
        p.update(theta_deg=(a, a, 90.0))
    if case["eos"] != "cs":
        p.update(eos=EOS[case["eos"]], rho_g=W.RHO_L / 10.0)
    if case["nu"]:
        p.update(nu=NU)
    if case["fp16"]:
        p.update(g_fp16=1)
    return p


def _geometry(case, seed):
    """(mask uint8 numpy, rho, phi, u float32 tensors) of a case; shapes (nz, ny, nx) and (D, nz, ny, nx)."""
    rng = random.Random("%s %s" % (seed, case["kind"]))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    D = 2 if case["lattice"] == "d2q9" else 3
    dev = _device()
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device=dev) for n in (nz, ny, nx)), indexing="ij")
    jit = [rng.uniform(-2.0, 2.0) for _ in range(3)]
    grow = rng.uniform(0.95, 1.05)
    mask = np.zeros((nz, ny, nx), np.uint8)
    zero = torch.zeros_like(x)

    def blob(dist, R):
        return 0.5 * (1.0 - torch.tanh((dist - R) / 2.0))

    kind = case["kind"]
    if kind == "drop":                       # a cap on the wall below, a wall above
        xc, yc = nx / 2.0 + jit[0], ny / 2.0 + jit[1]
        if D == 2:
            C2 = blob(torch.hypot(x - xc, y - 0.5), 0.25 * min(nx, ny) * grow)
            mask[:, 0] = mask[:, ny - 1] = 1
        else:
            C2 = blob(torch.sqrt((x - xc) ** 2 + (y - yc) ** 2 + (z - 0.5) ** 2), 0.25 * min(nx, ny, 2 * nz) * grow)
            mask[0] = mask[nz - 1] = 1
        C3 = zero
    elif kind == "channel":                  # a liquid reservoir, a channel between slabs, gas behind it
        wall, xi, xo = (12 * ny) // 64, nx // 4, nx - nx // 16
        mask[:, :wall, xi:xo] = mask[:, ny - wall:, xi:xo] = 1
        xp = torch.remainder(x - (0.5 * (xi - 1) + jit[0]) + nx / 2, nx) - nx / 2
        C2, C3 = blob(xp.abs(), 0.5 * xi * grow), zero
    elif kind == "bislug":                   # a slug of liquid 1 followed by one of liquid 2
        mask[:, 0] = mask[:, ny - 1] = 1
        L = 0.3 * nx * grow
        x0 = 0.2 * nx + jit[0]
        e = [0.5 * (1.0 + torch.tanh((x - x0 - k * L) / 2.0)) for k in range(3)]
        C2, C3 = e[0] - e[1], e[1] - e[2]
    elif kind == "bubble":                   # a drop in a periodic box
        d2 = (x - nx / 2.0 - jit[0]) ** 2 + (y - ny / 2.0 - jit[1]) ** 2
        if D == 3:
            d2 = d2 + (z - nz / 2.0 - jit[2]) ** 2
        C2, C3 = blob(torch.sqrt(d2), 0.25 * min((nx, ny, nz)[:D]) * grow), zero
    else:                                    # a drop of liquid 1 above a film of liquid 2
        R = grow * min(nx, ny, nz) / 6.0
        lub = max(3, nz // 20)
        C2 = blob(torch.sqrt((x - nx / 2.0 - jit[0]) ** 2 + (y - ny / 2.0 - jit[1]) ** 2 + (z - lub - 3 - R) ** 2), R)
        C3 = 0.5 * (1.0 - torch.tanh((z - (lub + 0.5)) / 2.0)) * (1.0 - C2)
        mask[0] = mask[nz - 1] = 1
    p = _params(case)
    fluid = torch.from_numpy(1 - mask).to(dev)
    C1 = 1.0 - C2 - C3
    rho = (p["rho_l"] + C1 * (p["rho_g"] - p["rho_l"])) * fluid
    phi = p["chi"] * (C2 - C3) * fluid
    u = torch.empty((D,) + x.shape, dtype=torch.float32, device=dev)
    for a in range(D):                       # acoustic and shear waves left by what went before
        w = zero
        for c, n in ((x, nx), (y, ny), (z, nz))[:D]:
            w = w + rng.uniform(0.5, 1.5) * torch.sin((2 * math.pi / n) * c + rng.uniform(0, 2 * math.pi))
        u[a] = 1e-2 * w * fluid
    return mask, rho.float(), phi.float(), u


def _lattice(case):
    lat = W.D2Q9 if case["lattice"] == "d2q9" else W.D3Q27
    return tlb.Lattice(lat, case["nx"], case["ny"], case["nz"], **_params(case))


class _Job:
    """A lattice, its initial fields and the tensors its results go to."""

    def __init__(self, case, seed):
        mask, self.rho, self.phi, self.u = _geometry(case, seed)
        self.lat = _lattice(case)
        self.lat.set_solid(mask)
        self.out = [torch.empty_like(t) for t in (self.rho, self.phi, self.u)]

    def start(self):
        tlb.tlb_init_fields_device(self.lat.h, self.rho.data_ptr(), self.phi.data_ptr(), self.u.data_ptr())

    def read(self):
        tlb.tlb_get_fields_device(self.lat.h, *(t.data_ptr() for t in self.out))
        return self.out


def _sweep_members(case, seed):
    """The lattices of a sweep: drops of sizes up to `largest`, both wetting schemes."""
    rng = random.Random("sweep %s" % seed)
    sizes = [s for s in (64, 128, 256, 512) if s <= case["largest"]]
    out = []
    for k in range(case["lattices"]):
        L = sizes[k // 2 % len(sizes)]
        angle = rng.uniform(50.0, 115.0)
        wet = ("force", "extrap")[k % 2]
        out.append(_case("m", "drop", "d2q9", L, L, 1, case["steps"], wet, angle,
                         kw=W.provisional_kw(angle) if wet == "force" else 0.0))
    return out


def _served_members(case, seed):
    """The requests of a served mix: drops, channels and substrates, each for its own number of steps."""
    rng = random.Random("served %s" % seed)
    out = []
    for k in range(case["requests"]):
        steps = max(20, int(case["steps"] * (0.5 + 0.125 * (k % 5))))
        if k % 6 == 5:
            n = min(64, case["largest"] // 2)
            out.append(_case("m", "lubricated", "d3q27", n, n, n, steps, kw=0.02))
        elif k % 3 == 2:
            out.append(_case("m", "channel", "d2q9", 2 * case["largest"], 64, 1, steps, "interp", rng.uniform(50.0, 115.0)))
        else:
            L = case["largest"] >> (k % 2)
            out.append(_case("m", "drop", "d2q9", L, L, 1, steps, "interp", rng.uniform(50.0, 115.0)))
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    if s.kind == "sweep":
        s.jobs = [_Job(m, seed * 1000 + k) for k, m in enumerate(_sweep_members(case, seed))]
        s.batch = tlb.Batch([j.lat for j in s.jobs])
    elif s.kind == "served":
        s.server = tlb.Server(budget_bytes=8 << 30)
        s.requests = []
        for k, m in enumerate(_served_members(case, seed)):
            mask, rho, phi, _ = _geometry(m, seed * 1000 + k)
            s.requests.append((m, mask, rho.double().cpu().numpy(), phi.double().cpu().numpy()))
    else:
        s.job = _Job(case, seed)
    return s


def run(s):
    if s.kind == "sweep":
        for j in s.jobs:
            j.start()
        s.batch.step(s.case["steps"])
        return [j.read() for j in s.jobs]
    if s.kind == "served":
        tickets = [s.server.submit(W.D2Q9 if m["lattice"] == "d2q9" else W.D3Q27, m["nx"], m["ny"], m["nz"], mask, rho,
                                   phi, m["steps"], **_params(m)) for m, mask, rho, phi in s.requests]
        while s.server.pump() > 0 or s.server.stats()["queued"]:
            pass
        done = [s.server.poll(t) for t in tickets]
        # the library computes in FP32 and hands FP64 arrays out: the fields in the precision they have
        return [[d["rho"].astype(np.float32), d["phi"].astype(np.float32)] for d in done]
    s.job.start()
    tlb.tlb_step(s.job.lat.h, s.case["steps"])
    return s.job.read()


def work(case):
    """Bytes: the populations f and g read and written once a step, the fields in and out once.  Flops: the arithmetic of
    a step per node (stencils, chemical potentials, equilibria, entropic collision, both relaxations), counted by hand."""
    if case["kind"] in ("sweep", "served"):
        parts = [work(m) for m in (_sweep_members if case["kind"] == "sweep" else _served_members)(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    d3 = case["lattice"] == "d3q27"
    Q, D = (27, 3) if d3 else (9, 2)
    N = case["nx"] * case["ny"] * case["nz"]
    g = 4 + 2 * (Q - 1) if case["fp16"] else 4 * Q
    return {"bytes": float(N * (case["steps"] * 2 * (4 * Q + g) + 2 * 4 * (2 + D))),
            "flops": float(N * case["steps"] * (1500 if d3 else 550))}


# ---------------------------------------------------------------------------
# The same job in 64 bits (plain torch)
# ---------------------------------------------------------------------------
def _pressure(kind, b, R, T, A, r):
    e = b * r / 4.0
    if kind == "cs":
        return r * R * T * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - A * r * r
    return r * R * T / (1 - b * r) - A * r * r / (1 + 2 * b * r - (b * r) ** 2)


def _psi(kind, b, R, T, A, C, r, log):
    """Psi_eos and its derivative: Carnahan-Starling as printed (Eq. PsiEOS), Peng-Robinson from p = rho Psi' - Psi."""
    br, RT = b * r, R * T
    if kind == "cs":
        q = br - 4.0
        psi = r * (C - A * r - 8 * RT * (br - 6) / (q * q) + RT * log(r))
        return psi, C - 2 * A * r + RT * (1 + log(r)) + 16 * RT * (br - 12) / q ** 3
    s2 = math.sqrt(2.0)
    lg, L = log(r / (1 - br)), A / (2 * s2 * b) * log((br + s2 - 1) / (s2 + 1 - br))
    return r * (C + RT * lg - L), C + RT * lg + RT / (1 - br) - L - A * r / (1 + 2 * br - br * br)


def _equation_of_state(kind, a, b, R, rho_l, rho_g):
    """(b, RT, attraction, C, Psi0): the temperature at which the densities' ratio coexists, a and b rescaled to them."""
    ratio = rho_l / rho_g

    def attraction(T):
        if kind == "cs":
            return a
        k = 0.37464 + 1.54226 * 0.344 - 0.26992 * 0.344 ** 2
        return a * (1 + k * (1 - math.sqrt(T / ((0.07780 / 0.45724) * a / (b * R))))) ** 2

    def temperature(rg):                     # equal pressures
        lo, hi = 1e-4 * a / (b * R), a / (b * R)
        for _ in range(200):
            T = 0.5 * (lo + hi)
            d = _pressure(kind, b, R, T, attraction(T), ratio * rg) - _pressure(kind, b, R, T, attraction(T), rg)
            lo, hi = (lo, T) if d > 0 else (T, hi)
        return 0.5 * (lo + hi)

    def gap(rg):                             # difference of the chemical potentials
        T = temperature(rg)
        return (_psi(kind, b, R, T, attraction(T), 0.0, ratio * rg, math.log)[1]
                - _psi(kind, b, R, T, attraction(T), 0.0, rg, math.log)[1])

    top = (4.0 if kind == "cs" else 1.0) / b / ratio
    grid = [top * (k + 0.5) / 400 for k in range(400)]
    g = [gap(r) for r in grid]
    k = next(k for k in range(len(g) - 1) if (g[k] < 0) != (g[k + 1] < 0))
    lo, hi = grid[k], grid[k + 1]
    for _ in range(100):
        m = 0.5 * (lo + hi)
        lo, hi = (m, hi) if (gap(m) < 0) == (g[k] < 0) else (lo, m)
    rg = 0.5 * (lo + hi)
    T = temperature(rg)
    s = ratio * rg / rho_l
    A, b = attraction(T) * s, b * s
    C = -_psi(kind, b, R, T, A, 0.0, rho_l, math.log)[1]
    return b, R * T, A, C, _psi(kind, b, R, T, A, C, rho_l, math.log)[0]


class _Exact:
    """The time step of Sec. II-IV (arXiv:1904.06881) on float64 tensors shaped (nz, ny, nx)."""

    def __init__(self, case, mask):
        self.p = p = _params(case)
        self.wet, self.kind = case["wetting"], case["eos"]
        self.D = D = 2 if case["lattice"] == "d2q9" else 3
        self.c = [(x, y, z) for z in ((0,) if D == 2 else (-1, 0, 1)) for y in (-1, 0, 1) for x in (-1, 0, 1)]
        self.Q = len(self.c)
        self.w = [math.prod((2 / 3 if k == 0 else 1 / 6) for k in c[:D]) for c in self.c]
        self.solid = torch.from_numpy(mask.astype(bool)).to(_device())
        self.walls = bool(mask.any())
        self.fluid = ~self.solid
        self.rl, self.rg, self.chi = p["rho_l"], p["rho_g"], p["chi"]
        drho = self.rl - self.rg
        k = p["kappa"]
        self.krr = k[0] + (k[1] + k[2]) / (4 * drho * drho)
        self.kpp = (k[1] + k[2]) / (4 * self.chi ** 2)
        self.krp = (k[1] - k[2]) / (4 * self.chi * drho)
        self.b, self.RT, self.A, self.C, self.Psi0 = _equation_of_state(self.kind, p["a"], p["b"], p["R"], self.rl, self.rg)
        self.cot = [1.0 / math.tan(math.radians(t)) for t in p["theta_deg"]]
        if self.walls:
            touch = torch.zeros_like(self.solid)
            for c in self.c:
                touch |= self.at(self.solid, c) != self.solid
            self.first = self.fluid & touch
            self.ghost = (self.solid & touch).nonzero().flip(1)       # columns x, y, z
            self.axis_wall = [self.at(self.solid, self.unit(a, 1)) | self.at(self.solid, self.unit(a, -1)) for a in range(3)]

    @staticmethod
    def unit(a, s):
        return tuple(s if b == a else 0 for b in range(3))

    @staticmethod
    def at(t, c):
        """t at the node x + c of every node x."""
        sh = [(-c[2 - k], k - 3) for k in range(3) if c[2 - k]]
        return torch.roll(t, [s for s, _ in sh], [d for _, d in sh]) if sh else t

    def index(self, X):
        nz, ny, nx = self.solid.shape
        return torch.remainder(X[:, 0], nx) + nx * (torch.remainder(X[:, 1], ny) + ny * torch.remainder(X[:, 2], nz))

    def fetch(self, X, own):
        """(is fluid, rho, phi) at the nodes X; rho and phi those of the node itself (`own`) off the fluid."""
        n = self.index(X)
        f = self.fluid.reshape(-1)[n]
        return f, torch.where(f, self.m[0].reshape(-1)[n], own[0]), torch.where(f, self.m[1].reshape(-1)[n], own[1])

    def ghost_axis(self, Y, own, axis):
        """Ghost values behind the first fluid nodes Y, `axis` the wall normal (Sec. IV.A-B)."""
        if self.wet == "force":
            return own
        t = [a for a in range(self.D) if a != axis]
        e = [torch.tensor(self.unit(a, 1), device=Y.device) for a in t]
        dr, dp = [], []
        for k in range(len(t)):
            (fa, ra, pa), (fb, rb, pb) = self.fetch(Y + e[k], own), self.fetch(Y - e[k], own)
            h = torch.where(fa & fb, 0.5, 1.0)          # a solid neighbour holds the node's own value: one-sided
            dr.append(h * (ra - rb))
            dp.append(h * (pa - pb))
        nr, npp = (torch.sqrt(sum(v * v for v in d)) for d in (dr, dp))
        dot = sum(a * b for a, b in zip(dr, dp))
        liquid = own[0] > 0.5 * self.rl
        p13 = torch.where(liquid & (own[1] < -0.95 * self.chi), True,
                          torch.where(liquid & (own[1] > 0.95 * self.chi), False, dot < 0))
        p23 = nr < 0.01 * (self.rl - self.rg) / self.chi * npp
        nc = torch.where(p23, npp, nr)
        cot = torch.where(p23, self.cot[2], torch.where(p13, self.cot[1], self.cot[0])).double()
        flat = ~(nc > 1e-12)
        tt = [torch.where(p23, b, a) / torch.where(flat, 1.0, nc) for a, b in zip(dr, dp)]
        if self.wet == "extrap":
            g = [own[0] + cot * sum(a * b for a, b in zip(dr, tt)), own[1] + cot * sum(a * b for a, b in zip(dp, tt))]
        elif len(t) == 1:
            l = cot * tt[0]
            l0 = torch.floor(l)
            a, b = (self.fetch(Y + (l0 + k).long()[:, None] * e[0], own) for k in (0, 1))
            g = [a[k] + (l - l0) * (b[k] - a[k]) for k in (1, 2)]
        else:
            lx, ly = cot * tt[0], cot * tt[1]
            flat = flat | (torch.hypot(lx, ly) < 1e-12)
            cx, cy = ([torch.floor(v) + k for k in d] for v, d in ((lx, (0, 1, 0, 1)), (ly, (0, 0, 1, 1))))
            dist = torch.stack([a * a + b * b for a, b in zip(cx, cy)])
            drop, best = torch.zeros_like(lx).long(), dist[0]
            for k in range(1, 4):                       # the first of the nearest corners
                nearer = dist[k] < best
                drop, best = torch.where(nearer, k, drop), torch.where(nearer, dist[k], best)
            kept = [torch.where(drop <= k, k + 1, k) for k in range(3)]
            px = [torch.stack(cx).gather(0, k[None])[0] for k in kept]
            py = [torch.stack(cy).gather(0, k[None])[0] for k in kept]
            v = [self.fetch(Y + a.long()[:, None] * e[0] + b.long()[:, None] * e[1], own) for a, b in zip(px, py)]
            ax, ay, bx, by = px[1] - px[0], py[1] - py[0], px[2] - px[0], py[2] - py[0]
            det = ax * by - bx * ay
            qx, qy = lx - px[0], ly - py[0]
            l1, l2 = (qx * by - bx * qy) / det, (ax * qy - qx * ay) / det
            g = [v[0][k] + l1 * (v[1][k] - v[0][k]) + l2 * (v[2][k] - v[0][k]) for k in (1, 2)]
        return [torch.where(flat, own[k], g[k]) for k in (0, 1)]

    def fill_ghosts(self):
        """rho and phi of the ghost nodes: the mean over the axis directions that meet fluid, else over the diagonals."""
        G = self.ghost
        zero = torch.zeros(len(G), dtype=torch.float64, device=G.device)
        tot, cnt = [zero, zero], zero
        for a in range(self.D):
            for s in (-1, 1):
                Y = G + torch.tensor(self.unit(a, s), device=G.device)
                f, r, ph = self.fetch(Y, [zero, zero])
                g = self.ghost_axis(Y, [r, ph], a)
                tot = [torch.where(f, t + v, t) for t, v in zip(tot, g)]
                cnt = cnt + f
        alone = cnt == 0
        for c in self.c:
            f, r, ph = self.fetch(G + torch.tensor(c, device=G.device), [zero, zero])
            f = f & alone
            tot = [torch.where(f, t + v, t) for t, v in zip(tot, (r, ph))]
            cnt = cnt + f
        n = self.index(G)
        for k in (0, 1):
            self.m[k].view(-1)[n] = tot[k] / cnt

    def thermo(self):
        """mu_phi and Q = rho c_s^2 I - P of the fluid nodes (0 at solid ones), from rho, phi with the ghost layer filled."""
        r, ph = self.m
        D, w = self.D, self.w
        g = [[torch.zeros_like(r) for _ in range(D)] for _ in range(2)]
        lap = [torch.zeros_like(r) for _ in range(2)]
        for c, wi in zip(self.c, w):
            if any(c):
                for k in range(2):
                    q = self.at(self.m[k], c)
                    for a in range(D):
                        if c[a]:
                            g[k][a] += 3 * wi * c[a] * q
                    lap[k] += 6 * wi * (q - self.m[k])
        p, drho, chi = self.p, self.rl - self.rg, self.chi
        safe = torch.where(self.fluid, r, self.rl)
        psi, dpsi = _psi(self.kind, self.b, 1.0, self.RT, self.A, self.C, safe, torch.log)
        C1 = (r - self.rl) / (self.rg - self.rl)
        C2, C3 = 0.5 * (1 + ph / chi - C1), 0.5 * (1 - ph / chi - C1)
        l = p["lam"]
        g2, g3 = (v * (v - 0.5) * (v - 1) for v in (C2, C3))
        fb = 0.5 * (l[0] * (psi - self.Psi0) + l[1] * (C2 * (1 - C2)) ** 2 + l[2] * (C3 * (1 - C3)) ** 2)
        mur = 0.5 * l[0] * dpsi + (l[1] * g2 + l[2] * g3) / drho
        mup = (l[1] * g2 - l[2] * g3) / chi
        krr, kpp, krp = self.krr, self.kpp, self.krp
        dots = [sum(a * b for a, b in zip(*v)) for v in ((g[0], g[0]), (g[1], g[1]), (g[0], g[1]))]
        iso = (r * mur + ph * mup - fb - krr * (r * lap[0] + 0.5 * dots[0]) - kpp * (ph * lap[1] + 0.5 * dots[1])
               - krp * (r * lap[1] + ph * lap[0] + dots[2]))
        mup = mup - kpp * lap[1] - krp * lap[0]
        q = {}
        for a in range(D):
            for b in range(a, D):
                v = krr * g[0][a] * g[0][b] + kpp * g[1][a] * g[1][b] + krp * (g[0][a] * g[1][b] + g[1][a] * g[0][b])
                v = (r / 3.0 - iso if a == b else 0.0) - v
                q[a, b] = q[b, a] = torch.where(self.fluid, v, 0.0)
        return mup, q

    def force(self, q):
        """F = div Q with the wall rules, and the wetting force of the force scheme (Sec. IV)."""
        D = self.D
        F = [torch.zeros_like(self.m[0]) for _ in range(D)]
        for c, wi in zip(self.c, self.w):
            for b in range(D):
                if c[b]:
                    for a in range(D):
                        F[a] += 3 * wi * c[b] * self.at(q[a, b], c)
        if not self.walls:
            return F
        X = self.first.nonzero().flip(1)
        n = self.index(X)
        wall = [v.reshape(-1)[n] for v in self.axis_wall]
        sol = self.solid.reshape(-1)
        val = {k: v.reshape(-1) for k, v in q.items()}
        Fw = [torch.zeros(len(n), dtype=torch.float64, device=n.device) for _ in range(D)]
        for c, wi in zip(self.c, self.w):
            if not any(c):
                continue
            m = self.index(X + torch.tensor(c, device=X.device))
            hit = sol[m]
            mc = torch.stack([torch.where(wall[a], -c[a], c[a]) for a in range(3)], 1)
            mm = self.index(X + mc)
            mirror = torch.where(hit, torch.where(sol[mm], n, mm), m)
            for b in range(D):
                if not c[b]:
                    continue
                for a in range(D):
                    v = val[a, b]
                    one = torch.where(hit, 0.0, 2.0 * (v[m] - v[n]))
                    Fw[a] += 3 * wi * c[b] * torch.where(wall[b], one, v[mirror])
        for a in range(D):
            F[a].view(-1)[n] = Fw[a]
        kr, kp = self.p["kw_rho"], self.p["kw_phi"]
        if self.wet == "force" and (kr or kp):
            amp = (self.m[0] - self.rg) / (self.rl - self.rg) * (kr + self.m[1] / self.chi * kp)
            amp = torch.where(self.fluid & ~self.first, amp, 0.0)
            for c, wi in zip(self.c, self.w):
                near = self.at(self.first, c)
                for a in range(D):
                    if c[a]:
                        F[a] += amp * near * (wi * c[a])
        return F

    def equilibrium(self, r, u):
        f = []
        for v in u:
            s = torch.sqrt(1 + 3 * v * v)
            A, B = 2 - s, (2 * v + s) / (1 - v)
            f.append({0: 2 / 3 * A, 1: A * B / 6, -1: A / B / 6})
        for c in self.c:
            e = r
            for a in range(self.D):
                e = e * f[a][c[a]]
            yield e

    def g_equilibrium(self, ph, v, mup):
        v2 = sum(a * a for a in v)
        out = []
        for c, wi in zip(self.c, self.w):
            cv = sum(c[a] * v[a] for a in range(self.D))
            out.append(wi * (3 * self.p["Gamma"] * mup + 3 * ph * cv + 4.5 * ph * cv * cv - 1.5 * ph * v2))
        rest = self.c.index((0, 0, 0))
        out[rest] = ph - sum(e for i, e in enumerate(out) if i != rest)
        return out

    def alpha(self, fp, x):
        """Root of the entropy condition (Eq. EntropyEquation) in x_i = (f^eq_i - f_i) / f'_i, by bracketed Newton."""
        xmax = torch.stack([v.abs() for v in x]).amax(0)
        neg = torch.stack([-v for v in x]).amax(0)
        bound = torch.where(neg > 0, 1.0 / torch.where(neg > 0, neg, 1.0), 1e30) * (1 - 1e-6)
        al = torch.full_like(xmax, 2.0)
        todo = (xmax >= 1e-6).reshape(-1).nonzero()[:, 0]
        if not len(todo):
            return al
        F = torch.stack([v.reshape(-1)[todo] for v in fp])
        X = torch.stack([v.reshape(-1)[todo] for v in x])
        L = torch.log1p(X)
        hi = bound.reshape(-1)[todo]
        lo = torch.ones_like(hi)

        def h(a):
            y = a * X
            ly = torch.log1p(y)
            ent = torch.where(y.abs() < 1e-3, y * y * (0.5 - y * (1 / 6 - y * (1 / 12 - y * (1 / 20 - y / 30)))),
                              (1 + y) * ly - y)
            return (F * (ent - y * L)).sum(0), (F * X * (ly - L)).sum(0)

        none = h(hi)[0] < 0                              # no root below the positivity bound
        a = torch.where(hi > 2.0, 2.0, 0.5 * (lo + hi))
        for _ in range(60):
            v, d = h(a)
            hi, lo = torch.where(v > 0, a, hi), torch.where(v > 0, lo, a)
            nxt = a - v / d
            nxt = torch.where((d > 0) & (nxt > lo) & (nxt < hi), nxt, 0.5 * (lo + hi))
            moved = (torch.where(none, a, nxt) - a).abs().max()
            a = nxt
            if moved < 1e-11:
                break
        al.view(-1)[todo] = torch.where(none, bound.reshape(-1)[todo], a)
        return al

    def beta(self):
        if "nu" not in self.p:
            return self.p["beta"]
        C1 = (self.m[0] - self.rl) / (self.rg - self.rl)
        ph = self.m[1] / self.chi
        c = [v.clamp(0, 1) for v in (C1, 0.5 * (1 + ph - C1), 0.5 * (1 - ph - C1))]
        return 1.0 / (6.0 * sum(a * n for a, n in zip(c, self.p["nu"])) / (c[0] + c[1] + c[2]) + 1.0)

    def stream(self, f):
        out = []
        for i, c in enumerate(self.c):
            back = (-c[0], -c[1], -c[2])
            v = self.at(f[i], back)
            if self.walls and i != self.c.index(back):
                v = torch.where(self.at(self.solid, back), f[self.c.index(back)], v)
            out.append(v)
        return out

    def velocity(self):
        r = torch.where(self.fluid, self.m[0], 1.0)
        return [sum(c[a] * f for c, f in zip(self.c, self.f) if c[a]) / r for a in range(self.D)]

    def moments(self):
        self.m = [torch.where(self.fluid, sum(v), 0.0) for v in (self.f, self.g)]

    def init(self, rho, phi, u):
        self.m = [rho.clone(), phi.clone()]
        if self.walls:
            self.fill_ghosts()
        self.start = [v.clone() for v in self.m]
        mup, q = self.thermo()
        F = self.force(q)
        r = torch.where(self.fluid, self.m[0], 1.0)
        self.f = list(self.equilibrium(r, [u[a] - 0.5 * F[a] / r for a in range(self.D)]))
        self.g = self.g_equilibrium(self.m[1], list(u), mup)

    def step(self):
        self.moments()
        if self.walls:
            self.fill_ghosts()
        mup, q = self.thermo()
        F = self.force(q)
        del q
        r = torch.where(self.fluid, self.m[0], 1.0)
        u = [torch.where(self.fluid, v, 0.0) for v in self.velocity()]
        du = [torch.where(self.fluid, v / r, 0.0) for v in F]
        fp, x, f = [], [], self.f
        for i, (e, ed) in enumerate(zip(self.equilibrium(r, u), self.equilibrium(r, [a + b for a, b in zip(u, du)]))):
            fi = torch.where(self.fluid, f[i], e) if self.walls else f[i]
            fp.append(fi + ed - e)
            x.append((e - fi) / fp[-1])
            f[i] = None
        ab = self.alpha(fp, x) * self.beta()
        for i in range(self.Q):
            fp[i] += ab * (x[i] * fp[i])
            x[i] = None
        self.f = self.stream(fp)
        ge = self.g_equilibrium(self.m[1], [a + 0.5 * b for a, b in zip(u, du)], mup)
        for i in range(self.Q):
            ge[i] = self.g[i] + (ge[i] - self.g[i]) / self.p["tau_g"]
        self.g = self.stream(ge)


def exact(case, seed):
    if case["kind"] == "served":
        return None
    if case["kind"] == "sweep":
        return [exact(m, seed * 1000 + k) for k, m in enumerate(_sweep_members(case, seed))]
    mask, rho, phi, u = _geometry(case, seed)
    e = _Exact(case, mask)
    e.init(rho.double(), phi.double(), u.double())
    start = e.start
    for _ in range(case["steps"]):
        e.step()
    e.moments()
    v = torch.stack([torch.where(e.fluid, a, 0.0) for a in e.velocity()])
    if e.walls:                       # device fields keep the initial ghost layer at the solid nodes next to fluid
        g = torch.zeros_like(e.solid)
        g.view(-1)[e.index(e.ghost)] = True
        e.m = [torch.where(g, a, b) for a, b in zip(start, e.m)]
    return [e.m[0], e.m[1], v]
