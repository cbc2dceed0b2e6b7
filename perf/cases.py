"""Performance cases of the viscoelastic lattice-Boltzmann framework.

Each case is one call that a user's program makes through the package's
public classes: stepping a lattice and reading its fields, a run from host
buffers to host buffers, stepping a parameter sweep as an ensemble, and the
layers and the prediction of the warm-start network.  `listed()` names the
sizes that are quoted, `draw()` gives further ones of the same ranges, and
`exact()` is the same mathematics in plain FP64 torch.

Set-up of the flows (units of the lattice): G = 1.5, densities 2.0 / 0.1, a
droplet of radius a quarter of the smallest side between walls sheared at
Ca = 0.1, De = 1, L^2 = 100, kappa = 1e-3, polymer in the droplet; started
from the Couette profile with a seeded centre, phase noise and a seeded
deformation of the conformation tensor.
"""
import math

import numpy as np
import torch

RHO_IN, RHO_OUT, WIDTH, SIGMA = 2.0, 0.1, 5.0, 0.09
ETA_B = (RHO_IN + RHO_OUT) / 3.0 * 0.5
STORAGE = {"fp32": 0, "fp16": 1, "bf16": 2}


# --- the cases ---------------------------------------------------------------

def listed():
    return [
        # the smallest flow: single-component FENE-P Couette shear on D2Q9 (the closed-form check), bound by latency
        dict(name="couette_d2q9_64x32", kind="step", lattice="d2q9", nx=64, ny=32, nz=1, ncomp=1, storage="fp32",
             model="default", steps=200),
        # the training box of the warm start: an emulsion time's steps, then the fields
        dict(name="droplet_64cube", kind="step", lattice="d3q19", nx=64, ny=64, nz=64, ncomp=2, storage="fp32",
             model="default", steps=50),
        # the benchmark droplet
        dict(name="droplet_128x64x128", kind="step", lattice="d3q19", nx=128, ny=64, nz=128, ncomp=2, storage="fp32",
             model="default", steps=50),
        # the precision study: 16-bit population deviations on the larger droplet
        dict(name="droplet_256x128x256_fp16", kind="step", lattice="d3q19", nx=256, ny=128, nz=256, ncomp=2,
             storage="fp16", model="default", steps=10),
        # the paper's own scheme (moment space, stress in the equilibrium, Cholesky update) in a box of no round size
        dict(name="paper_model_100x50x70", kind="step", lattice="d3q19", nx=100, ny=50, nz=70, ncomp=2,
             storage="fp32", model="paper", steps=20),
        # a parameter sweep of uneven boxes stepped together, as the warm start's data are made
        dict(name="sweep_20_boxes", kind="ensemble", boxes=20, layout=7, steps=50),
        # a short run from host densities to host fields and diagnostics
        dict(name="host_run_128x64x128", kind="host", lattice="d3q19", nx=128, ny=64, nz=128, ncomp=2,
             storage="fp32", model="default", steps=20),
        # the warm start's prediction for one 64^3 box
        dict(name="unet_predict_64cube", kind="unet", n=64, channels="16,32,80,152"),
        # training of the network's layers: the widest one at full resolution, a down-sampling one of ragged
        # size, and one of the deep levels
        dict(name="conv_48to16_64cube", kind="conv", batch=1, d=64, h=64, w=64, cin=48, cout=16, stride=1),
        dict(name="conv_16to32_down_60x52x44", kind="conv", batch=1, d=60, h=52, w=44, cin=16, cout=32, stride=2),
        dict(name="conv_232to80_16cube", kind="conv", batch=1, d=16, h=16, w=16, cin=232, cout=80, stride=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_box(rng, lo_nodes, hi_nodes):
    nodes = _log_int(rng, lo_nodes, hi_nodes)
    side = nodes ** (1.0 / 3.0)
    nx = max(8, int(side * rng.uniform(0.7, 1.6)))
    ny = max(8, int(side * rng.uniform(0.5, 1.0)))
    if rng.random() < 0.6:  # whole tiles, as most programs choose them; the others are of any size
        nx, ny = max(32, 32 * round(nx / 32)), max(8, 8 * round(ny / 8))
    return nx, ny, max(4, nodes // (nx * ny))


def draw(rng):
    pick = rng.random()
    if pick < 0.10:
        ncomp, steps = rng.choice([1, 1, 2]), rng.randint(40, 300)
        nx, ny = _log_int(rng, 24, 1500), _log_int(rng, 12, 700)
        return dict(kind="step", lattice="d2q9", nx=nx, ny=ny, nz=1, ncomp=ncomp, storage="fp32",
                    model=rng.choice(["default", "default", "paper"]), steps=min(steps, 60_000_000 // (nx * ny)))
    if pick < 0.55:
        nx, ny, nz = _draw_box(rng, 20_000, 6_000_000)
        return dict(kind="step", lattice="d3q19", nx=nx, ny=ny, nz=nz, ncomp=rng.choice([1, 2, 2, 2]),
                    storage=rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"]),
                    model=rng.choice(["default", "default", "paper"]),
                    steps=max(4, min(rng.randint(10, 64), 50_000_000 // (nx * ny * nz))))
    if pick < 0.62:
        return dict(kind="ensemble", boxes=rng.randint(4, 18), layout=rng.randint(1, 10_000), steps=rng.randint(10, 40))
    if pick < 0.70:
        nx, ny, nz = _draw_box(rng, 50_000, 900_000)
        return dict(kind="host", lattice="d3q19", nx=nx, ny=ny, nz=nz, ncomp=2, storage="fp32", model="default",
                    steps=rng.randint(8, 40))
    if pick < 0.78:
        return dict(kind="unet", n=rng.choice([32, 40, 48, 56]), channels=rng.choice(["16,32,64,128", "16,32,80,152",
                                                                                       "8,16,32,64"]))
    cin, cout = rng.choice([5, 8, 16, 24, 32, 48, 80, 112, 152]), rng.choice([8, 16, 32, 80, 152])
    voxels = _log_int(rng, 500, min(262_144, 262_144 * 48 * 16 // (cin * cout)))
    side = voxels ** (1.0 / 3.0)
    d, h, stride = max(3, int(side * rng.uniform(0.7, 1.2))), max(3, int(side * rng.uniform(0.7, 1.2))), rng.choice([1, 1, 2])
    # the backward pass takes layers whose output voxels are a multiple of 8
    w = 8 * stride * max(1, round(voxels / (d * h * 8 * stride)))
    return dict(kind="conv", batch=rng.choice([1, 1, 1, 2]), d=d, h=h, w=w, cin=cin, cout=cout, stride=stride)


# --- set-ups and seeded inputs ------------------------------------------------

def _flow(c):
    """Parameters of the flow in box c (see the module docstring)."""
    if c["lattice"] == "d2q9" and c["ncomp"] == 1:
        eta_s = 1.0 / 6.0
        return dict(c, G=0.0, eta_A=eta_s, eta_B=eta_s, u_wall=0.01, tau_p=1000.0, eta_p=eta_s * 0.4 / 0.6,
                    kappa=0.0, phase=0, R=0.0)
    R = 0.25 * min(c["nx"], c["ny"], c["nz"] if c["lattice"] == "d3q19" else c["ny"])
    rate = 0.1 * SIGMA / (R * ETA_B)
    return dict(c, G=1.5, eta_A=0.6 * ETA_B, eta_B=ETA_B, u_wall=min(0.08, rate * c["ny"] / 2.0),
                tau_p=R * ETA_B / SIGMA / 0.4, eta_p=0.4 * ETA_B, kappa=1e-3, phase=1, R=R)


def _fields(p, seed):
    """(rho_A, rho_B or None, u, C) as FP32 CUDA tensors."""
    nx, ny, nz, dim = p["nx"], p["ny"], p["nz"], 3 if p["lattice"] == "d3q19" else 2
    g = torch.Generator(device="cuda").manual_seed(1 + seed)

    def noise():
        return torch.rand((nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0

    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, None, :]
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[None, :, None]
    z = torch.arange(nz, device="cuda", dtype=torch.float64)[:, None, None]
    if p["ncomp"] == 2:
        off = torch.rand(3, generator=g, device="cuda", dtype=torch.float64).tolist()
        r2 = (x - (nx - 1) / 2.0 - off[0]) ** 2 + (y - (ny - 1) / 2.0 - off[1]) ** 2
        r2 = r2 + ((z - (nz - 1) / 2.0 - off[2]) ** 2 if dim == 3 else 0.0)
        a = RHO_OUT + (RHO_IN - RHO_OUT) * 0.5 * (1.0 + torch.tanh(2.0 * (p["R"] - torch.sqrt(r2)) / WIDTH))
        dphi = 0.5 * (RHO_IN + RHO_OUT) * 1e-3 * noise()
        rhoA, rhoB = (a + dphi).float(), (RHO_IN + RHO_OUT - a - dphi).float()
    else:
        rhoA, rhoB = (1.0 + 1e-3 * noise()).float(), None
    u = torch.zeros((dim, nz, ny, nx), device="cuda", dtype=torch.float64)
    u[0] = p["u_wall"] * (1.0 - 2.0 * (y + 0.5) / ny)
    nc = 6 if dim == 3 else 4
    C = torch.empty((nc, nz, ny, nx), device="cuda", dtype=torch.float64)
    for k in range(nc):
        C[k] = 1.0 + 0.05 * (1.0 + noise()) if k in _DIAG[nc] else 0.02 * noise()
    return rhoA, rhoB, u.float(), C.float()


def _lattice(p, fields):
    from paper_1406_2686_gb300 import vefd
    lat = vefd.Lattice(lattice=vefd.D3Q19 if p["lattice"] == "d3q19" else vefd.D2Q9, nx=p["nx"], ny=p["ny"],
                       nz=p["nz"], ncomp=p["ncomp"], walls=1, G=p["G"], eta_A=p["eta_A"], eta_B=p["eta_B"],
                       delta=0.1, precision=STORAGE[p["storage"]])
    lat.set_wall_shear(p["u_wall"])
    lat.set_fenep(p["tau_p"], p["eta_p"], 100.0, p["kappa"], p["phase"], 1)
    if p["model"] == "paper":
        lat.set_collision(1)
        lat.set_polymer_coupling(1)
        lat.set_conformation_update(1)
    if fields is not None:
        lat.init_fields(*fields)
    return lat


def _boxes(c):
    """The uneven boxes of a sweep: NX in {32, 64, 96}, NY and NZ in {32, 40, ..., 96}."""
    r = np.random.RandomState(c["layout"])
    return [dict(lattice="d3q19", nx=32 * int(r.randint(1, 4)), ny=8 * int(r.randint(4, 13)),
                 nz=8 * int(r.randint(4, 13)), ncomp=2, storage="fp32", model="default") for _ in range(c["boxes"])]


def _conv_inputs(c, seed):
    g = torch.Generator(device="cuda").manual_seed(1 + seed)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    s = c["stride"]
    out = (c["batch"], (c["d"] - 1) // s + 1, (c["h"] - 1) // s + 1, (c["w"] - 1) // s + 1, c["cout"])
    # activations after a ReLU, gradients as a mean loss gives them
    x = torch.relu(randn(c["batch"], c["d"], c["h"], c["w"], c["cin"]))
    dy = randn(*out) / math.sqrt(math.prod(out))
    w = randn(c["cout"], 27 * c["cin"]) * (2.0 / (27 * c["cin"])) ** 0.5
    return x, dy, w, 0.1 * randn(c["cout"])


def _unet_layers(c):
    """(cin, cout, stride, relu) of the network's layers, in the order of UNet.layers."""
    c0, c1, c2, c3 = (int(v) for v in c["channels"].split(","))
    return [(8, c0, 1, True), (c0, c0, 1, True), (c0, c1, 2, True), (c1, c1, 1, True), (c1, c2, 2, True),
            (c2, c2, 1, True), (c2, c3, 2, True), (c3, c3, 1, True), (c3 + c2, c2, 1, True), (c2, c2, 1, True),
            (c2 + c1, c1, 1, True), (c1, c1, 1, True), (c1 + c0, c0, 1, True), (c0, 16, 1, False)]


def _unet_inputs(c, seed):
    n = c["n"]
    g = torch.Generator(device="cuda").manual_seed(1 + seed)
    i = torch.arange(n, device="cuda", dtype=torch.float64) - (n - 1) / 2.0
    r = torch.sqrt(i[:, None, None] ** 2 + i[None, :, None] ** 2 + i[None, None, :] ** 2)
    sc = torch.rand(6, generator=g, device="cuda", dtype=torch.float64)
    x = torch.zeros((1, n, n, n, 8), device="cuda")
    noise = torch.rand((n, n, n), generator=g, device="cuda") * 2e-3 - 1e-3
    # initial phase field, wall-normal coordinate, the five scalars of the set-up
    x[0, ..., 0] = (0.9 * torch.tanh(2.0 * (n * (0.18 + 0.12 * sc[0]) - r) / WIDTH)).float() + noise
    x[0, ..., 1] = (i / (n / 2.0)).float()[None, :, None]
    x[0, ..., 2:7] = (2.0 * sc[1:] - 1.0).float()
    w = [torch.randn(co, 27 * ci, generator=g, device="cuda") * (2.0 / (27 * ci)) ** 0.5
         for ci, co, _, _ in _unet_layers(c)]
    b = [0.05 * torch.randn(co, generator=g, device="cuda") for _, co, _, _ in _unet_layers(c)]
    return x, w, b


# --- what is measured ---------------------------------------------------------

def prepare(case, seed):
    from paper_1406_2686_gb300 import nn, vefd
    c = case
    if c["kind"] == "step":
        p = _flow(c)
        return dict(kind="step", steps=c["steps"], lat=_lattice(p, _fields(p, seed)))
    if c["kind"] == "ensemble":
        ps = [_flow(b) for b in _boxes(c)]
        lats = [_lattice(p, _fields(p, 1000 * seed + i)) for i, p in enumerate(ps)]
        return dict(kind="ensemble", steps=c["steps"], lats=lats, ens=vefd.Ensemble(lats))
    if c["kind"] == "host":
        p = _flow(c)
        rhoA, rhoB, u, _ = _fields(p, seed)
        host = [t.cpu().pin_memory().numpy() for t in (rhoA, rhoB, u)]
        return dict(kind="host", steps=c["steps"], lat=_lattice(p, None), host=host)
    if c["kind"] == "unet":
        x, w, b = _unet_inputs(c, seed)
        net = nn.UNet(8, 16, channels=tuple(int(v) for v in c["channels"].split(",")))
        for lay, wl, bl in zip(net.layers, w, b):
            lay.w.copy_(wl)
            lay.b.copy_(bl)
            lay.pack()
        return dict(kind="unet", net=net, x=x)
    x, dy, w, b = _conv_inputs(c, seed)
    lay = nn.Conv3d(c["cin"], c["cout"], c["stride"], relu=True)
    lay.w.copy_(w)
    lay.b.copy_(b)
    lay.pack()
    return dict(kind="conv", lay=lay, x=x, dy=dy)


def run(state):
    from paper_1406_2686_gb300 import vefd
    s = state
    if s["kind"] == "step":
        lat = s["lat"]
        lat.step(s["steps"])
        return [lat.read(f, device=True) for f in (vefd.PHI, vefd.U, vefd.C)]
    if s["kind"] == "ensemble":
        s["ens"].step(s["steps"], chunk=s["steps"] - s["steps"] % 2)
        return [[lat.read(f, device=True) for f in (vefd.PHI, vefd.U, vefd.C)] for lat in s["lats"]]
    if s["kind"] == "host":
        lat = s["lat"]
        lat.init_fields(*s["host"])
        lat.step(s["steps"])
        return [lat.read(f) for f in (vefd.PHI, vefd.U, vefd.C)] + [lat.diagnostics()]
    if s["kind"] == "unet":
        return s["net"].forward(s["x"])
    lay = s["lay"]
    y = lay.forward(s["x"])
    dx = lay.backward(s["dy"])
    return [y, dx, lay.dw, lay.db]


def _flow_work(c):
    n = c["nx"] * c["ny"] * c["nz"]
    q, nc, dim = (19, 6, 3) if c["lattice"] == "d3q19" else (9, 4, 2)
    ps = 4 if c["storage"] == "fp32" else 2
    # per step: moving populations in their storage type, rest population, C and the AB2 history, read and written
    step = 2 * c["ncomp"] * ((q - 1) * ps + 4) + 4 * 4 * nc
    flop = (30 * q * c["ncomp"] + 60 * nc) + (500 if c["model"] == "paper" else 0)
    return c["steps"] * n * step + n * 4 * (1 + dim + nc), c["steps"] * n * flop


def work(case):
    c = case
    if c["kind"] in ("step", "host"):
        b, f = _flow_work(c)
    elif c["kind"] == "ensemble":
        per = [_flow_work(dict(p, steps=c["steps"])) for p in _boxes(c)]
        b, f = sum(v[0] for v in per), sum(v[1] for v in per)
    elif c["kind"] == "unet":
        b = f = 0
        level = [1, 1, 2, 2, 4, 4, 8, 8, 4, 4, 2, 2, 1, 1]
        for (ci, co, _, _), k in zip(_unet_layers(c), level):
            f += 2 * (c["n"] // k) ** 3 * 27 * ci * co
            b += 4 * 27 * ci * co
        b += 4 * c["n"] ** 3 * (8 + 16)
    else:
        vi = c["batch"] * c["d"] * c["h"] * c["w"]
        s = c["stride"]
        vo = c["batch"] * ((c["d"] - 1) // s + 1) * ((c["h"] - 1) // s + 1) * ((c["w"] - 1) // s + 1)
        f = 3 * 2 * vo * 27 * c["cin"] * c["cout"]
        b = 4 * (2 * vi * c["cin"] + 2 * vo * c["cout"] + 2 * 27 * c["cin"] * c["cout"])
    return {"bytes": b, "flops": f}


# --- the same in FP64 torch ---------------------------------------------------

_DIAG = {6: (0, 3, 5), 4: (0, 2, 3)}
_IJ = {6: [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)], 4: [(0, 0), (0, 1), (1, 1), (2, 2)]}


def _velocities(dim):
    """Velocities and weights (the order does not matter here)."""
    if dim == 2:
        cs = [(x, y, 0) for x in (-1, 0, 1) for y in (-1, 0, 1)]
        return cs, [(4 / 9, 1 / 9, 1 / 36)[abs(x) + abs(y)] for x, y, _ in cs]
    cs = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1) for z in (-1, 0, 1) if abs(x) + abs(y) + abs(z) <= 2]
    return cs, [(1 / 3, 1 / 18, 1 / 36)[abs(x) + abs(y) + abs(z)] for x, y, z in cs]


class _Exact:
    """Two-component Shan-Chen lattice Boltzmann coupled to FENE-P between moving walls (arXiv:1406.2686 Sec. 2)."""

    def __init__(self, p, rhoA, rhoB, u, C):
        self.p, self.dim = p, 3 if p["lattice"] == "d3q19" else 2
        self.nc = 6 if self.dim == 3 else 4
        self.cs, self.w = _velocities(self.dim)
        self.opp = [self.cs.index((-a, -b, -d)) for a, b, d in self.cs]
        self.L2 = 100.0
        rho = [r.double() for r in (rhoA, rhoB) if r is not None]
        u = [v.double() for v in u]
        self.C = [v.double() for v in C]
        self.f = [[self.equilibrium(a, r, u) for a in range(len(self.cs))] for r in rho]
        self.hist = None

    def equilibrium(self, a, rho, u):
        cu = sum(ci * ui for ci, ui in zip(self.cs[a], u) if ci)
        usq = sum(v * v for v in u)
        return self.w[a] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)

    @staticmethod
    def at(v, c, clamp):
        """v at the neighbour x + c: periodic in x and z, in y the wall row itself (clamp) or periodic."""
        if c[0] or c[2]:
            v = torch.roll(v, shifts=(-c[2], -c[0]), dims=(0, 2))
        if c[1]:
            w = torch.roll(v, shifts=-c[1], dims=1)
            if clamp:
                row = -1 if c[1] > 0 else 0
                w[:, row] = v[:, row]
            v = w
        return v

    def grad(self, v, axis):
        """Central difference, one-sided at the walls."""
        if axis != 1:
            e = [0, 0, 0]
            e[axis] = 1
            return 0.5 * (self.at(v, e, False) - self.at(v, [-k for k in e], False))
        d = 0.5 * (self.at(v, (0, 1, 0), True) - self.at(v, (0, -1, 0), True))
        d[:, 0] *= 2.0
        d[:, -1] *= 2.0
        return d

    def lap(self, v):
        l = self.at(v, (1, 0, 0), False) + self.at(v, (-1, 0, 0), False) - 2.0 * v
        y = self.at(v, (0, 1, 0), True) + self.at(v, (0, -1, 0), True) - 2.0 * v
        y[:, 0] = 0.0
        y[:, -1] = 0.0
        if self.dim == 3:
            y += self.at(v, (0, 0, 1), False) + self.at(v, (0, 0, -1), False) - 2.0 * v
        return l + y

    def local(self):
        """Densities, forces, velocity and relaxation of the present state."""
        p, dim = self.p, self.dim
        rho = [sum(f) for f in self.f]
        tot = sum(rho)
        j = [0.0, 0.0, 0.0][:dim]
        for f in self.f:
            for a, c in enumerate(self.cs):
                for k in range(dim):
                    if c[k]:
                        j[k] = j[k] + c[k] * f[a]
        g = [[torch.zeros_like(tot) for _ in range(dim)] for _ in rho]
        if len(rho) == 2:
            for s in range(2):
                for a, c in enumerate(self.cs):
                    if any(c):
                        n = self.at(rho[1 - s], c, True) * self.w[a]
                        for k in range(dim):
                            if c[k]:
                                g[s][k] -= p["G"] * c[k] * rho[s] * n
        phi = (rho[0] - rho[1]) / tot if len(rho) == 2 else torch.ones_like(tot)
        t = torch.tanh(phi / 0.1)
        m = {0: 1.0, 1: 0.5 * (1.0 + t), -1: 0.5 * (1.0 - t)}[p["phase"]]
        ff = (self.L2 - 3.0) / (self.L2 - sum(self.C[k] for k in _DIAG[self.nc]))
        Q = {}
        for k, (a, b) in enumerate(_IJ[self.nc]):
            Q[a, b] = Q[b, a] = (ff * self.C[k] - (1.0 if a == b else 0.0)) * m
        Fp = [torch.zeros_like(tot) for _ in range(dim)]
        beta = p["eta_p"] / p["tau_p"]
        if p["model"] != "paper":
            for k in range(dim):
                for a in range(dim):
                    Fp[k] += beta * self.grad(Q[a, k], a)
        u = [(j[k] + 0.5 * (Fp[k] + sum(g[s][k] for s in range(len(rho))))) / tot for k in range(dim)]
        tau = 0.5 + 3.0 * (p["eta_A"] * 0.5 * (1.0 + t) + p["eta_B"] * 0.5 * (1.0 - t)) / tot
        F = [[g[s][k] + rho[s] / tot * Fp[k] for k in range(dim)] for s in range(len(rho))]
        return rho, tot, phi, u, 1.0 / tau, F, Q, beta

    def collide(self, rho, tot, u, omega, F, Q, beta):
        cs, w, dim = self.cs, self.w, self.dim
        out = []
        usq = sum(v * v for v in u)
        trQ = sum(Q[k, k] for k in range(dim))
        for s, f in enumerate(self.f):
            uF = sum(a * b for a, b in zip(u, F[s]))
            E, S = [], []
            for a, c in enumerate(cs):
                cu = sum((ci * ui for ci, ui in zip(c, u) if ci), torch.zeros_like(tot))
                cF = sum((ci * Fi for ci, Fi in zip(c, F[s]) if ci), torch.zeros_like(tot))
                e = w[a] * rho[s] * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
                if self.p["model"] == "paper":
                    cQc = sum((c[i] * c[k] * Q[i, k] for i in range(dim) for k in range(dim) if c[i] * c[k]),
                              torch.zeros_like(tot))
                    e -= 4.5 * w[a] * rho[s] / tot * beta * (cQc - trQ / 3.0)
                E.append(e)
                S.append(w[a] * (3.0 * (cF - uF) + 9.0 * cu * cF))
            if self.p["model"] == "paper":
                # shear and bulk modes relax with omega, all others at unit rate
                sq = [sum(k * k for k in c) for c in cs]
                if dim == 3:
                    rows = [[19 * q - 30 for q in sq], [3 * c[0] ** 2 - q for c, q in zip(cs, sq)],
                            [c[1] ** 2 - c[2] ** 2 for c in cs], [c[0] * c[1] for c in cs],
                            [c[1] * c[2] for c in cs], [c[0] * c[2] for c in cs]]
                else:
                    rows = [[3 * q - 4 for q in sq], [c[0] ** 2 - c[1] ** 2 for c in cs], [c[0] * c[1] for c in cs]]
                new = [e + 0.5 * q for e, q in zip(E, S)]
                for r in rows:
                    coef = sum(r[a] * (f[a] - E[a] + 0.5 * S[a]) for a in range(len(cs)) if r[a])
                    coef = coef * (1.0 - omega) / sum(v * v for v in r)
                    new = [v + r[a] * coef if r[a] else v for a, v in enumerate(new)]
            else:
                new = [f[a] + omega * (E[a] - f[a]) + (1.0 - 0.5 * omega) * S[a] for a in range(len(cs))]
            out.append(new)
        return out

    def stream(self, post, rho):
        U = self.p["u_wall"]
        self.f = []
        for s, f in enumerate(post):
            new = []
            for a, c in enumerate(self.cs):
                v = torch.roll(f[a], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
                if c[1]:
                    b, row = self.opp[a], 0 if c[1] > 0 else -1
                    cxU = self.cs[b][0] * (U if c[1] > 0 else -U)
                    v[:, row] = f[b][:, row] - 6.0 * self.w[a] * rho[s][:, row] * cxU
                new.append(v)
            self.f.append(new)

    def polymer(self, u):
        nc, dim, p = self.nc, self.dim, self.p
        idx = {}
        for k, (a, b) in enumerate(_IJ[nc]):
            idx[a, b] = idx[b, a] = k
        C = self.C
        Gu = [[self.grad(u[b], a) for b in range(dim)] for a in range(dim)]
        ff = (self.L2 - 3.0) / (self.L2 - sum(C[k] for k in _DIAG[nc]))
        R = []
        for k, (a, b) in enumerate(_IJ[nc]):
            r = p["kappa"] * self.lap(C[k]) - (ff * C[k] - (1.0 if a == b else 0.0)) / p["tau_p"]
            for e in range(dim):
                r -= u[e] * self.grad(C[k], e)
                if (a, e) in idx and b < dim:
                    r += C[idx[a, e]] * Gu[e][b]
                if (e, b) in idx and a < dim:
                    r += Gu[e][a] * C[idx[e, b]]
            R.append(r)
        if p["model"] != "paper":
            old, self.hist = self.hist, R
            self.C = [c + (1.5 * r - 0.5 * q if old else r) for c, r, q in zip(C, R, old or R)]
            return
        # AB2 on the log-Cholesky factor of sigma = f C
        zero = torch.zeros_like(ff)

        def full(v):
            return torch.stack([torch.stack([v[idx[i, j]] if (i, j) in idx else zero for j in range(3)], -1)
                                for i in range(3)], -2)

        fC = ff[..., None, None]
        Cm, Rm = full(C), full(R)
        tr = Rm.diagonal(dim1=-2, dim2=-1).sum(-1)[..., None, None]
        Sm = fC * Cm
        Sd = fC * Rm + Sm * fC * tr / (self.L2 - 3.0)
        L = torch.zeros_like(Sm)
        for i in range(3):
            for j in range(i + 1):
                v = Sm[..., i, j] - (L[..., i, :j] * L[..., j, :j]).sum(-1)
                L[..., i, j] = torch.sqrt(v) if i == j else v / L[..., j, j]
        Li = torch.zeros_like(L)
        for j in range(3):
            Li[..., j, j] = 1.0 / L[..., j, j]
            for i in range(j + 1, 3):
                Li[..., i, j] = -(L[..., i, j:i] * Li[..., j:i, j]).sum(-1) / L[..., i, i]
        A = torch.einsum("...ik,...kl,...jl->...ij", Li, Sd, Li)
        A = torch.tril(A) - 0.5 * torch.diag_embed(A.diagonal(dim1=-2, dim2=-1))
        Ld = torch.einsum("...ik,...kj->...ij", L, A)
        eye = torch.eye(3, device=L.device, dtype=torch.bool)
        lam, rate = torch.where(eye, torch.log(L.where(eye, torch.ones_like(L))), L), torch.where(eye, Ld / L.where(eye, torch.ones_like(L)), Ld)
        old, self.hist = self.hist, rate
        lam = lam + (1.5 * rate - 0.5 * old if old is not None else rate)
        L = torch.where(eye, torch.exp(lam), lam)
        Sn = torch.einsum("...ik,...jk->...ij", L, L)
        fn = (self.L2 - 3.0 + Sn.diagonal(dim1=-2, dim2=-1).sum(-1)) / self.L2
        self.C = [Sn[..., a, b] / fn for a, b in _IJ[nc]]

    def step(self, n):
        for _ in range(n):
            rho, tot, _, u, omega, F, Q, beta = self.local()
            self.stream(self.collide(rho, tot, u, omega, F, Q, beta), rho)
            self.polymer(u)

    def fields(self):
        _, _, phi, u, _, _, _, _ = self.local()
        return [phi, torch.stack(u), torch.stack(self.C)]

    def diagnostics(self):
        """The sixteen reductions, in the order of vefd_diagnostics."""
        rho, tot, phi, u, _, _, _, _ = self.local()
        C, (a, b, d) = self.C, _DIAG[self.nc]
        tr = C[a] + C[b] + C[d]
        ff = (self.L2 - 3.0) / (self.L2 - tr)
        out = np.zeros(16)
        out[0], out[1] = float(rho[0].sum()), float(rho[1].sum())
        for k, v in enumerate(u):
            out[2 + k] = float((tot * v).sum())
        out[5], out[6] = float((ff * C[1]).mean()), float((ff * (C[a] - C[b])).mean())
        out[7], out[8] = float(tr.max()) / self.L2, math.sqrt(float(sum(v * v for v in u).max()))
        inside = (phi[phi.shape[0] // 2] > 0).double()
        y = torch.arange(inside.shape[0], device=phi.device, dtype=torch.float64)[:, None]
        x = torch.arange(inside.shape[1], device=phi.device, dtype=torch.float64)[None, :]
        m = float(inside.sum())
        out[9] = m
        if m > 0:
            cx, cy = float((inside * x).sum()) / m, float((inside * y).sum()) / m
            xx, yy = float((inside * (x - cx) ** 2).sum()) / m, float((inside * (y - cy) ** 2).sum()) / m
            xy = float((inside * (x - cx) * (y - cy)).sum()) / m
            r = math.sqrt(max(0.25 * (xx - yy) ** 2 + xy * xy, 0.0))
            la, lb = math.sqrt(0.5 * (xx + yy) + r), math.sqrt(max(0.5 * (xx + yy) - r, 0.0))
            out[10:14] = (la - lb) / (la + lb) if la + lb > 0 else 0.0, 0.5 * math.atan2(2.0 * xy, xx - yy), cx, cy
        out[14], out[15] = float((phi > 0).sum()), float((ff * tr).mean()) - 3.0
        return out


def _conv(x, w, b, stride, relu):
    """3x3x3 convolution of channels-first x with w [Cout, 27 Cin] (tap-major columns)."""
    cin = x.shape[1]
    k = w.view(w.shape[0], 3, 3, 3, cin).permute(0, 4, 1, 2, 3)
    y = torch.nn.functional.conv3d(x, k, b, stride=stride, padding=1)
    return torch.relu(y) if relu else y


def exact(case, seed):
    c = case
    if c["kind"] in ("step", "host"):
        p = _flow(c)
        rhoA, rhoB, u, C = _fields(p, seed)
        if c["kind"] == "host":  # started from C = I
            C = torch.zeros_like(C)
            C[list(_DIAG[C.shape[0]])] = 1.0
        e = _Exact(p, rhoA, rhoB, u, C)
        e.step(c["steps"])
        if c["kind"] == "step":
            return e.fields()
        return [v.cpu().numpy() for v in e.fields()] + [e.diagnostics()]
    if c["kind"] == "ensemble":
        out = []
        for i, b in enumerate(_boxes(c)):
            p = _flow(b)
            e = _Exact(p, *_fields(p, 1000 * seed + i))
            e.step(c["steps"])
            out.append(e.fields())
        return out
    if c["kind"] == "unet":
        x, w, b = _unet_inputs(c, seed)
        h, skip = x.double().permute(0, 4, 1, 2, 3), []
        layers = [(wl.double(), bl.double(), s, r) for wl, bl, (_, _, s, r) in zip(w, b, _unet_layers(c))]
        for lv in range(4):
            for lay in layers[2 * lv:2 * lv + 2]:
                h = _conv(h, *lay)
            skip.append(h)
        for lv in (2, 1, 0):
            up = h.repeat_interleave(2, 2).repeat_interleave(2, 3).repeat_interleave(2, 4)
            h = torch.cat([up, skip[lv]], 1)
            k = 8 + 2 * (2 - lv)
            for lay in layers[k:k + 2]:
                h = _conv(h, *lay)
        return h.permute(0, 2, 3, 4, 1).contiguous()
    x, dy, w, b = _conv_inputs(c, seed)
    x, w, b = (t.double().requires_grad_() for t in (x, w, b))
    y = _conv(x.permute(0, 4, 1, 2, 3), w, b, c["stride"], True).permute(0, 2, 3, 4, 1)
    dx, dw, db = torch.autograd.grad(y, (x, w, b), dy.double())
    return [y.detach().contiguous(), dx, dw, db]
