"""What the performance of this library is measured on: the simulations and the
surrogate's layers that its users run, through the public entry points.

Solver cases ("kind": "lbm") make a context, set geometry and fields, and a
pass is one of
  "restart"  lbm_set_fields, lbm_step, lbm_get_fields (a parameter study: every
             run starts from new fields on the same geometry);
  "solve"    lbm_set_geometry, lbm_set_fields, lbm_step, lbm_get_fields (a new
             geometry every time);
  "steady"   lbm_set_fields, lbm_run_to_steady, lbm_get_fields (calibrations,
             permeabilities);
  "advance"  lbm_step, lbm_reduce, lbm_get_fields on a running simulation (a
             long run that is looked at now and then).
Host arrays of more than a few MB are page-locked, as bench.py has them.

Surrogate cases: "layer" is one 3x3x3 convolution layer of the U-Net in
training (forward with ReLU, ReLU adjoint, weight and bias gradients, data
gradient); "unet" is one inference of the whole network.

exact() restates both in 64 bits with plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1711_03254_gb300 import lbm, surrogate, wetting, workloads, ws

T0 = 1.0 / 3.0
STORAGE_BYTES = {"fp64": 8, "fp32": 4, "fp16s": 2, "bf16s": 2}
# share of non-solid cells by geometry, for the work estimates
OPEN_SHARE = {"droplet": 1.0, "porous": 0.40, "rough": 0.97, "channel": 126.0 / 128.0, "slug": 30.0 / 32.0,
              "incline": 0.55}
NU_LOW = 0.0017


def listed():
    return [
        # the smallest call: one 16^3 droplet stepped on its own (surface-tension
        # and Laplace checks step droplets of this kind)
        dict(name="droplet16-fp32", kind="lbm", geometry="droplet", nx=16, ny=16, nz=16, batch=1, precision="fp32",
             mode="restart", updates=200, eq_order=0),
        # the batched viscosity sweep: 16 two-layer channels 4 x 128 x 4
        dict(name="sweep-channels-fp32", kind="lbm", geometry="channel", nx=4, ny=128, nz=4, batch=16,
             precision="fp32", mode="restart", updates=300, eq_order=0),
        # contact-angle calibration: 104 static slugs 128 x 32 relaxed to steady state
        dict(name="slugs-steady-fp32", kind="lbm", geometry="slug", nx=128, ny=32, nz=1, batch=104, precision="fp32",
             mode="steady", updates=400, eq_order=0),
        # double precision, the storage results are checked in: an odd-sized
        # droplet with the full equilibrium
        dict(name="droplet-fp64", kind="lbm", geometry="droplet", nx=67, ny=61, nz=59, batch=1, precision="fp64",
             mode="restart", updates=30, eq_order=1),
        # training data of the learned warm start: 32 droplets on inclined walls
        dict(name="inclines-batch32-fp32", kind="lbm", geometry="incline", nx=64, ny=64, nz=64, batch=32,
             precision="fp32", mode="advance", updates=100, eq_order=0),
        # porous media scanned one geometry after the other, ragged sizes
        dict(name="porous-ragged-fp32", kind="lbm", geometry="porous", nx=183, ny=121, nz=157, batch=1,
             precision="fp32", mode="solve", updates=100, eq_order=0),
        # the headline workload: packed spheres 256^3 in 16-bit storage
        dict(name="porous256-fp16", kind="lbm", geometry="porous", nx=256, ny=256, nz=256, batch=1,
             precision="fp16s", mode="advance", updates=100, eq_order=0),
        # the rough channel of the displacement runs in the other 16-bit storage
        dict(name="rough-channel-bf16", kind="lbm", geometry="rough", nx=256, ny=128, nz=128, batch=1,
             precision="bf16s", mode="advance", updates=100, eq_order=0),
        # the U-Net's finest level, where most of its time goes
        dict(name="layer64-32to32", kind="layer", n=4, d=64, h=64, w=64, ci=32, co=32),
        # a decoder layer on the concatenated tensor one level down
        dict(name="layer32-160to64", kind="layer", n=4, d=32, h=32, w=32, ci=160, co=64),
        # a small ragged volume at the channel counts of the coarse levels
        dict(name="layer-ragged-96to128", kind="layer", n=2, d=14, h=19, w=23, ci=96, co=128),
        # inference: one warm start predicted at 64^3
        dict(name="unet64-predict", kind="unet", n=1, size=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lbm"] * 8 + ["layer"] * 4 + ["unet"])
    if kind == "unet":
        return dict(kind="unet", n=rng.choice([1, 2, 3, 4]), size=rng.choice([32, 40, 48, 56, 64]))
    if kind == "layer":
        s = _log_int(rng, 8, 64)
        d, h, w = (max(6, min(64, s + rng.randint(-5, 5))) for _ in range(3))
        return dict(kind="layer", n=rng.choice([1, 2, 3, 4]), d=d, h=h, w=w, ci=16 * rng.randint(1, 10),
                    co=16 * rng.randint(1, 8))
    g = rng.choice(["droplet", "droplet", "porous", "porous", "rough", "channel", "slug", "incline"])
    prec = rng.choice(["fp32", "fp32", "fp16s", "bf16s", "fp64"])
    if g == "channel":
        return dict(kind="lbm", geometry=g, nx=rng.choice([3, 4, 5, 8]), ny=rng.randint(30, 160),
                    nz=rng.choice([1, 3, 4]), batch=_log_int(rng, 2, 32), precision="fp32", mode="restart",
                    updates=rng.randint(100, 300), eq_order=0)
    if g == "slug":
        return dict(kind="lbm", geometry=g, nx=4 * rng.randint(20, 40), ny=rng.randint(20, 40), nz=1,
                    batch=_log_int(rng, 4, 128), precision="fp32", mode="steady", updates=400, eq_order=0)
    if g == "incline":
        n = 4 * rng.randint(8, 16)
        return dict(kind="lbm", geometry=g, nx=n, ny=n, nz=n, batch=_log_int(rng, 1, 24), precision="fp32",
                    mode="advance", updates=100, eq_order=0)
    lo, hi = (14, 200) if prec != "fp64" else (14, 72)
    if g != "droplet":
        lo = min(48, hi)
    s = _log_int(rng, lo, hi)
    nx, ny, nz = (max(12, s + rng.randint(-s // 6, s // 6)) for _ in range(3))
    if g == "rough":
        nx, ny, nz = max(48, min(nx, 160)), max(40, min(ny, 120)), max(40, min(nz, 120))
    return dict(kind="lbm", geometry=g, nx=nx, ny=ny, nz=nz, batch=1, precision=prec,
                mode=rng.choice(["restart", "solve", "advance"]), updates=50 if prec != "fp64" else 20,
                eq_order=rng.choice([0, 0, 1]) if g == "droplet" else 0)


# ------------------------------------------------------------------ solver inputs

def _stamp(mask, centres, r):
    """Sets mask (bool [nz, ny, nx], periodic) inside spheres of radius r."""
    nz, ny, nx = mask.shape
    k = int(math.ceil(r)) + 1
    off = torch.arange(-k, k + 1, device=mask.device)
    for c in centres.split(256):
        base = c.floor().to(torch.int64)
        frac = c - base
        ax = [(base[:, a, None] + off) % n for a, n in enumerate((nz, ny, nx))]
        d2 = [(off + 0.5 - frac[:, a, None]) ** 2 for a in range(3)]
        inside = d2[0][:, :, None, None] + d2[1][:, None, :, None] + d2[2][:, None, None, :] < r * r
        at = (ax[0][:, :, None, None] * ny + ax[1][:, None, :, None]) * nx + ax[2][:, None, None, :]
        mask.view(-1)[at[inside]] = True


def _porous(case, seed):
    """Overlapping spheres (radius 12, smaller in small boxes) to a porosity of
    0.40 and a minority of 1 % of the pore volume in droplets of radius 4."""
    nz, ny, nx = case["nz"], case["ny"], case["nx"]
    gen = torch.Generator().manual_seed(seed)
    dims = torch.tensor([nz, ny, nx], dtype=torch.float64)
    cells = nz * ny * nx
    r = min(12.0, min(nx, ny, nz) / 6.0)
    solid = torch.zeros((nz, ny, nx), dtype=torch.bool, device="cuda")
    count = max(4, int(-math.log(0.40) * cells / (4.0 / 3.0 * math.pi * r ** 3)))
    _stamp(solid, (torch.rand((count, 3), generator=gen, dtype=torch.float64) * dims).cuda(), r)
    drops = torch.zeros_like(solid)
    few = max(2, int(0.01 * cells / (4.0 / 3.0 * math.pi * 4.0 ** 3)))
    _stamp(drops, (torch.rand((few, 3), generator=gen, dtype=torch.float64) * dims).cuda(), 4.0)
    drops &= ~solid
    t = solid.to(torch.uint8)
    return t, (~solid & ~drops).double(), drops.double(), torch.zeros(solid.shape + (3,), dtype=torch.float64)


def _instances(case, seed):
    """(cell types, rho1, rho2, u) with a leading instance axis as CPU or GPU
    tensors, and the instances' parameters."""
    rng = np.random.default_rng(seed)
    nx, ny, nz, B = case["nx"], case["ny"], case["nz"], case["batch"]
    g = case["geometry"]
    if g == "porous":
        one = _porous(case, seed)
        p = dict(tau=(1.0 / T0 + 0.5, 0.01 / T0 + 0.5), G=-2.2, g=(1e-6, 0.0, 0.0))
        return [x[None] for x in one], [p]
    rows, params = [], []
    for b in range(B):
        if g == "droplet":
            c = tuple(n / 2.0 + rng.uniform(-2.0, 2.0) for n in (nx, ny, nz))
            rows.append(workloads.droplet(nx, ny, nz, min(nx, ny, nz) * rng.uniform(0.22, 0.30), center=c))
            params.append(dict(tau=(1.0, 1.0), G=-2.2))
        elif g == "rough":
            rows.append(workloads.rough_channel(nx, ny, nz, seed=seed, invaded_length=32, ends="periodic"))
            params.append(dict(tau=(1.7 / T0 + 0.5, NU_LOW / T0 + 0.5), G=-2.2, rho_s=0.2, g=(1e-5, 0.0, 0.0)))
        elif g == "channel":
            ratio = 10.0 ** rng.uniform(0.0, 3.0)
            nu = (NU_LOW, NU_LOW * ratio) if rng.random() < 0.5 else (NU_LOW * ratio, NU_LOW)
            rows.append(workloads.layered_channel(nx, ny, nz, layout=("121", "12")[b % 2], wall_comp_nu=nu[0],
                                                  core_comp_nu=nu[1], g=4e-8))
            params.append(dict(tau=(nu[0] / T0 + 0.5, nu[1] / T0 + 0.5), G=-1.8, g=(4e-8, 0.0, 0.0)))
        elif g == "slug":
            rows.append(wetting.slug_channel(nx, ny))
            nu = 10.0 ** rng.uniform(-1.5, -0.5, size=2)
            params.append(dict(tau=(nu[0] / T0 + 0.5, nu[1] / T0 + 0.5), G=-2.2, rho_s=rng.uniform(-0.4, 0.4)))
        elif g == "incline":
            th = rng.uniform(0.0, 45.0)
            rows.append(workloads.inclined_droplet(nx, th, R=nx / 8.0))
            nu = 1.7 / 10.0 ** rng.uniform(0.0, 2.0)
            gn = rng.uniform(0.0, 1e-4)
            params.append(dict(tau=(1.7 / T0 + 0.5, nu / T0 + 0.5), G=-1.8, rho_s=rng.uniform(-0.3, 0.3),
                               g=(gn * math.sin(math.radians(th)), -gn * math.cos(math.radians(th)), 0.0)))
        else:
            raise ValueError(g)
    return [torch.from_numpy(np.stack([r[k] for r in rows])) for k in range(4)], params


def _host(x):
    """x as a NumPy array on the host, page-locked when it is large."""
    x = x.contiguous()
    if x.numel() * x.element_size() < (4 << 20):
        return x.cpu().numpy()
    h = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
    h.copy_(x)
    return h.numpy()


def _prepare_lbm(case, seed):
    (t, r1, r2, u), params = _instances(case, seed)
    sim = lbm.Sim(case["nx"], case["ny"], case["nz"], params, precision=case["precision"],
                  eq_order=case["eq_order"])
    s = dict(case=case, sim=sim, t=_host(t), fields=[_host(x) for x in (r1, r2, u)])
    s["out"] = [_host(torch.zeros(x.shape, dtype=torch.float64)) for x in (r1, r2, u)]
    sim.set_geometry(s["t"])
    if case["mode"] == "advance":
        sim.set_fields(*s["fields"])
        s["fields"] = None
    return s


def _run_lbm(s):
    case, sim = s["case"], s["sim"]
    if case["mode"] == "solve":
        sim.set_geometry(s["t"])
    if case["mode"] != "advance":
        sim.set_fields(*s["fields"])
    got = []
    if case["mode"] == "steady":
        done, res = lbm.lbm_run_to_steady(sim.ctx, case["updates"] // 4, 1e-9, case["updates"], case["batch"])
        got = [done, res]
    else:
        sim.step(case["updates"])
        if case["mode"] == "advance":
            got = [sim.reduce(allow_diverged=True)]
    lbm.lbm_get_fields(sim.ctx, *s["out"])
    return got + s["out"]


# ------------------------------------------------------------------ surrogate inputs

def _prepare_layer(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, d, h, w, ci, co = (case[k] for k in ("n", "d", "h", "w", "ci", "co"))

    def rand(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    bf = dict(dtype=torch.bfloat16, device="cuda")
    weight = (rand(co, 3, 3, 3, ci) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16)
    return dict(case=case, x=rand(n, d, h, w, ci).clamp_(min=0.0).to(torch.bfloat16), w=weight,
                b=rand(co) * 0.1, dy=(rand(n, d, h, w, co) * 1e-3).to(torch.bfloat16),
                y=torch.empty((n, d, h, w, co), **bf), dx=torch.empty((n, d, h, w, ci), **bf),
                wf=torch.empty((ci, 3, 3, 3, co), **bf), dw=torch.zeros((co, 3, 3, 3, ci), device="cuda"),
                db=torch.zeros(co, device="cuda"))


def _run_layer(s):
    ws.ws_conv3d_fwd(s["x"], s["w"], s["b"], s["y"], True)
    ws.ws_relu_bwd(s["y"], s["dy"])
    s["dw"].zero_()
    s["db"].zero_()
    ws.ws_conv3d_bwd_weight(s["x"], s["dy"], s["dw"], s["db"], 3)
    ws.ws_conv3d_flip_weights(s["w"], s["wf"])
    ws.ws_conv3d_fwd(s["dy"], s["wf"], None, s["dx"], False)
    return [s["y"], s["dw"], s["db"], s["dx"]]


def _unet_input(case, seed):
    rng = np.random.default_rng(seed)
    x = []
    for _ in range(case["n"]):
        th = rng.uniform(0.0, 45.0)
        t, _, r2, _ = workloads.inclined_droplet(case["size"], th, R=case["size"] / 8.0)
        x.append(surrogate.encode_inputs(t, rng.uniform(30.0, 150.0), 10.0 ** rng.uniform(0.0, 3.0), th,
                                         rng.uniform(0.0, 1e-4), r2))
    return torch.from_numpy(np.stack(x)).cuda()


def _prepare_unet(case, seed):
    net = surrogate.UNet3D(case["n"], case["size"], seed=seed)
    return dict(case=case, net=net, x=_unet_input(case, seed))


# ------------------------------------------------------------------ entry points

def prepare(case, seed):
    return {"lbm": _prepare_lbm, "layer": _prepare_layer, "unet": _prepare_unet}[case["kind"]](case, seed)


def run(state):
    kind = state["case"]["kind"]
    if kind == "lbm":
        return _run_lbm(state)
    if kind == "layer":
        return _run_layer(state)
    return state["net"].forward(state["x"])


def work(case):
    if case["kind"] == "lbm":
        cells = case["nx"] * case["ny"] * case["nz"] * case["batch"]
        open_cells = OPEN_SHARE[case["geometry"]] * cells
        # f read once and written once per update (38 values each way), the cell's
        # type, and the FP64 fields in and out of the call
        per_update = 76 * STORAGE_BYTES[case["precision"]] + 1
        fields = 40 if case["mode"] == "advance" else 80
        return dict(bytes=case["updates"] * open_cells * per_update + fields * cells,
                    flops=case["updates"] * open_cells * 900)
    if case["kind"] == "layer":
        pos, ci, co = case["n"] * case["d"] * case["h"] * case["w"], case["ci"], case["co"]
        return dict(bytes=2 * pos * (2 * ci + 2 * co) + 27 * ci * co * 6, flops=3 * 2 * 27 * pos * ci * co)
    c = (16,) + surrogate.LEVELS
    pos, flops = case["n"] * case["size"] ** 3, 0.0
    pairs = [(0, c[0], c[1]), (0, c[1], c[1]), (1, c[1], c[2]), (1, c[2], c[2]), (2, c[2], c[3]), (2, c[3], c[3]),
             (3, c[3], c[4]), (3, c[4], c[4]), (2, c[4] + c[3], c[3]), (2, c[3], c[3]), (1, c[3] + c[2], c[2]),
             (1, c[2], c[2]), (0, c[2] + c[1], c[1]), (0, c[1], c[1])]
    weights = 0
    for level, ci, co in pairs:
        flops += 2.0 * 27 * ci * co * pos / 8 ** level
        weights += 27 * ci * co
    return dict(bytes=pos * (16 * 4 + 16 * 4) + 2 * weights, flops=flops + 2.0 * pos * 32 * 16)


# ------------------------------------------------------------------ 64-bit restatement

_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
      (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
      (0, -1, 1)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12


def _opp(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


def _at(x, i, sign):
    """x at the position sign * c_i away (last three axes z, y, x; periodic)."""
    cx, cy, cz = _C[i]
    return torch.roll(x, (-sign * cz, -sign * cy, -sign * cx), (-3, -2, -1))


def _dot(i, v):
    r = None
    for a in range(3):
        if _C[i][a]:
            r = v[a] * _C[i][a] if r is None else r + v[a] * _C[i][a]
    return r


def _equilibrium(i, rho, u, uu, eq_order):
    if i == 0:
        e = torch.ones_like(uu)
    else:
        cu = _dot(i, u)
        e = 1.0 + cu * (3.0 + 4.5 * cu * cu - 4.5 * uu)
        if eq_order:
            e = e + 4.5 * cu * cu
    if eq_order:
        e = e - 1.5 * uu
    return _W[i] * rho * e


class _Exact:
    """The update of Sec. 2 in 64 bits (walls read as model 2) on [B, z, y, x]."""

    def __init__(self, t, r1, r2, u, params, eq_order):
        dev = r1.device
        self.eq = eq_order
        self.solid = t.to(dev) == 1
        self.fluid = ~self.solid
        self.to_solid = [_at(self.solid, i, 1) for i in range(19)]

        def per(f):
            return torch.tensor([f(p) for p in params], dtype=torch.float64, device=dev).view(-1, 1, 1, 1)

        self.nu = [per(lambda p, a=a: T0 * (p["tau"][a] - 0.5)) for a in range(2)]
        self.G = per(lambda p: p["G"])
        self.rs = [per(lambda p: max(-p.get("rho_s", 0.0), 0.0)), per(lambda p: max(p.get("rho_s", 0.0), 0.0))]
        self.g = [per(lambda p, a=a: p.get("g", (0.0, 0.0, 0.0))[a]) for a in range(3)]
        self.wall = [sum(2.0 * _W[i] * _C[i][a] * self.to_solid[i].double() for i in range(1, 19) if _C[i][a])
                     for a in range(3)]
        vel = [u[..., a] for a in range(3)]
        uu = vel[0] ** 2 + vel[1] ** 2 + vel[2] ** 2
        self.f = [torch.stack([_equilibrium(i, r, vel, uu, eq_order) for i in range(19)]) for r in (r1, r2)]
        self.rho, self.u = [r1, r2], vel

    def step(self):
        rho, mom, rd, pi = [], [], [], []
        for f in self.f:
            fs = torch.empty_like(f)
            for i in range(19):
                torch.where(self.to_solid[_opp(i)], f[_opp(i)], _at(f[i], i, -1), out=fs[i])
            r = fs.sum(0) * self.fluid
            rho.append(r)
            mom.append([sum(fs[i] * _C[i][a] for i in range(1, 19) if _C[i][a]) for a in range(3)])
            pi.append({(a, b): sum(fs[i] * (_C[i][a] * _C[i][b]) for i in range(1, 19) if _C[i][a] * _C[i][b])
                       for a in range(3) for b in range(a, 3)})
            del fs
        force = []
        for al in range(2):
            psi = rho[1 - al]
            s = [self.wall[a] * self.rs[1 - al] for a in range(3)]
            for i in range(1, 19):
                q = torch.where(self.to_solid[i], psi, _at(psi, i, 1))
                for a in range(3):
                    if _C[i][a]:
                        s[a] = s[a] + q * (2.0 * _W[i] * _C[i][a])
            force.append([rho[al] * (self.G * s[a] + self.g[a]) for a in range(3)])
        total = torch.where(self.fluid, rho[0] + rho[1], 1.0)
        u = [(mom[0][a] + mom[1][a] + 0.5 * (force[0][a] + force[1][a])) / total * self.fluid for a in range(3)]
        share = (rho[0] / total).clamp(0.0, 1.0)
        itau = 1.0 / ((share * self.nu[0] + (1.0 - share) * self.nu[1]) / T0 + 0.5)
        omega, half = 1.0 - itau, 1.0 - 0.5 * itau
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        for al in range(2):
            A = {}
            for (a, b), m in pi[al].items():
                m = m - rho[al] * T0 if a == b else m
                if self.eq:
                    m = m - rho[al] * u[a] * u[b]
                A[a, b] = omega * m + half * (u[a] * force[al][b] + u[b] * force[al][a])
            tr = A[0, 0] + A[1, 1] + A[2, 2]
            for i in range(19):
                e = -1.5 * tr
                for (a, b), m in A.items():
                    k = _C[i][a] * _C[i][b]
                    if k:
                        e = e + m * (4.5 * k * (1 if a == b else 2))
                if i:
                    e = e + 1.5 * _dot(i, force[al])
                self.f[al][i] = (_equilibrium(i, rho[al], u, uu, self.eq) + _W[i] * e) * self.fluid
        self.rho, self.u = rho, u


def _exact_lbm(case, seed):
    cells = case["nx"] * case["ny"] * case["nz"] * case["batch"]
    if cells * case["updates"] > 2e9:
        return None  # too long in plain torch
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    fields, params = _instances(case, seed)
    t, r1, r2, u = (x.to(dev) for x in fields)
    e = _Exact(t, r1, r2, u, params, case["eq_order"])
    chunk = case["updates"] // 4 if case["mode"] == "steady" else case["updates"]
    u0 = e.u
    for k in range(case["updates"]):
        if k and k % chunk == 0:
            u0 = e.u
        e.step()
    vel = torch.stack(e.u, -1)
    dims = (1, 2, 3, 4)
    du = ((vel - torch.stack(u0, -1)) ** 2).sum(dims).sqrt()
    res = du / (chunk * (vel ** 2).sum(dims).sqrt() + 1e-30)
    out = [e.rho[0], e.rho[1], vel]
    if case["mode"] == "steady":
        return [case["updates"], res] + out
    if case["mode"] == "advance":
        rho = e.rho[0] + e.rho[1]
        sums = [r.sum((1, 2, 3)) for r in e.rho] + [(rho * v).sum((1, 2, 3)) for v in e.u]
        speed = (vel ** 2).sum(-1).amax((1, 2, 3)).sqrt()
        return [torch.stack(sums + [res, speed], -1)] + out
    return out


def _shifted(x, dz, dy, dx):
    """x[n, z + dz, y + dy, x + dx, c], zero outside."""
    n, d, h, w, c = x.shape
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    return p[:, 1 + dz:1 + dz + d, 1 + dy:1 + dy + h, 1 + dx:1 + dx + w].reshape(-1, c)


_TAPS = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _conv(x, w, b=None):
    """x [n, d, h, w, ci], w [co, 27, ci], in 64 bits."""
    y = sum(_shifted(x, *t) @ w[:, k].T for k, t in enumerate(_TAPS))
    y = y.view(x.shape[:4] + (w.shape[0],))
    return y if b is None else y + b


def _exact_layer(case, seed):
    s = {k: v.double() for k, v in _prepare_layer(case, seed).items() if k != "case"}
    w = s["w"].view(case["co"], 27, case["ci"])
    y = _conv(s["x"], w, s["b"]).clamp(min=0.0)
    dy = torch.where(y > 0.0, s["dy"], 0.0)
    rows = dy.reshape(-1, case["co"])
    dw = torch.stack([rows.T @ _shifted(s["x"], *t) for t in _TAPS], 1)
    dx = _conv(dy, w.flip(1).permute(2, 1, 0).contiguous())
    return [y, dw.view(s["w"].shape), rows.sum(0), dx]


def _exact_unet(case, seed):
    s = _prepare_unet(case, seed)
    net, x = s["net"], s["x"].double()
    p = {k: (d["wb"].double().view(d["co"], -1, d["ci"]), d["b"].double()) for k, d in net.p.items()}

    def block(name, v):
        for half in "ab":
            v = _conv(v, *p[name + half]).clamp(min=0.0)
        return v

    def pool(v):
        n, d, h, w, c = v.shape
        return v.view(n, d // 2, 2, h // 2, 2, w // 2, 2, c).mean((2, 4, 6))

    def up(v):
        return v.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    e0 = block("enc0", x)
    e1 = block("enc1", pool(e0))
    e2 = block("enc2", pool(e1))
    v = block("bot", pool(e2))
    for name, skip in (("dec2", e2), ("dec1", e1), ("dec0", e0)):
        v = block(name, torch.cat([up(v), skip], -1))
    w, b = p["head"]
    return v @ w[:, 0].T + b


def exact(case, seed):
    return {"lbm": _exact_lbm, "layer": _exact_layer, "unet": _exact_unet}[case["kind"]](case, seed)
