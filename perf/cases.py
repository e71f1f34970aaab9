"""Workloads of the lattice Boltzmann library, as programs run them: one pass is one whole
request -- set the initial fields, advance a number of steps, read the moments back.

Each case is a dict of plain values; prepare() builds what a program holds before the call
(input fields, lattices, output buffers, the tuned launch shape where programs tune),
run() makes one pass through the public entry points, exact() computes the same pass in
plain FP64 torch operations.  Fields come back in the precision of the lattice.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_05197_gb300 import lbm, tune

PRECISIONS = {"fp64": lbm.FP64, "fp32": lbm.FP32, "fp16": lbm.FP16, "bf16": lbm.BF16}
DTYPES = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
MODELS = {"cg": lbm.CG, "sc": lbm.SC_MP, "sc2c": lbm.SC_2C, "mr": lbm.SC_MR}
# Shan-Chen multiphase coexistence densities at G = -5
LIQUID, GAS = 1.8884, 0.1194


def _case(name, kind, model, precision, nx, ny, nz, steps, reads=1, tuned=True, inplace=False, count=1):
    return dict(name=name, kind=kind, model=model, precision=precision, nx=nx, ny=ny, nz=nz, steps=steps, reads=reads,
                tuned=tuned, inplace=inplace, count=count)


def listed():
    return [
        # static droplet on a 2D lattice in FP64, the Laplace-law check: the smallest lattice,
        # where a step is one short launch
        _case("laplace_2d_fp64", "drop", "cg", "fp64", 128, 128, 1, 100, tuned=False),
        # a stability-map request on the 2D grid of the parameter sweep
        _case("sweep_2d_sc_fp32", "drop", "sc", "fp32", 256, 256, 1, 100),
        # a stability-map request on the sweep's smallest 3D grid, stepped alone
        _case("sweep_32_cg_fp32", "drop", "cg", "fp32", 32, 32, 32, 100),
        # the oscillating droplet, the benchmark workload, with either model
        _case("droplet_cg_fp32", "drop", "cg", "fp32", 128, 128, 128, 20),
        _case("droplet_sc_fp32", "drop", "sc", "fp32", 128, 128, 128, 20),
        # the Rayleigh-Plateau jet: 16-bit storage with the colour-gradient model, FP32 with
        # the two-component Shan-Chen model
        _case("jet_cg_fp16", "jet", "cg", "fp16", 64, 64, 512, 20),
        _case("jet_sc2c_fp32", "jet", "sc2c", "fp32", 64, 64, 512, 20),
        # dense emulsion with the repulsion force, FP16 storage: the largest lattice
        _case("emulsion_cg_fp16", "emulsion", "cg", "fp16", 256, 256, 256, 6),
        # head-on collision of two drops with the multirange Shan-Chen model, fields read
        # every 10 steps to follow the gap
        _case("collision_mr_fp32", "collision", "mr", "fp32", 128, 64, 64, 10, reads=2, tuned=False),
        # the droplet with in-place streaming, which programs choose to halve the memory
        _case("droplet_cg_inplace", "drop", "cg", "fp32", 128, 128, 128, 20, tuned=False, inplace=True),
        # two-phase channel flow between walls under a body force, a size with no alignment
        # at all, profile read every 10 steps
        _case("channel_cg_fp32", "channel", "cg", "fp32", 101, 75, 67, 10, reads=4),
        # one tick of the serving loop: 12 small lattices of the sweep advancing together in
        # the batched launch, FP16 storage
        _case("serving_batch_fp16", "drop", "mix", "fp16", 32, 32, 32, 100, count=12),
    ]


def _size(rng, lo, hi, aligned):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if aligned:
        step = 32 if v >= 48 else 16
        v = max(step, min(hi // step * step, (v + step // 2) // step * step))
    return max(lo, min(hi, v))


def draw(rng):
    """Sizes over the listed ranges: half of the lattices have round sizes, as programs
    mostly choose them, half have any."""
    aligned = rng.random() < 0.5
    pick = rng.random()
    if pick < 0.2:  # 2D droplet
        nx, ny = (_size(rng, 96, 768, aligned) for _ in range(2))
        return _strip(_case("", "drop", rng.choice(["cg", "sc"]), rng.choice(["fp64", "fp32", "fp32", "fp16"]), nx, ny, 1,
                            rng.choice([50, 100]), tuned=rng.random() < 0.5))
    if pick < 0.5:  # 3D droplet
        nx, ny, nz = (_size(rng, 28, 160, aligned) for _ in range(3))
        return _strip(_case("", "drop", rng.choice(["cg", "sc"]), rng.choice(["fp32", "fp32", "fp16", "bf16"]), nx, ny, nz,
                            20, tuned=rng.random() < 0.7, inplace=rng.random() < 0.2))
    if pick < 0.65:  # jet along z
        nx = _size(rng, 40, 96, aligned)
        return _strip(_case("", "jet", rng.choice(["cg", "sc", "sc2c"]), rng.choice(["fp32", "fp16", "bf16"]), nx,
                            nx, _size(rng, 128, 512, aligned), 20))
    if pick < 0.73:
        n = _size(rng, 96, 192, aligned)
        return _strip(_case("", "emulsion", "cg", "fp16", n, n, n, rng.choice([4, 6])))
    if pick < 0.81:
        return _strip(_case("", "collision", "mr", "fp32", _size(rng, 80, 160, aligned), _size(rng, 48, 80, aligned),
                            _size(rng, 48, 80, aligned), 10, reads=rng.choice([1, 2]), tuned=False))
    if pick < 0.91:
        nx, ny, nz = (_size(rng, 32, 128, aligned) for _ in range(3))
        return _strip(_case("", "channel", rng.choice(["cg", "sc2c"]), rng.choice(["fp32", "fp16"]), nx, ny, nz, 10,
                            reads=rng.choice([1, 4])))
    n = _size(rng, 24, 40, aligned)
    return _strip(_case("", "drop", "mix", rng.choice(["fp32", "fp16"]), n, n, n, rng.choice([20, 50, 100]),
                        count=rng.randint(4, 16)))


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


# ---- what the lattices of a case are: parameters and initial fields ------------------

def _members(case):
    """(model, nx, ny, nz) of every lattice of a case; a mix takes the sweep's small grids."""
    if case["model"] != "mix":
        return [(case["model"], case["nx"], case["ny"], case["nz"])]
    grids = [(256, 256, 1), (case["nx"], case["ny"], case["nz"]), (48, 48, 48)]
    return [(("cg", "sc")[i % 2],) + grids[(i // 2) % 3] for i in range(case["count"])]


def _physics(case, model):
    """Model parameters (lbm.Params fields besides lattice, model, precision and size)."""
    kind = case["kind"]
    if model == "cg":
        p = dict(rho_r0=1.0, rho_b0=0.1, tau_r=1.0, tau_b=1.0, A=5e-3)
        if kind == "jet" or case["precision"] == "fp64":  # equal densities, as in the Laplace-law check
            p.update(rho_b0=1.0, A=1e-2)
        if kind == "emulsion":
            p = dict(rho_r0=1.36, rho_b0=1.36, tau_r=1.0, tau_b=1.0, A=0.0518, rep_pi=0.012, rep_chi=2.0, grad_eps=1e-4)
        if kind == "channel":
            p = dict(rho_r0=1.0, rho_b0=0.5, tau_r=0.9, tau_b=0.6, A=4e-3, body_force=(1e-5, 0.0, 2e-6))
        return p
    if model == "sc":
        return dict(G=-5.0, rho0_psi=1.0, tau_r=1.0)
    if model == "sc2c":
        p = dict(G=0.9, rho0_psi=0.577, tau_r=1.0, tau_b=0.8)
        if kind == "channel":
            p["body_force"] = (1e-5, 0.0, 2e-6)
        return p
    return dict(Ga=(-9.0, -8.0), Gr=(8.1, 7.1), G=1.215, rho0_psi=0.83, tau_r=1.0, tau_b=1.0)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _fields(case, member, seed):
    """Initial densities (and velocity, wall mask) of one lattice as flat FP64 tensors:
    sharp interfaces with +-1% noise, the geometry moved a little by the seed."""
    model, nx, ny, nz = member
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    r = np.random.default_rng(seed)
    z, y, x = torch.meshgrid(*(torch.arange(n, dtype=torch.float64, device=dev) for n in (nz, ny, nx)), indexing="ij")
    c = [(n - 1) / 2 + float(r.uniform(-1, 1)) for n in (nx, ny, nz)]
    kind = case["kind"]
    u = solid = None
    if kind == "jet":
        waves = max(1, round(nz / 90.0))
        radius = 0.16 * nx + torch.cos(2 * math.pi * (waves * z / nz + float(r.uniform())))
        inside = (x - c[0]) ** 2 + (y - c[1]) ** 2 <= radius ** 2
        u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=dev)
        u[2] = 0.05 * inside.double()  # moving along its axis
    elif kind == "emulsion":
        inside = torch.zeros((nz, ny, nx), dtype=torch.bool, device=dev)
        placed = np.zeros((0, 4))
        want, tries = int(200 * nx * ny * nz / 256 ** 3), 0
        while len(placed) < want and tries < 100000:
            tries += 1
            s = np.append(r.uniform(0, 1, 3) * (nx, ny, nz), r.uniform(8, 12))
            d = np.abs(placed[:, :3] - s[:3])
            d = np.minimum(d, np.array([nx, ny, nz]) - d)
            if np.all(np.sqrt((d * d).sum(1)) >= placed[:, 3] + s[3] + 3.0):
                placed = np.vstack([placed, s])
        for px, py, pz, pr in placed:
            ax = [torch.arange(math.floor(v - pr), math.ceil(v + pr) + 1, device=dev) for v in (px, py, pz)]
            bz, by, bx = torch.meshgrid(ax[2] - pz, ax[1] - py, ax[0] - px, indexing="ij")
            iz, iy, ix = torch.meshgrid(ax[2] % nz, ax[1] % ny, ax[0] % nx, indexing="ij")
            box = bx * bx + by * by + bz * bz <= pr * pr
            inside[iz[box], iy[box], ix[box]] = True
        u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=dev)
        u[0] = 0.06 * torch.sin(2 * math.pi * y / ny)  # sheared
    elif kind == "collision":
        rad = 14.0 / 64.0 * min(nx, ny, nz)
        d1 = (x - c[0] + 1.15 * rad) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= rad ** 2
        d2 = (x - c[0] - 1.15 * rad) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2 <= rad ** 2
        inside = d1 | d2
        u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=dev)
        u[0] = 0.06 * d1.double() - 0.06 * d2.double()
    elif kind == "channel":
        solid = ((y == 0) | (y == ny - 1)).to(torch.uint8)
        inside = (y - c[1]).abs() < ny / 4 + 1.5 * torch.cos(2 * math.pi * x / nx)
    else:
        semi = (24 / 128 * nx, 20 / 128 * ny, 20 / 128 * nz)
        inside = ((x - c[0]) / semi[0]) ** 2 + ((y - c[1]) / semi[1]) ** 2 <= 1 if nz == 1 else \
            ((x - c[0]) / semi[0]) ** 2 + ((y - c[1]) / semi[1]) ** 2 + ((z - c[2]) / semi[2]) ** 2 <= 1

    def noisy(a):
        return a * (1 + 0.01 * (2 * torch.rand(a.shape, generator=g, dtype=torch.float64, device=dev) - 1))

    ins = inside.double()
    p = _physics(case, model)
    if model == "cg":
        rr, rb = noisy(p["rho_r0"] * ins), noisy(p["rho_b0"] * (1 - ins))
    elif model == "sc":
        rr, rb = noisy(LIQUID * ins + GAS * (1 - ins)), None
    elif model == "sc2c":
        rr, rb = noisy(ins + 0.03), noisy(1.03 - ins)
    else:
        rr, rb = noisy(1.18 * ins + 0.18 * (1 - ins)), noisy(0.18 * ins + 1.18 * (1 - ins))
    if solid is not None:
        fluid = 1 - solid.double()
        rr, rb = rr * fluid, rb * fluid
    flat = lambda a: None if a is None else a.reshape(-1).contiguous()  # noqa: E731
    return dict(rho_r=flat(rr), rho_b=flat(rb), u=None if u is None else u.reshape(3, -1).contiguous(), solid=flat(solid))


# ---- the pass ------------------------------------------------------------------------

def prepare(case, seed):
    precision = PRECISIONS[case["precision"]]
    lats, fields, reads = [], [], []
    for m, member in enumerate(_members(case)):
        model, nx, ny, nz = member
        p = lbm.Params(lattice=lbm.D3Q19 if nz > 1 else lbm.D2Q9, model=MODELS[model], precision=precision, nx=nx, ny=ny,
                       nz=nz, streaming=lbm.STREAM_AA if case["inplace"] else lbm.STREAM_AB, **_physics(case, model))
        lat = lbm.Lattice(p)
        f = _fields(case, member, seed * 64 + m)
        lat.init(**f)
        if case["model"] == "mix":
            lat.set_tiling(32, 8, tune.batch_chunk(p))  # as the serving loop prepares a job
        elif case["tuned"]:
            tune.autotune(lat)
        out = [torch.empty(p.n, dtype=torch.float64, device=lat.device), None,
               torch.empty(3, p.n, dtype=torch.float64, device=lat.device)]
        if p.ncomp == 2:
            out[1] = torch.empty_like(out[0])
        lats.append(lat)
        fields.append(f)
        reads.append(out)
    batch = None
    if case["model"] == "mix":
        batch = lbm.Batch(precision, 64, 1 << 14, stream=lats[0].stream)
    torch.cuda.synchronize()
    return dict(case=case, lats=lats, fields=fields, reads=reads, batch=batch, dtype=DTYPES[case["precision"]])


def run(state):
    case, lats, batch = state["case"], state["lats"], state["batch"]
    for lat, f in zip(lats, state["fields"]):
        lat.init(**f)
    if batch is not None:
        batch.set(lats, [case["steps"]] * len(lats))
        batch.step(case["steps"])
        return [_read(lat, out, state["dtype"]) for lat, out in zip(lats, state["reads"])]
    got = []
    for _ in range(case["reads"]):
        lats[0].step(case["steps"])
        got.append(_read(lats[0], state["reads"][0], state["dtype"]))
    return got


def _read(lat, out, dtype):
    """Densities and velocity of the current state, kept in the lattice's precision."""
    lat.moments_into(*out)
    return [None if a is None else a.to(dtype, copy=True) for a in out]


# ---- the work ------------------------------------------------------------------------

def work(case):
    """Every step reads and writes each population once; the initial fields are read once
    and the returned fields written once.  Operations per node of a step: the moments,
    stencils and collision of the models' equations."""
    elt = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["precision"]]
    total, flops = 0.0, 0.0
    for model, nx, ny, nz in _members(case):
        n, k, q = nx * ny * nz, 1 if model == "sc" else 2, 19 if nz > 1 else 9
        steps = case["steps"] * case["reads"]
        total += n * (steps * 2 * k * q * elt + 8 * k + case["reads"] * (k + 3) * elt)
        total += n * (24 * (case["kind"] in ("jet", "emulsion", "collision")) + (case["kind"] == "channel"))
        per = {"cg": 700, "sc": 370, "sc2c": 680, "mr": 1250}[model] * q / 19 + 250 * (case["kind"] == "emulsion")
        flops += n * steps * per
    return {"bytes": total, "flops": flops}


# ---- the same pass in FP64 -----------------------------------------------------------

_D3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
       (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_D2 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
# per |c|^2: weights w, perturbation B, enhanced-equilibrium psi and xi, share of 1 - alpha
_G3 = dict(w=(1 / 3, 1 / 18, 1 / 36), B=(-2 / 9, 1 / 54, 1 / 27), psi=(-5 / 2, -1 / 6, 1 / 24), xi=(0, 1 / 4, 1 / 8),
           phi=(0, 1 / 12, 1 / 24))
_G2 = dict(w=(4 / 9, 1 / 9, 1 / 36), B=(-4 / 27, 2 / 27, 5 / 108), psi=(-8 / 3, -1 / 6, 1 / 12), xi=(0, 1 / 2, 1 / 8),
           phi=(0, 1 / 5, 1 / 20))
_BELT = {1: 4 / 135, 2: 1 / 63, 3: 2 / 315, 4: 5 / 1512, 5: 1 / 945, 6: 1 / 1890, 8: 1 / 15120}


class _Exact:
    """One lattice in FP64: populations f[k][i] shaped (nz, ny, nx)."""

    def __init__(self, model, p, shape, rho_r, rho_b, u, solid):
        self.model, self.p = model, p
        self.cs, g = (_D2, _G2) if shape[0] == 1 else (_D3, _G3)
        self.r2 = [sum(a * a for a in c) for c in self.cs]
        self.w, self.B, self.ps, self.xi = ([g[n][r] for r in self.r2] for n in ("w", "B", "psi", "xi"))
        self.solid = None if solid is None else solid.reshape(shape) != 0
        self.rho = [a.reshape(shape) for a in (rho_r, rho_b) if a is not None][:1 if model == "sc" else 2]
        if model == "cg":
            al = [1 - 0.8 * p["rho_b0"] / p["rho_r0"], 0.2]
            self.phi = [[a if r == 0 else g["phi"][r] * (1 - a) for r in self.r2] for a in al]
        vel = [torch.zeros_like(self.rho[0])] * 3 if u is None else [a.reshape(shape) for a in u]
        self.f = []
        for k, rho in enumerate(self.rho):
            eq = self.equilibrium(k, vel, self.gradient(rho) if model == "cg" else None)
            self.f.append([self.fluid(eq(i)) for i in range(len(self.cs))])

    def fluid(self, a):
        return a if self.solid is None else torch.where(self.solid, 0.0, a)

    def at(self, a, c):
        """a(x + c), a wall neighbour replaced by the centre."""
        s = (-c[2], -c[1], -c[0])
        v = torch.roll(a, s, (0, 1, 2))
        return v if self.solid is None else torch.where(torch.roll(self.solid, s, (0, 1, 2)), a, v)

    @staticmethod
    def dot(c, v):
        t = [x if s > 0 else -x for s, x in zip(c, v) if s]
        return sum(t[1:], t[0]) if t else torch.zeros_like(v[0])

    def gradient(self, a, weights=None, cs=None):
        """sum_j w_j a(x + c_j) c_j over the lattice (3 w: the isotropic gradient) or a belt."""
        cs = cs or self.cs
        weights = weights or [3 * w for w in self.w]
        out = [torch.zeros_like(a) for _ in range(3)]
        for c, w in zip(cs, weights):
            if c > (0, 0, 0):
                d = w * (self.at(a, c) - self.at(a, tuple(-s for s in c)))
                for o, s in zip(out, c):
                    if s:
                        o += s * d
        return out

    def nu(self):
        p = self.p
        rr, rb = self.rho
        return (rr + rb) / (rr * 3 / (p["tau_r"] - 0.5) + rb * 3 / (p["tau_b"] - 0.5))

    def equilibrium(self, k, u, grad):
        rho, uu = self.rho[k], sum(a * a for a in u)
        if grad is not None:
            nu, ug = self.nu(), sum(a * b for a, b in zip(u, grad))

        def eq(i):
            cu = self.dot(self.cs[i], u)
            v = rho * self.w[i] * (3 * cu + 4.5 * cu * cu - 1.5 * uu)
            if grad is None:
                return v + rho * self.w[i]
            return v + rho * self.phi[k][i] + nu * (self.ps[i] * ug + 2 * self.xi[i] * cu * self.dot(self.cs[i], grad))

        return eq

    def forces(self):
        """Force on each component (colour gradient: on the total)."""
        p, rho = self.p, self.rho
        body = p.get("body_force", (0.0, 0.0, 0.0))
        if self.model == "cg":
            rr, rb = rho
            self.colour = (rr - rb) / (rr + rb)
            if self.solid is not None:
                self.colour = torch.where(self.solid, 0.0, self.colour)
            self.gn = self.gradient(self.colour)
            self.gabs = torch.sqrt(sum(a * a for a in self.gn))
            self.has = self.gabs > p.get("grad_eps", 0.0)
            F = [torch.full_like(rr, b) for b in body]
            if p.get("rep_pi"):
                n = [torch.where(self.has, a / self.gabs, 0.0) for a in self.gn]
                acc = [torch.zeros_like(rr) for _ in range(3)]
                for c, r2 in zip(self.cs[1:], self.r2[1:]):
                    m = [torch.roll(a, (-c[2], -c[1], -c[0]), (0, 1, 2)) for a in n]
                    nc, mc = self.dot(c, n), self.dot(c, m)
                    on = (nc * mc < 0).double() / math.sqrt(r2)
                    for a in range(3):
                        acc[a] += on * (nc * n[a] + mc * m[a])
                s = p["rep_pi"] * (1 - self.colour.abs()) ** p["rep_chi"]
                F = [a - s * b for a, b in zip(F, acc)]
            return [F]
        psi = [p["rho0_psi"] * (1 - torch.exp(-a / p["rho0_psi"])) for a in rho]
        if self.model == "sc":
            return [[b - p["G"] * psi[0] * a for a, b in zip(self.gradient(psi[0], self.w), body)]]
        G, out = p["G"] / p["rho0_psi"] ** 2, []
        total = rho[0] + rho[1]
        for s in range(2):
            cross = self.gradient(rho[1 - s], self.w)
            F = [-G * rho[s] * a + b * rho[s] / total for a, b in zip(cross, body)]
            if self.model == "mr":
                span = range(-2, 3)
                belt = [(x, y, z) for x in span for y in span for z in span if x * x + y * y + z * z in _BELT]
                rep = self.gradient(psi[s], [_BELT[sum(a * a for a in c)] for c in belt], belt)
                att = self.gradient(psi[s], self.w)
                F = [f - p["Ga"][s] * psi[s] * a - p["Gr"][s] * psi[s] * b for f, a, b in zip(F, att, rep)]
            out.append(F)
        return out

    def velocity(self, forces):
        j = [torch.zeros_like(self.rho[0]) for _ in range(3)]
        for fk in self.f:
            for c, v in zip(self.cs, fk):
                for a, s in zip(j, c):
                    if s:
                        a += s * v
        total = sum(self.rho)
        return [self.fluid((a + 0.5 * sum(F[d] for F in forces)) / total) for d, a in enumerate(j)]

    def fields(self):
        self.rho = [sum(fk) for fk in self.f]
        forces = self.forces()
        return forces, self.velocity(forces)

    def source(self, i, u, F, omega):
        cu, cF = self.dot(self.cs[i], u), self.dot(self.cs[i], F)
        return self.w[i] * (1 - 0.5 * omega) * (3 * (cF - sum(a * b for a, b in zip(u, F))) + 9 * cu * cF)

    def step(self):
        forces, u = self.fields()
        q, p = len(self.cs), self.p
        new = [[torch.zeros_like(self.rho[0]) for _ in range(q)] for _ in self.f]
        if self.model == "cg":
            rr, rb = self.rho
            rho = rr + rb
            omega = 2 / (6 * self.nu() + 1)
            eqs = [self.equilibrium(k, u, self.gradient(self.rho[k])) for k in range(2)]
            rec = 0.7 * rr * rb / rho ** 2
            gabs = torch.where(self.has, self.gabs, 1.0)
        else:
            eqs = [self.equilibrium(k, u, None) for k in range(len(self.f))]
        for i, c in enumerate(self.cs):
            if self.model == "cg":
                total = self.f[0][i] + self.f[1][i]
                post = total - omega * (total - eqs[0](i) - eqs[1](i)) + self.source(i, u, forces[0], omega)
                cn = self.dot(c, self.gn) / gabs
                post = post + torch.where(self.has, p["A"] * gabs * (self.w[i] * cn * cn - self.B[i]), 0.0)
                cos = torch.where(self.has, cn, 0.0) / math.sqrt(max(1, self.r2[i]))
                part = rec * cos * (rr * self.phi[0][i] + rb * self.phi[1][i])
                posts = [rr / rho * post + part, rb / rho * post - part]
            else:
                posts = []
                for k, tau in enumerate((p["tau_r"], p.get("tau_b", 1.0))[:len(self.f)]):
                    v = self.f[k][i]
                    posts.append(v - (v - eqs[k](i)) / tau + self.source(i, u, forces[k], 1 / tau))
            for k, v in enumerate(posts):
                v = self.fluid(v)
                if self.solid is not None:  # halfway bounce-back at walls
                    wall = torch.roll(self.solid, (-c[2], -c[1], -c[0]), (0, 1, 2))
                    new[k][self.cs.index(tuple(-s for s in c))] += torch.where(wall, v, 0.0)
                    v = torch.where(wall, 0.0, v)
                new[k][i] += torch.roll(v, (c[2], c[1], c[0]), (0, 1, 2))
        self.f = new


def exact(case, seed):
    got = []
    for m, (model, nx, ny, nz) in enumerate(_members(case)):
        f = _fields(case, (model, nx, ny, nz), seed * 64 + m)
        sim = _Exact(model, _physics(case, model), (nz, ny, nx), f["rho_r"], f["rho_b"], f["u"], f["solid"])
        for _ in range(case["reads"]):
            for _ in range(case["steps"]):
                sim.step()
            _, u = sim.fields()
            rho = [a.reshape(-1).clone() for a in sim.rho] + [None] * (2 - len(sim.rho))
            got.append(rho + [torch.stack([a.reshape(-1) for a in u])])
    return got
