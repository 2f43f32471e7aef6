"""What a user of libsphtv has it do, as measurable cases.

Every case goes through the package's public entry points on device tensors,
the way a program that keeps its particles on the GPU uses the library:

* ``advance``: load a state (``sph_set_state``), build the cells, take some
  steps (kick-drift-kick, or advection steps of the dual-criteria integrator)
  and read the whole state back;
* ``rollout``: the differentiable rollout, forward and backward, with the
  kinetic energy at the end as the loss.

The workloads are the repository's own: the 2-D and 3-D Taylor-Green vortices,
the lid-driven cavity, the variable-resolution cylinder with its free-stream
forcing.  A Taylor-Green lattice is jittered by 1e-3 dp, as a run starts, or by
a tenth to a fifth of dp, as disordered as a run some hundred steps later.
"""
import math

import numpy as np
import torch

import paper_2411_13992_gb300 as sph
from paper_2411_13992_gb300 import cases as layouts
from paper_2411_13992_gb300 import cylinder as cylinder_runner

DEVICE = "cuda"


def listed():
    def adv(name, flow, side, precision, steps, jitter=1e-3, dual=False):
        return {"name": name, "kind": "advance", "flow": flow, "side": side, "precision": precision, "steps": steps,
                "jitter": jitter, "dual": dual}

    def roll(name, flow, side, precision, steps, every, jitter=1e-3):
        return {"name": name, "kind": "rollout", "flow": flow, "side": side, "precision": precision, "steps": steps,
                "every": every, "jitter": jitter}

    return [
        # a small cavity stepped one step at a time, state in and out: a host loop that looks at every step
        adv("cavity_48_f32_one_step", "cavity", 48, 32, 1),
        # the paper's coarse 2-D vortex in double precision: a parity or convergence run of few particles
        adv("tgv2d_50_f64", "tgv2d", 50, 64, 20),
        # the low-velocity cavity workload of the benchmark, walls included
        adv("cavity_256_f32", "cavity", 256, 32, 20),
        # a ragged mid-size 3-D box, part-way into a run
        adv("tgv3d_101_f32", "tgv3d", 101, 32, 10, jitter=0.1),
        # the headline workload as most steps of a long run see it: a disordered lattice
        adv("tgv3d_128_f32", "tgv3d", 128, 32, 10, jitter=0.2),
        # the large 3-D run, from its start
        adv("tgv3d_256_f32", "tgv3d", 256, 32, 4),
        # double precision in 3-D
        adv("tgv3d_96_f64", "tgv3d", 96, 64, 2, jitter=0.1),
        # flow past the cylinder: per-particle h, walls, free-stream forcing, body force
        adv("cylinder_36_f32", "cylinder", 36, 32, 10),
        # the paper's dual-criteria integrator: the cavity study's resolution, and the large 3-D box
        adv("cavity_200_f32_dual", "cavity", 200, 32, 5, dual=True),
        adv("tgv3d_128_f32_dual", "tgv3d", 128, 32, 2, jitter=0.1, dual=True),
        # gradients of a rollout: the adjoint workload, and a double-precision gradient check
        roll("rollout_256_f32", "tgv2d", 256, 32, 20, 10),
        roll("rollout_64_f64", "tgv2d", 64, 64, 10, 5, jitter=0.05),
    ]


# What a drawn case of each family may be: (kind, flow, precision, dual, smallest side, largest side, steps).
FAMILIES = [
    ("advance", "cavity", 32, False, 20, 400, (1, 20)),
    ("advance", "cavity", 64, False, 20, 150, (1, 10)),
    ("advance", "tgv2d", 32, False, 30, 700, (1, 20)),
    ("advance", "tgv2d", 64, False, 30, 200, (1, 20)),
    ("advance", "tgv3d", 32, False, 20, 200, (1, 6)),
    ("advance", "tgv3d", 64, False, 16, 80, (1, 2)),
    ("advance", "cylinder", 32, False, 6, 36, (1, 10)),
    ("advance", "cavity", 32, True, 30, 250, (1, 5)),
    ("advance", "tgv3d", 32, True, 20, 128, (1, 2)),
    ("rollout", "tgv2d", 32, False, 40, 280, (4, 20)),
    ("rollout", "tgv2d", 64, False, 30, 90, (4, 10)),
    ("rollout", "tgv3d", 32, False, 16, 40, (3, 8)),
]


def draw(rng):
    kind, flow, precision, dual, lo, hi, (s0, s1) = FAMILIES[rng.randrange(len(FAMILIES))]
    case = {"kind": kind, "flow": flow, "side": int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))),
            "precision": precision, "steps": rng.randint(s0, s1),
            "jitter": rng.choice([1e-3, 0.05, 0.1, 0.2]) if flow.startswith("tgv") else 1e-3}
    if kind == "rollout":
        case["every"] = rng.randint(2, case["steps"])
        case["jitter"] = min(case["jitter"], 0.1)
    else:
        case["dual"] = dual
    return case


# ----------------------------------------------------------------- inputs

def _layout(case, seed):
    """The flow's particles on the GPU and its parameters: the dict that
    ``sph.Simulation`` takes, with device tensors in place of arrays."""
    flow, n = case["flow"], case["side"]
    if flow in ("cavity", "cylinder"):
        if flow == "cavity":
            c = dict(layouts.cavity2d(n, seed=seed))
        else:
            c = dict(layouts.cylinder2d(res=n, seed=seed))
        for k in ("x", "v", "h", "m", "kind", "vw"):
            c[k] = torch.from_numpy(np.array(c[k])).to(DEVICE)
        return c
    dim = 2 if flow == "tgv2d" else 3
    box = 1.0 if dim == 2 else 2.0 * math.pi
    dp = box / n
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    axis = (torch.arange(n, dtype=torch.float64, device=DEVICE) + 0.5) * dp
    grid = torch.meshgrid(*([axis] * dim), indexing="ij")
    count = n ** dim
    x = torch.zeros((count, 3), dtype=torch.float64, device=DEVICE)
    for d in range(dim):
        x[:, d] = grid[dim - 1 - d].reshape(-1)       # x runs fastest
        x[:, d] += (2.0 * torch.rand(count, dtype=torch.float64, device=DEVICE, generator=gen) - 1.0) * (
            case["jitter"] * dp)
    v = torch.zeros_like(x)
    if dim == 2:
        k = 2.0 * math.pi
        v[:, 0] = torch.sin(k * x[:, 0]) * torch.cos(k * x[:, 1])
        v[:, 1] = -torch.cos(k * x[:, 0]) * torch.sin(k * x[:, 1])
        nu, L, periodic = 1.0 / 100.0, (1.0, 1.0, 1.0), (1, 1, 0)
    else:
        cz = torch.cos(x[:, 2])
        v[:, 0] = torch.sin(x[:, 0]) * torch.cos(x[:, 1]) * cz
        v[:, 1] = -torch.cos(x[:, 0]) * torch.sin(x[:, 1]) * cz
        nu, L, periodic = 1.0 / 1600.0, (box, box, box), (1, 1, 1)
    h = 1.3 * dp
    full = lambda value: torch.full((count,), value, dtype=torch.float64, device=DEVICE)
    return dict(name=flow, dim=dim, n=count, lo=(0.0, 0.0, 0.0), L=L, periodic=periodic, rho0=1.0, c=10.0, eta=nu,
                nu=nu, u_ref=1.0, g=(0.0, 0.0, 0.0), x=x, v=v, h=full(h), m=full(dp ** dim), h_min=h, h_max=h, dp=dp)


def _rollout_dt(c):
    """Fixed step of a rollout: the acoustic criterion with |v| up to 1.2."""
    return 0.6 * c["h_min"] / (1.2 + c["c"])


def _fringe(case):
    return cylinder_runner.FRINGE if case["flow"] == "cylinder" else None


def prepare(case, seed):
    c = _layout(case, seed)
    opts = {}
    if case["kind"] == "rollout":
        opts = dict(fixed_dt=_rollout_dt(c), adjoint_steps=case["every"])
    elif case["dual"]:
        opts = dict(integrator=sph.INT_DUAL)
    fringe = _fringe(case)
    if fringe:
        opts.update(body_force=1, fringe_lambda=fringe[0], fringe_u=fringe[1], fringe_x=fringe[2])
    sim = sph.Simulation(c, precision=case["precision"], **opts)
    state = {"case": case, "sim": sim, "c": c}
    if case["kind"] == "rollout":
        state["x0"] = c["x"].clone().requires_grad_(True)
        state["v0"] = c["v"].clone().requires_grad_(True)
        state["nu"] = torch.tensor(c["nu"], dtype=torch.float64, requires_grad=True)
    return state


# ------------------------------------------------------------------- a pass

def run(state):
    case, sim, c = state["case"], state["sim"], state["c"]
    if case["kind"] == "rollout":
        x0, v0, nu = state["x0"], state["v0"], state["nu"]
        x0.grad = v0.grad = nu.grad = None
        xT, vT = sph.Rollout.apply(x0, v0, nu, sim, case["steps"], case["every"])
        loss = 0.5 * (c["m"][:, None] * vT * vT).sum()
        loss.backward()
        return [xT.detach(), vT.detach(), x0.grad, v0.grad, nu.grad]
    n = sim.n
    sim.set_state()
    sim.build_cells()
    sim.step(case["steps"])
    vector = lambda: torch.empty((n, 3), dtype=torch.float64, device=DEVICE)
    scalar = lambda: torch.empty(n, dtype=torch.float64, device=DEVICE)
    if case["dual"]:
        # what the integrator goes on from: x, v and the density rate; with dr and the density
        x, v, dr, rho, rate = vector(), vector(), vector(), scalar(), scalar()
        sph.sph_get_state(sim.ctx, x, v, None, dr, rho)
        sph.sph_get_density_rate(sim.ctx, rate)
        return [x, v, dr, rho, rate]
    out = [vector(), vector(), vector(), vector(), scalar()]
    sph.sph_get_state(sim.ctx, *out)
    return out


# --------------------------------------------------------------------- work

def work(case):
    flow, side, steps = case["flow"], case["side"], case["steps"]
    dim = 3 if flow == "tgv3d" else 2
    n = side ** dim
    if flow == "cavity":
        n = (side + 6) ** 2
    elif flow == "cylinder":
        n = int(991918 * (side / 36.0) ** 2)
    pairs = n * (80 if dim == 3 else 20.2)
    density, forces = 25.0 * (pairs + n), 111.0 * pairs
    if case["kind"] == "rollout":
        # in: x, v, h, m and the loss's gradient; out: x, v and the gradients of x and v
        reverse = 2 * 130.0 * pairs + 30.0 * pairs
        return {"bytes": n * (48 + 16 + 48 + 48.0), "flops": (2 * steps + 2) * (density + forces) + (steps + 1) * reverse}
    bytes_ = n * (48 + 16 + 96 + 8.0)                   # in: x, v, h, m; out: x, v, a, dr, rho
    if case["dual"]:
        sub = 5                                         # acoustic substeps of an advection step
        return {"bytes": bytes_, "flops": (steps + 1) * density + steps * pairs * (45.0 + sub * (65.0 + 50.0))}
    return {"bytes": bytes_, "flops": (steps + 1) * (density + forces)}


# -------------------------------------------------- the same in plain torch

class _Flow:
    """The method in 64-bit torch: neighbour pairs from a cell grid, sums by
    index_add.  rho0 = 1; walls stand in with the fluid particle's density and
    pressure and their own velocity."""

    CFL_AD, CFL_AC, SLOPE, XI, TV_C, TV_MIN = 0.25, 0.6, 3.0, -0.2, 1.0e3, 5.0e-4

    def __init__(self, c, case):
        self.D = D = c["dim"]
        self.n = c["n"]
        self.lo = torch.tensor(c["lo"][:D], dtype=torch.float64, device=DEVICE)
        self.L = torch.tensor(c["L"][:D], dtype=torch.float64, device=DEVICE)
        self.per = [bool(p) for p in c["periodic"][:D]]
        self.cs, self.nu, self.u_ref = c["c"], c["eta"], c["u_ref"]
        self.h, self.m = c["h"], c["m"]
        self.h_min, self.h_max = c["h_min"], c["h_max"]
        kind = c.get("kind")
        self.fluid = torch.ones(self.n, dtype=torch.bool, device=DEVICE) if kind is None else kind == 0
        self.walls = bool((~self.fluid).any())
        self.norm = 7.0 / (4.0 * math.pi) if D == 2 else 21.0 / (16.0 * math.pi)
        self.fringe = _fringe(case)
        self.sigma0 = self._sigma0()

    # kernel: W = a h^-D (1 - q/2)^4 (2q + 1), support 2h
    def W(self, r, h):
        q = r / h
        return torch.where(q < 2.0, self.norm / h ** self.D * (1 - 0.5 * q) ** 4 * (2 * q + 1), torch.zeros_like(q))

    def dW(self, r, h):
        q = r / h
        return torch.where(q < 2.0, self.norm / h ** (self.D + 1) * (-5.0 * q) * (1 - 0.5 * q) ** 3,
                           torch.zeros_like(q))

    def _sigma0(self):
        """The perfect-lattice sum at each particle's own spacing m^(1/D) and h."""
        hm, inverse = torch.unique(torch.stack([self.h, self.m], 1), dim=0, return_inverse=True)
        out = torch.empty(len(hm), dtype=torch.float64, device=DEVICE)
        for at in range(0, len(hm), 65536):
            h, dp = hm[at:at + 65536, 0], hm[at:at + 65536, 1] ** (1.0 / self.D)
            reach = int(math.ceil(float((2.0 * h / dp).max()))) + 1
            ax = torch.arange(-reach, reach + 1, dtype=torch.float64, device=DEVICE)
            k2 = sum(g.reshape(-1) ** 2 for g in torch.meshgrid(*([ax] * self.D), indexing="ij"))
            r = torch.sqrt(k2)[None, :] * dp[:, None]
            out[at:at + 65536] = self.W(r, h[:, None].expand_as(r)).sum(1)
        return out[inverse]

    def image(self, d):
        parts = []
        for k in range(self.D):
            t = d[:, k]
            if self.per[k]:
                t = t - self.L[k] * torch.round(t.detach() / self.L[k])
            parts.append(t)
        return torch.stack(parts, 1)

    def pairs(self, x):
        """Yield (i, j) index tensors: every pair with r < 2 h_ij (self
        included), in blocks of particles i."""
        x = x[:, :self.D].detach()
        reach = 2.0 * self.h_max
        nc, cell = [], []
        for d in range(self.D):
            lo = self.lo[d] if self.per[d] else x[:, d].min()
            hi = self.lo[d] + self.L[d] if self.per[d] else x[:, d].max()
            k = max(int(float((hi - lo) / reach)), 1)
            nc.append(k)
            cell.append(((x[:, d] - lo) / ((hi - lo) / k)).floor().long().clamp_(0, k - 1))
        key = cell[0]
        stride = nc[0]
        for d in range(1, self.D):
            key = key + cell[d] * stride
            stride *= nc[d]
        order = torch.argsort(key)
        count = torch.bincount(key, minlength=stride)
        start = torch.cumsum(count, 0) - count
        steps = torch.cartesian_prod(*([torch.arange(-1, 2)] * self.D)).tolist()
        block = 1 << 21
        for at in range(0, self.n, block):
            ii = order[at:at + block]
            found_i, found_j = [], []
            seen = []
            for st in steps:
                ok = torch.ones(len(ii), dtype=torch.bool, device=DEVICE)
                other = torch.zeros(len(ii), dtype=torch.long, device=DEVICE)
                stride, mark = 1, []
                for d in range(self.D):
                    k = cell[d][ii] + st[d]
                    if self.per[d]:
                        k = k % nc[d]
                    else:
                        ok &= (k >= 0) & (k < nc[d])
                        k = k.clamp(0, nc[d] - 1)
                    other += k * stride
                    stride *= nc[d]
                    mark.append(st[d] % nc[d] if self.per[d] else st[d])
                if tuple(mark) in seen:           # an axis of fewer than three cells meets itself
                    continue
                seen.append(tuple(mark))
                cnt = torch.where(ok, count[other], torch.zeros_like(other))
                i = torch.repeat_interleave(ii, cnt)
                first = torch.repeat_interleave(start[other] - (torch.cumsum(cnt, 0) - cnt), cnt)
                j = order[first + torch.arange(len(i), device=DEVICE)]
                r = self.image(x[i] - x[j]).norm(dim=1)
                near = r < self.h[i] + self.h[j]
                found_i.append(i[near])
                found_j.append(j[near])
            yield torch.cat(found_i), torch.cat(found_j)

    def density(self, x, blocks):
        sigma = torch.zeros(self.n, dtype=torch.float64, device=DEVICE)
        for i, j in blocks:
            r2 = (self.image(x[i, :self.D] - x[j, :self.D]) ** 2).sum(1)
            zero = r2 == 0
            r = torch.where(zero, torch.zeros_like(r2), torch.sqrt(torch.where(zero, torch.ones_like(r2), r2)))
            sigma = sigma.index_add(0, i, self.W(r, 0.5 * (self.h[i] + self.h[j])))
        return torch.where(self.fluid, sigma / self.sigma0, torch.ones_like(sigma))

    def pair(self, x, v, rho, i, j):
        keep = (i != j) & self.fluid[i]
        i, j = i[keep], j[keep]
        rv = self.image(x[i, :self.D] - x[j, :self.D])
        r = torch.sqrt((rv * rv).sum(1))
        dv = v[i, :self.D] - v[j, :self.D]
        dw = self.dW(r, 0.5 * (self.h[i] + self.h[j]))
        ri = rho[i]
        rj = torch.where(self.fluid[j], rho[j], ri) if self.walls else rho[j]
        return i, j, rv, r, dv, dw, ri, rj

    def interface_pressure(self, rv, r, dv, ri, rj):
        dU = -(dv * rv).sum(1) / r
        beta = torch.clamp(self.SLOPE * dU / self.cs, 0.0, 1.0)
        p = self.cs ** 2 * (0.5 * (ri + rj) - 1.0)
        return p + 0.5 * beta * (0.5 * (ri + rj)) * self.cs * dU

    def limiter(self, s):
        return torch.where(s > self.TV_MIN, torch.clamp(self.TV_C * s, max=1.0), torch.zeros_like(s))

    def _pad(self, t):
        return t if self.D == 3 else torch.nn.functional.pad(t, (0, 1))

    def forces(self, x, v, rho, blocks, nu, terms=("p", "nu", "R")):
        zero = lambda: torch.zeros((self.n, self.D), dtype=torch.float64, device=DEVICE)
        a, R = zero(), zero()
        for bi, bj in blocks:
            i, j, rv, r, dv, dw, ri, rj = self.pair(x, v, rho, bi, bj)
            f = 0.0
            if "p" in terms:
                p = self.interface_pressure(rv, r, dv, ri, rj)
                f = f + (-2.0 * self.m[j] / (ri * rj) * p * dw / r)[:, None] * rv
            if "nu" in terms:
                f = f + (2.0 * nu * self.m[j] / (ri * rj) * dw / r)[:, None] * dv
            if "R" in terms:
                R = R.index_add(0, i, (self.m[j] / rj * dw / r)[:, None] * rv)
            a = a.index_add(0, i, f)
        if self.fringe and "p" in terms:
            lam, u, (x0, x1, rise, fall) = self.fringe
            def ramp(t):
                inner = t.clamp(1e-9, 1.0 - 1e-9)
                s = 1.0 / (1.0 + torch.exp(1.0 / (inner - 1.0) + 1.0 / inner))
                return torch.where(t <= 0, torch.zeros_like(t), torch.where(t >= 1, torch.ones_like(t), s))
            rate = lam * (ramp((x[:, 0] - x0) / rise) - ramp((x[:, 0] - x1) / fall + 1.0))
            uinf = torch.tensor(u[:self.D], dtype=torch.float64, device=DEVICE)
            a = a + rate[:, None] * (uinf - v[:, :self.D]) * self.fluid[:, None]
        dr = self.XI * self.limiter(self.h_min ** 2 * (R * R).sum(1))[:, None] * self.h_min ** 2 * R
        return self._pad(a), self._pad(dr)

    def vmax(self, v):
        return float(v.detach()[self.fluid].norm(dim=1).max())

    def dt_ad(self, vmax):
        return self.CFL_AD * self.h_min / max(vmax, self.nu / self.h_min, self.u_ref)

    def dt_ac(self, vmax):
        return self.CFL_AC * self.h_min / (vmax + self.cs)

    def wrap(self, x):
        cols = []
        for d in range(3):
            t = x[:, d]
            if d < self.D and self.per[d]:
                lo, L = self.lo[d], self.L[d]
                t = torch.where(t.detach() < lo, t + L, torch.where(t.detach() >= lo + L, t - L, t))
            cols.append(t)
        return torch.stack(cols, 1)

    def force_pass(self, x, v, nu):
        """Density and forces, the pairs of one block of particles at a time
        (the density of all first)."""
        if self.n <= 1 << 21:
            blocks = list(self.pairs(x))
        else:
            blocks = None
        rho = self.density(x, blocks if blocks is not None else self.pairs(x))
        a, dr = self.forces(x, v, rho, blocks if blocks is not None else self.pairs(x), nu)
        return rho, a, dr

    def kdk(self, x, v, steps, nu, fixed_dt=0.0):
        f = self.fluid[:, None]
        rho, a, dr = self.force_pass(x, v, nu)
        for _ in range(steps):
            vmax = 0.0 if fixed_dt else self.vmax(v)
            dt = fixed_dt or min(self.dt_ad(vmax), self.dt_ac(vmax))
            vh = torch.where(f, v + 0.5 * dt * a, v)
            x = self.wrap(torch.where(f, x + dt * vh + dr, x))
            rho, a, dr = self.force_pass(x, vh, nu)
            v = torch.where(f, vh + 0.5 * dt * a, vh)
        return x, v, a, dr, rho

    def continuity(self, x, v, rho, blocks):
        out = torch.zeros(self.n, dtype=torch.float64, device=DEVICE)
        for bi, bj in blocks:
            i, j, rv, r, dv, dw, ri, rj = self.pair(x, v, rho, bi, bj)
            du = 0.5 * (dv * rv).sum(1) / r + 0.5 * self.cs * (ri - rj) / (0.5 * (ri + rj))
            out = out.index_add(0, i, 2.0 * ri * self.m[j] / rj * du * dw)
        return out

    def dual(self, x, v, steps):
        f = self.fluid[:, None]
        rate = torch.zeros(self.n, dtype=torch.float64, device=DEVICE)
        for _ in range(steps):
            blocks = list(self.pairs(x))                # frozen for the advection step
            rho = self.density(x, blocks)
            Dt = self.dt_ad(self.vmax(v))
            held, _ = self.forces(x, v, rho, blocks, self.nu, terms=("nu",))
            _, dr = self.forces(x, v, rho, blocks, self.nu)
            x = torch.where(f, x + dr, x)
            t, last = 0.0, False
            while not last:
                dt = self.dt_ac(self.vmax(v))
                last = not dt < Dt - t
                if last:
                    dt = Dt - t
                rho = torch.where(self.fluid, rho + 0.5 * dt * rate, rho)
                x = torch.where(f, x + 0.5 * dt * v, x)
                a, _ = self.forces(x, v, rho, blocks, self.nu, terms=("p",))
                a = torch.where(f, a + held, torch.zeros_like(a))
                v = torch.where(f, v + dt * a, v)
                x = torch.where(f, x + 0.5 * dt * v, x)
                rate = self.continuity(x, v, rho, blocks)
                rho = torch.where(self.fluid, rho + 0.5 * dt * rate, rho)
                t += dt
            x = self.wrap(x)
        return x, v, dr, rho, rate


def exact(case, seed):
    if case["flow"] == "tgv3d" and case["side"] ** 3 * (case["steps"] + 1) > 50e6:
        return None                                     # over 20 s
    c = _layout(case, seed)
    flow = _Flow(c, case)
    v = c["v"]
    if "vw" in c:
        v = torch.where(flow.fluid[:, None], v, c["vw"])
    if case["kind"] == "rollout":
        x0 = c["x"].clone().requires_grad_(True)
        v0 = v.clone().requires_grad_(True)
        nu = torch.tensor(c["nu"], dtype=torch.float64, device=DEVICE, requires_grad=True)
        x, v, _, _, _ = flow.kdk(x0, v0, case["steps"], nu, fixed_dt=_rollout_dt(c))
        (0.5 * (c["m"][:, None] * v * v).sum()).backward()
        return [x.detach(), v.detach(), x0.grad, v0.grad, nu.grad.cpu()]
    with torch.no_grad():
        if case["dual"]:
            return list(flow.dual(c["x"], v, case["steps"]))
        return list(flow.kdk(c["x"], v, case["steps"], flow.nu))
