"""Performance cases of the fused multiphase lattice-Boltzmann step, through the public Python API.

A case is one uninterrupted stretch of a simulation as a user's program runs it: advance a domain (or a
batch of domains) by `steps` time steps and read the result back on the device.  The simulation goes on
from pass to pass, as it does in a run of thousands of steps.  What is read back is either the whole
state (`out` = "populations": a checkpoint) or the fields (`out` = "moments": a frame of a movie, a
monitored quantity).

`kind` of a case:
  droplets   periodic box of liquid spheres in vapour: one sphere is the Laplace test and the job of a
             parameter sweep, many are the method at scale
  impact     a droplet moving towards the lower of two walls in z
  cylinder   a droplet falling onto a solid cylinder on the bottom wall (a solid mask), wetting force on
  vortex     single-phase decaying vortex, no equation of state
  batch      independent droplet and impact domains of uneven edges and both lattices, advanced together
"""
import math

import numpy as np
import torch

from paper_2306_16274_gb300 import Batch, Params, Simulation

# Carnahan-Starling at 0.7 T_c and its Maxwell densities; the piecewise equation of state with density
# ratio 1000 (workloads/constants.json)
CS_P, CS_L, CS_V = (0.5, 4.0, 1.0, 0.03301504609688092), 0.35813094118772437, 0.009294146215100382
PW_P = (0.0013246030524049143, 0.9758004064414756, 1.0 / 6.0, -0.008333333333333333, 1.0 / 3.0)
PW_L, PW_V = 1.0, 0.001
RATES = {"s0": 1.0, "s1": 1.0, "s2": 1.2, "s2b": 0.6, "s3": 1.2, "s3b": 0.6, "s4": 1.2, "s4b": 1.2, "s5": 1.2,
         "s6": 1.2}


def _case(kind, lattice, shape, steps, out="populations", store="fp32", onepass=False, eos="cs", kappa=0.0,
          spheres=1, jobs=0, layout=0):
    nx, ny, nz = shape
    return {"kind": kind, "lattice": lattice, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "out": out,
            "store": store, "onepass": onepass, "eos": eos, "kappa": kappa, "spheres": spheres, "jobs": jobs,
            "layout": layout}


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # a coupled or monitored run: one step of a small ragged domain, then its fields
        named("monitor_q27_24x20x17", "vortex", 27, (24, 20, 17), 1, out="moments", eos="none"),
        # the Laplace test: 32^3, one droplet, a tick of 100 steps between checks
        named("laplace_q19_32", "droplets", 19, (32, 32, 32), 100),
        # a parameter-sweep job on D3Q27 whose edges divide by nothing
        named("sweep_q27_61x83x70", "droplets", 27, (61, 83, 70), 50, kappa=0.3),
        # ordinary single-phase validation flow
        named("vortex_q19_128", "vortex", 19, (128, 128, 128), 40, eos="none"),
        # the density-ratio-1000 droplet of the validation runs, piecewise equation of state
        named("ratio1000_q19_160", "droplets", 19, (160, 160, 160), 25, eos="piecewise"),
        # the method at scale, both lattices: the benchmark's domain
        named("scale_q19_256", "droplets", 19, (256, 256, 256), 20, kappa=0.5, spheres=24),
        named("scale_q27_256", "droplets", 27, (256, 256, 256), 20, kappa=0.5, spheres=24),
        # the same step on two population copies
        named("onepass_q27_192", "droplets", 27, (192, 192, 192), 20, kappa=0.5, spheres=12, onepass=True),
        # droplet impact at half scale in FP32, frames of a movie
        named("impact_q19_200x200x100", "impact", 19, (200, 200, 100), 25, out="moments"),
        # droplet impact at full scale with the FP16 population store
        named("impact_fp16_q19_400x400x200", "impact", 19, (400, 400, 200), 10, store="fp16"),
        # a serving job: impact on a cylinder
        named("cylinder_q19_127x127x106", "cylinder", 19, (127, 127, 106), 25, kappa=0.3),
        # many uneven jobs together
        named("batch_10_jobs", "batch", 19, (48, 48, 112), 20, jobs=10, layout=7),
    ]


def draw(rng):
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["droplets", "droplets", "droplets", "impact", "cylinder", "vortex", "batch"])
    Q = rng.choice([19, 27])
    if kind == "batch":
        lo = rng.randint(32, 64)
        return _case(kind, Q, (lo, lo, rng.randint(lo + 8, 112)), rng.randint(5, 20), jobs=rng.randint(4, 12),
                     layout=rng.randrange(1 << 20))
    if kind == "droplets":
        e = edge(24, 240)
        shape = tuple(max(20, min(256, int(e * rng.uniform(0.75, 1.25)))) for _ in range(3))
    elif kind == "vortex":
        e = edge(16, 160)
        shape = tuple(max(12, int(e * rng.uniform(0.75, 1.25))) for _ in range(3))
    else:
        e = edge(48, 224)
        shape = (e, int(e * rng.uniform(0.8, 1.2)), int(e * rng.uniform(0.7, 0.9)))
    cells = shape[0] * shape[1] * shape[2]
    steps = rng.randint(1, max(2, min(100, int(2.5e8 / cells))))
    store, onepass, eos, spheres = "fp32", False, "cs", 1
    if kind == "vortex":
        eos = "none"
    elif kind == "droplets":
        opt = rng.random()
        if opt < 0.15:
            store = "fp16"
        elif opt < 0.3:
            onepass = True
        elif opt < 0.45 and min(shape) >= 40:
            eos = "piecewise"
        if eos == "cs" and min(shape) >= 64:
            spheres = rng.choice([1, 4, 12, 24])
    elif kind == "impact" and rng.random() < 0.3:
        store = "fp16"
    out = "moments" if kind in ("vortex", "impact") and rng.random() < 0.4 else "populations"
    kappa = rng.choice([0.0, 0.3, 0.5]) if eos == "cs" else 0.0
    return _case(kind, Q, shape, steps, out, store, onepass, eos, kappa, spheres)


# ---------------------------------------------------------------- inputs
def _members(case):
    """The domains of a batch: edges between nx and nz, alternating lattices and kinds."""
    rng = np.random.default_rng(case["layout"])
    out = []
    for k in range(case["jobs"]):
        L = int(rng.integers(case["nx"], case["nz"] + 1))
        Q = case["lattice"] if k % 2 == 0 else 46 - case["lattice"]
        out.append(_case("impact" if rng.random() < 0.5 else "droplets", Q, (L, L, L), case["steps"]))
    return out


def _params(case):
    p = dict(lattice=case["lattice"], shape=(case["nx"], case["ny"], case["nz"]), store=case["store"],
             onepass=case["onepass"], sigma=0.1, G=-1.0, kappa=case["kappa"])
    if case["eos"] == "cs":
        p.update(eos="cs", eos_p=CS_P)
    elif case["eos"] == "piecewise":
        p.update(eos="piecewise", eos_p=PW_P)
    if case["kind"] in ("impact", "cylinder"):
        p.update(bc=("periodic", "periodic", "wall"))
    if case["kind"] == "cylinder":
        p.update(G_ads=0.23)
    return p


def _axes(case):
    a = [torch.arange(n, dtype=torch.float64, device="cuda") for n in (case["nx"], case["ny"], case["nz"])]
    return a[0][None, None, :], a[1][None, :, None], a[2][:, None, None]


def _spheres(case, rng):
    """Non-overlapping periodic spheres (centre, radius)."""
    L = np.array([case["nx"], case["ny"], case["nz"]], dtype=float)
    if case["spheres"] <= 1:
        return [(rng.uniform(0.4, 0.6, 3) * L, float(rng.uniform(0.22, 0.28) * L.min()))]
    got = []
    for _ in range(4000):
        r, c = float(rng.uniform(0.06, 0.15) * L.min() + 3.0), rng.uniform(0.0, 1.0, 3) * L
        ok = True
        for c2, r2 in got:
            d = c - c2
            d -= L * np.round(d / L)
            ok = ok and np.sqrt((d * d).sum()) > r + r2 + 4.0
        if ok:
            got.append((c, r))
        if len(got) == case["spheres"]:
            break
    return got


def _fields(case, seed):
    """(rho, u, solid): float32 fields and a uint8 mask (or None) on the GPU, from the seed alone."""
    rng = np.random.default_rng([seed, case["lattice"], case["nx"], case["ny"], case["nz"]])
    x, y, z = _axes(case)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    solid = None
    if case["kind"] == "vortex":
        U, ph = rng.uniform(0.03, 0.05), rng.uniform(0.0, 2 * np.pi, 3)
        kx, ky, kz = 2 * np.pi / nx, 2 * np.pi / ny, 2 * np.pi / nz
        sx, cx, sy, cy = (torch.sin(kx * x + ph[0]), torch.cos(kx * x + ph[0]), torch.sin(ky * y + ph[1]),
                          torch.cos(ky * y + ph[1]))
        u = torch.stack([(U * sx * cy).expand(shape), (-U * (kx / ky) * cx * sy).expand(shape),
                         (0.3 * U * torch.sin(kx * x + ky * y + ph[2])).expand(shape)])
        rho = (1.0 + 0.01 * torch.sin(kz * z + ph[2])).expand(shape)
        return rho.float().contiguous(), u.float().contiguous(), None
    lo, hi = (PW_V, PW_L) if case["eos"] == "piecewise" else (CS_V, CS_L)
    W = 4.0 if case["eos"] == "piecewise" else 3.0

    def sphere(c, r, periodic):
        d2 = 0.0
        for a, k, n in ((x, 0, nx), (y, 1, ny), (z, 2, nz)):
            d = a - float(c[k])
            if periodic:
                d = d - n * torch.round(d / n)
            d2 = d2 + d * d
        return 0.5 * (hi + lo) - 0.5 * (hi - lo) * torch.tanh(2.0 * (torch.sqrt(d2) - r) / W)

    u = torch.zeros((3,) + shape, dtype=torch.float64, device="cuda")
    if case["kind"] == "droplets":
        rho = torch.full(shape, lo, dtype=torch.float64, device="cuda")
        for c, r in _spheres(case, rng):
            rho = torch.maximum(rho, sphere(c, r, True))
        return rho.float(), u.float(), None
    m = min(nx, ny, nz)
    if case["kind"] == "impact":
        R = rng.uniform(0.23, 0.26) * m
        rho = sphere((nx / 2 + rng.uniform(-2, 2), ny / 2 + rng.uniform(-2, 2), R + rng.uniform(3.0, 6.0)), R, False)
    else:
        R, Rc = rng.uniform(0.17, 0.19) * m, rng.uniform(0.13, 0.15) * m
        solid = (torch.sqrt((x - nx / 2) ** 2 + (z - (Rc - 0.5)) ** 2) <= Rc).expand(shape)
        rho = sphere((nx / 2 + rng.uniform(-2, 2), ny / 2 + rng.uniform(-2, 2), 2 * Rc + 3.0 + R), R, False)
    u[2] = -rng.uniform(0.03, 0.04) * ((rho - lo) / (hi - lo)).clamp(0.0, 1.0)
    if solid is not None:
        rho = torch.where(solid, torch.full_like(rho, lo), rho)
        u = torch.where(solid[None], torch.zeros_like(u), u)
        solid = solid.to(torch.uint8).contiguous()
    return rho.float().contiguous(), u.float().contiguous(), solid


# ---------------------------------------------------------------- the pass
def _simulation(case, seed):
    sim = Simulation(Params(**_params(case)))
    rho, u, solid = _fields(case, seed)
    sim.init_fields(rho, u, solid)
    torch.cuda.synchronize()   # the inputs' memory goes back to torch's allocator here
    return sim


def prepare(case, seed):
    if case["kind"] == "batch":
        sims = [_simulation(m, seed * 131 + k) for k, m in enumerate(_members(case))]
        return {"case": case, "sims": sims, "batch": Batch(sims)}
    return {"case": case, "sim": _simulation(case, seed)}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        return [s.populations() for s in state["sims"]]
    sim = state["sim"]
    sim.step(case["steps"])
    if case["out"] == "moments":
        rho, u, _ = sim.moments(sums=False)
        return {"rho": rho, "u": u}
    return sim.populations()


def work(case):
    """A step reads and writes every population once (8 Q bytes a cell; 4 Q in half precision); the
    result is read from the state and written once.  Operations: additions and multiplications of one
    cell's moment transforms, relaxation, forces and equation of state, counted in the formulas."""
    if case["kind"] == "batch":
        w = [work(m) for m in _members(case)]
        return {"bytes": sum(v["bytes"] for v in w), "flops": sum(v["flops"] for v in w)}
    Q, cells = case["lattice"], case["nx"] * case["ny"] * case["nz"]
    slot = 2 if case["store"] == "fp16" else 4
    per_step = 2 * slot * Q
    result = slot * Q + 4 * (Q if case["out"] == "populations" else 4)
    flops = {19: 260, 27: 420}[Q] + (0 if case["eos"] == "none" else {19: 190, 27: 270}[Q])
    return {"bytes": cells * (case["steps"] * per_step + result), "flops": cells * case["steps"] * flops}


# ---------------------------------------------------------------- the same in 64 bits, plain torch
class _Exact:
    """The method written out in 64-bit torch: raw moments by matrix products, shifts by torch.roll."""

    def __init__(self, case):
        self.p = _params(case)
        self.Q = case["lattice"]
        self.wall_z = case["kind"] in ("impact", "cylinder")
        e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
             (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1),
             (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1),
             (1, 1, 1), (-1, 1, 1), (1, -1, 1), (-1, -1, 1), (1, 1, -1), (-1, 1, -1), (1, -1, -1), (-1, -1, -1)]
        self.e = e[:self.Q]
        self.opp = [self.e.index((-a, -b, -c)) for a, b, c in self.e]
        wn = {19: {1: 1 / 6, 2: 1 / 12}, 27: {1: 2 / 9, 2: 1 / 18, 3: 1 / 72}}[self.Q]
        self.w = [wn.get(a * a + b * b + c * c, 0.0) for a, b, c in self.e]
        rows = []
        for x, y, z in self.e:
            r = [1, x, y, z, x * y, x * z, y * z, x * x + y * y + z * z, x * x - y * y, x * x - z * z, x * y * y,
                 x * z * z, x * x * y, x * x * z, y * z * z, y * y * z, x * y * z, x * x * y * y, x * x * z * z,
                 y * y * z * z, x * x * y * z, x * y * y * z, x * y * z * z, x * y * y * z * z, x * x * y * z * z,
                 x * x * y * y * z, x * x * y * y * z * z]
            rows.append(r if self.Q == 27 else r[:16] + r[17:20])
        M = np.array(rows, dtype=np.float64).T
        self.M = torch.tensor(M, device="cuda")
        self.Mi = torch.tensor(np.linalg.inv(M), device="cuda")

    def at(self, k):
        return k if self.Q == 27 or k < 16 else k - 1

    def shift(self, a, e):
        """a(x + e), periodic"""
        return torch.roll(a, (-e[2], -e[1], -e[0]), (-3, -2, -1))

    def start(self, rho, u, solid):
        self.shape = rho.shape
        rho, u = rho.double(), u.double()
        self.solid = torch.zeros(self.shape, dtype=torch.bool, device="cuda") if solid is None else solid.bool()
        self.open = solid is None and not self.wall_z
        self.f = self.back(self.equilibrium(rho, u))
        if solid is not None:
            self.f[:, self.solid] = 0.0

    def solid_at(self, i):
        """Is x + e_i solid (mask, or beyond a wall)?"""
        e = self.e[i]
        s = self.shift(self.solid, e)
        if self.wall_z and e[2] != 0:
            s = s.clone()
            s[0 if e[2] < 0 else -1] = True
        return s

    def back(self, m):
        return (self.Mi @ m.reshape(self.Q, -1)).reshape((self.Q,) + self.shape)

    def equilibrium(self, rho, u):
        x, y, z = u
        xx, yy, zz, c = x * x, y * y, z * z, 1.0 / 3.0
        m = [rho, rho * x, rho * y, rho * z, rho * x * y, rho * x * z, rho * y * z, rho * (1 + xx + yy + zz),
             rho * (xx - yy), rho * (xx - zz), c * rho * x, c * rho * x, c * rho * y, c * rho * z, c * rho * y,
             c * rho * z, 0.0 * rho, c * rho * (c + xx + yy), c * rho * (c + xx + zz), c * rho * (c + yy + zz)]
        if self.Q == 27:
            m += [c * rho * y * z, c * rho * x * z, c * rho * x * y, c * c * rho * x, c * c * rho * y, c * c * rho * z,
                  c * c * rho * (xx + yy + zz) + c ** 3 * rho]
        else:
            del m[16]
        return torch.stack(m)

    def psi(self, rho):
        if self.p["eos"] == "cs":
            a, b, R, T = self.p["eos_p"]
            n = b * rho / 4.0
            p = rho * R * T * (1 + n + n * n - n ** 3) / (1 - n) ** 3 - a * rho * rho
        else:
            r1, r2, tv, tm, tl = self.p["eos_p"]
            p = torch.where(rho <= r1, rho * tv, torch.where(rho <= r2, r1 * tv + (rho - r1) * tm,
                                                             r1 * tv + (r2 - r1) * tm + (rho - r2) * tl))
        psi = torch.sqrt((2.0 / self.p["G"] * (p - rho / 3.0)).clamp(min=0.0))
        return torch.where(self.solid, torch.zeros_like(psi), psi)

    def forces(self, rho):
        """(F, Q tensor, |S|^2), or None without an equation of state"""
        if self.p.get("eos") is None:
            return None
        psi = self.psi(rho)
        zero = torch.zeros_like(rho)
        S, A, T = [zero.clone() for _ in range(3)], [zero.clone() for _ in range(3)], [zero.clone() for _ in range(6)]
        pairs = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
        for i in range(1, self.Q):
            e, w, nb = self.e[i], self.w[i], self.shift(psi, self.e[i])
            if not self.open:
                s = self.solid_at(i)
                nb = torch.where(s, psi, nb)
                for a in range(3):
                    if e[a]:
                        A[a] += w * e[a] * s
            for a in range(3):
                if e[a]:
                    S[a] += w * e[a] * nb
            for k, (a, b) in enumerate(pairs):
                if e[a] and e[b]:
                    T[k] += w * e[a] * e[b] * (nb - psi)
        G, Ga = self.p["G"], self.p.get("G_ads", 0.0)
        F = [-G * psi * S[a] - Ga * psi * psi * A[a] for a in range(3)]
        return F, [0.5 * self.p["kappa"] * G * psi * t for t in T], sum(s * s for s in S)

    def macroscopic(self):
        f = self.f
        rho = f.sum(0)
        if not self.open:
            rho = torch.where(self.solid, torch.ones_like(rho), rho)
        FT = self.forces(rho)
        j = (self.M[1:4] @ f.reshape(self.Q, -1)).reshape((3,) + self.shape)
        if FT is not None:
            j = j + 0.5 * torch.stack(FT[0])
        return rho, j / rho, FT

    def step(self):
        rho, u, FT = self.macroscopic()
        r, at = RATES, self.at
        s = [0, 0, 0, 0] + [r["s2"]] * 3 + [r["s2b"]] + [r["s2"]] * 2 + [r["s3"]] * 6 + [r["s3b"]] + [r["s4"]] * 3 \
            + [r["s4b"]] * 3 + [r["s5"]] * 3 + [r["s6"]]
        if self.Q == 19:
            s = s[:16] + s[17:20]
        s = torch.tensor(s, dtype=torch.float64, device="cuda").reshape(-1, 1, 1, 1)
        m = (self.M @ self.f.reshape(self.Q, -1)).reshape((self.Q,) + self.shape)
        m += s * (self.equilibrium(rho, u) - m)
        if FT is not None:
            (X, Y, Z), (qxx, qyy, qzz, qxy, qxz, qyz), S2 = FT
            x, y, z = u
            c, te, tn = 1.0 / 3.0, 1.0 / r["s2b"] - 0.5, 1.0 / r["s2"] - 0.5
            Xx, Yy, Zz = X * x, Y * y, Z * z
            t = {1: X, 2: Y, 3: Z, 4: X * y + Y * x - qxy / tn, 5: X * z + Z * x - qxz / tn,
                 6: Y * z + Z * y - qyz / tn,
                 7: 2 * (Xx + Yy + Zz) + 6 * self.p["sigma"] * self.p["G"] ** 2 * S2 / te
                 + 4 * (qxx + qyy + qzz) / (5 * te),
                 8: 2 * (Xx - Yy) - (qxx - qyy) / tn, 9: 2 * (Xx - Zz) - (qxx - qzz) / tn,
                 10: c * X, 11: c * X, 12: c * Y, 13: c * Z, 14: c * Y, 15: c * Z,
                 17: 2 * c * (Xx + Yy), 18: 2 * c * (Xx + Zz), 19: 2 * c * (Yy + Zz)}
            if self.Q == 27:
                t.update({20: c * (Y * z + Z * y), 21: c * (X * z + Z * x), 22: c * (X * y + Y * x), 23: c * c * X,
                          24: c * c * Y, 25: c * c * Z, 26: 2 * c * c * (Xx + Yy + Zz)})
            for k, v in t.items():
                m[at(k)] += (1 - 0.5 * s[at(k)]) * v
        out = self.back(m)
        for i in range(self.Q):
            b = self.opp[i]
            g = self.shift(out[i], self.e[b])
            if not self.open:
                g = torch.where(self.solid_at(b), out[b], g)
                g = torch.where(self.solid, torch.zeros_like(g), g)
            self.f[i] = g


def exact(case, seed):
    if case["kind"] == "batch":
        return [exact(m, seed * 131 + k) for k, m in enumerate(_members(case))]
    x = _Exact(case)
    x.start(*_fields(case, seed))
    for _ in range(case["steps"]):
        x.step()
    if case["out"] == "moments":
        rho, u, _ = x.macroscopic()
        return {"rho": torch.where(x.solid, torch.zeros_like(rho), rho), "u": torch.where(x.solid, torch.zeros_like(u), u)}
    return x.f
