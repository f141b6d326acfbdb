"""Performance cases of the library: what its users have it do, through the public binding.

A pass advances a simulation (or a batch of them, or one iteration of the inverse problem) by the
steps between two looks at it and takes the density and velocity fields into device buffers, or the
observables.  Geometries, equations of state and sizes are those of the paper's set-ups and of this
project's workloads: a drop on a circular cylinder (2D) or a sphere (3D) in a periodic box.

FP32 simulations return their fields in FP32 (the precision the state is held in), FP64 ones in FP64.
"""
import math

import numpy as np
import torch

from paper_1908_04443_gb300 import lbmwet as L
from paper_1908_04443_gb300.autograd import DensityFromWettability

SIGMA = {"CS": 0.12, "PR": 0.11}
EOS_CONST = {"CS": (0.25, 4.0), "PR": (2.0 / 49.0, 2.0 / 21.0)}
OMEGA = 0.344
RATES = dict(s_rho=1.0, s_e=0.8, s_eps=0.8, s_j=1.0, s_q=1.1, s_nu=1.0 / 0.95, s_pi=1.1, s_m=1.1)


# ---- the cases -------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest grid of the configurations: 100 x 100 in FP64, the parity run; a pass is launch
        # and latency bound
        _single("cylinder_100x100_fp64", 100, 100, 1, "fp64", "CS", 0.7, "IVD", 10),
        # Sec. IV.A static drop (300 x 350, Peng-Robinson) with the constant virtual density, one grid
        _single("cylinder_300x350_vd_fp32", 300, 350, 1, "fp32", "PR", 0.86, "VD", 50),
        # the 600 x 400 drop on a cylinder alone, as when one contact angle is wanted
        _single("cylinder_600x400_fp32", 600, 400, 1, "fp32", "CS", 0.6, "IVD", 40),
        # the headline workload: the 24-point wall-parameter sweep of the 600 x 400 grid, one batch
        _batch("sweep24_600x400_fp32", 24, 600, 400, 600, 400, "fp32", "CS", 0.6, 20),
        # 96 uneven square grids of 128 to 512 nodes a side (odd widths among them), one batch
        _batch("batch96_128to512_fp32", 96, 128, 128, 512, 512, "fp32", "CS", 0.7, 16),
        # the sweep in FP64, as a reference run for the FP32 one
        _batch("sweep24_600x400_fp64", 24, 600, 400, 600, 400, "fp64", "CS", 0.6, 4),
        # contact angles, extremes and masses of the sweep, as logged while it runs
        dict(_batch("sweep24_observables", 24, 600, 400, 600, 400, "fp32", "CS", 0.6, 1), kind="observe"),
        # a small 3D drop on a sphere in an odd box (no side a multiple of 4)
        _single("sphere_97x83x75_fp32", 97, 83, 75, "fp32", "CS", 0.7, "IVD", 20),
        # the 64^3 sphere in FP64, the 3D parity run
        _single("sphere_64_fp64", 64, 64, 64, "fp64", "CS", 0.7, "IVD", 4),
        # Sec. IV.C sphere as the paper sets it up (200 x 200 x 280, Peng-Robinson)
        _single("sphere_200x200x280_fp32", 200, 200, 280, "fp32", "PR", 0.86, "IVD", 10),
        # the largest grid of the configurations: the 256^3 sphere
        _single("sphere_256_fp32", 256, 256, 256, "fp32", "CS", 0.7, "IVD", 8),
        # one iteration of fitting the wettability of a 256 x 256 cylinder: forward run with
        # checkpoints, loss on the final density, backward
        dict(kind="adjoint", name="adjoint_256_fp32", nx=256, ny=256, nz=1, precision="fp32", eos="CS", t=0.7,
             wall="IVD", steps=300, every=100),
    ]


def _single(name, nx, ny, nz, precision, eos, t, wall, steps):
    return dict(kind="single", name=name, nx=nx, ny=ny, nz=nz, precision=precision, eos=eos, t=t, wall=wall, steps=steps)


def _batch(name, n, nx0, ny0, nx1, ny1, precision, eos, t, steps):
    """n grids: all nx0 x ny0 when both ends agree, else squares of sides drawn from nx0 .. nx1."""
    return dict(kind="batch", name=name, n=n, nx0=nx0, ny0=ny0, nx1=nx1, ny1=ny1, precision=precision, eos=eos, t=t,
                wall="IVD", steps=steps)


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    eos, t = rng.choice([("CS", 0.7), ("PR", 0.86)])
    kind = rng.choice(["single2", "single2", "batch", "batch", "single3", "single3", "observe", "adjoint"])
    if kind == "single2":
        prec = rng.choice(["fp32", "fp32", "fp64"])
        nx, ny = log_int(48, 1024), log_int(48, 1024)
        c = _single("", nx, ny, 1, prec, eos, t, rng.choice(["IVD", "IVD", "VD", "GF"]), log_int(1, 64))
        c["steps"] = max(1, min(c["steps"], int((2.0e7 if prec == "fp64" else 1.0e8) / (nx * ny))))
    elif kind == "single3":
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        top = 256 if prec == "fp32" else 96
        nx, ny, nz = (log_int(24, top) for _ in range(3))
        c = _single("", nx, ny, nz, prec, eos, t, rng.choice(["IVD", "IVD", "VD"]), log_int(1, 32))
        c["steps"] = max(1, min(c["steps"], int((5.0e6 if prec == "fp64" else 1.2e8) / (nx * ny * nz))))
    elif kind in ("batch", "observe"):
        prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
        n, a = log_int(2, 96), log_int(64, 320)
        b = log_int(a, 512)
        n = max(2, min(n, int(1.0e7 / (a * a + b * b) * 2)))
        c = _batch("", n, a, a if rng.random() < 0.5 else log_int(64, 512), b, b, prec, eos, t, log_int(1, 32))
        if rng.random() < 0.4:   # a sweep: grids of one shape
            c["nx1"], c["ny1"] = c["nx0"], c["ny0"]
        if kind == "observe":
            c["kind"], c["steps"] = "observe", 1
        nodes = n * max(c["nx0"] * c["ny0"], c["nx1"] * c["ny1"])
        c["steps"] = max(1, min(c["steps"], int((2.0e7 if prec == "fp64" else 1.2e8) / nodes)))
    else:
        c = dict(kind="adjoint", nx=log_int(64, 256), ny=log_int(64, 256), nz=1,
                 precision=rng.choice(["fp32", "fp32", "fp64"]), eos="CS", t=0.7, wall="IVD",
                 steps=log_int(20, 200), every=rng.choice([20, 50, 100]))
    c.pop("name", None)
    return c


# ---- inputs ----------------------------------------------------------------------------------------

def _pressure(kind, T, rho):
    a, b = EOS_CONST[kind]
    if kind == "CS":
        eta = b * rho / 4.0
        return rho * T * (1.0 + eta + eta ** 2 - eta ** 3) / (1.0 - eta) ** 3 - a * rho ** 2
    return rho * T / (1.0 - b * rho) - a * _pr_phi(T) * rho ** 2 / (1.0 + 2.0 * b * rho - b ** 2 * rho ** 2)


def _pr_phi(T):
    a, b = EOS_CONST["PR"]
    tc = 0.0778 * a / (0.45724 * b)
    return (1.0 + (0.37464 + 1.54226 * OMEGA - 0.26992 * OMEGA ** 2) * (1.0 - math.sqrt(T / tc))) ** 2


def _temperature(kind, t):
    a, b = EOS_CONST[kind]
    return t * (0.0778 * a / (0.45724 * b) if kind == "PR" else 0.3773 * a / b)


_coexistence_of = {}


def _coexistence(kind, t):
    """Densities of the coexisting phases (rho_g, rho_l): equal pressures, equal areas."""
    key = (kind, t)
    if key in _coexistence_of:
        return _coexistence_of[key]
    T, top = _temperature(kind, t), (0.999 / EOS_CONST["PR"][1] if kind == "PR" else 0.9 * 4.0 / EOS_CONST["CS"][1])
    grid = np.linspace(top * 1e-6, top, 200001)
    p = _pressure(kind, T, grid)
    down = np.flatnonzero(np.diff(p) < 0)
    i1, i2 = int(down[0]), int(down[-1]) + 1       # spinodal densities on the grid
    x, w = np.polynomial.legendre.leggauss(400)

    def root(lo, hi, ps):
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if _pressure(kind, T, mid) < ps else (lo, mid)
        return 0.5 * (lo + hi)

    def densities(ps):
        return root(1e-12, grid[i1], ps), root(grid[i2], top, ps)

    def area(ps):
        g, l = densities(ps)
        s = 0.5 * (math.log(l) - math.log(g))
        r = np.exp(math.log(g) + s * (x + 1.0))
        return float(np.sum(w * s * (_pressure(kind, T, r) - ps) / r))

    lo, hi = max(float(p[i2]), 0.0) + 1e-12, float(p[i1]) - 1e-12
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if area(mid) > 0 else (lo, mid)
    _coexistence_of[key] = densities(0.5 * (lo + hi))
    return _coexistence_of[key]


def _shapes(case):
    """(nx, ny, nz) of every grid of a case; the sides of uneven batches come from the case alone."""
    if case["kind"] in ("single", "adjoint"):
        return [(case["nx"], case["ny"], case["nz"])]
    if (case["nx0"], case["ny0"]) == (case["nx1"], case["ny1"]):
        return [(case["nx0"], case["ny0"], 1)] * case["n"]
    rng = np.random.default_rng(20190812)
    lo, hi = sorted((case["nx0"], case["nx1"]))
    return [(s, s, 1) for s in rng.integers(lo, hi + 1, size=case["n"]).tolist()]


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _inputs(case, seed):
    """Per grid: solid mask, initial density, wall parameter, body and drop (host arrays, as the
    library takes them)."""
    rg, rl = _coexistence(case["eos"], case["t"])
    rng = np.random.default_rng([int(seed) & 0x7FFFFFFF, 77])
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed))
    out = []
    shapes = _shapes(case)
    # the wall scheme's parameters other than kappa are the same for every grid of a batch
    rho_w, theta = rg + (0.3 + 0.4 * rng.random()) * (rl - rg), rng.uniform(60.0, 120.0)
    for i, s in enumerate(shapes):
        d = 2 if s[2] == 1 else 3
        s = s[:d]
        n = min(s)
        # body and drop as in the workloads: a drop of 1.1 to 1.4 body radii set on top of the body
        # (the fit's body is known: its wall nodes are the same for every seed)
        R = (0.15 + (0.0 if case["kind"] == "adjoint" else 0.07) * rng.random()) * n
        r = (1.1 + 0.3 * rng.random()) * R if d == 2 else (1.05 + 0.2 * rng.random()) * R
        c = [0.5 * m for m in s]
        c[-1] = 0.38 * s[-1]
        dc = list(c)
        dc[-1] += R + r + rng.uniform(-0.5, 0.5)
        if case["kind"] in ("batch", "observe") and len(shapes) > 1 and len(set(shapes)) == 1:
            u = i / (len(shapes) - 1.0)                     # a sweep from wetting to repelling
            kappa = 0.5 * (1 - 2 * u) if u < 0.5 else -0.5 * (u - 0.5) * (rl - rg)
            kappa *= 0.9 + 0.1 * rng.random()
        else:
            kappa = rng.uniform(-0.6, 0.6)
            kappa = kappa if kappa >= 0 else kappa * (rl - rg)
        co = torch.meshgrid(*[torch.arange(m, dtype=torch.float64, device=_device()) for m in s[::-1]], indexing="ij")[::-1]
        solid = sum((x - cc) ** 2 for x, cc in zip(co, c)) <= R * R
        d2 = 0.0
        for x, cc, m in zip(co, dc, s):
            dx = x - cc
            dx = dx - m * torch.round(dx / m)
            d2 = d2 + dx * dx
        rho = 0.5 * (rl + rg) + 0.5 * (rl - rg) * torch.tanh(r - torch.sqrt(d2))
        rho = rho + 1e-6 * (2.0 * torch.rand(rho.shape, generator=gen, dtype=torch.float64, device=_device()) - 1.0)
        rho = torch.where(solid, torch.full_like(rho, rg), rho)
        out.append(dict(mask=solid.to(torch.uint8).cpu().numpy(), rho0=rho.cpu().numpy(), kappa=kappa,
                        body=("ball", tuple(c), R), hint=tuple(dc), rho_w=rho_w, theta=theta))
    return out


def _wall_kappa(n, seed):
    """A smooth wall parameter per wall node, the starting point of a fit (phi between 1.02 and about 1.3)."""
    c = np.random.default_rng(int(seed)).normal(size=5)
    ang = np.linspace(0.0, 2 * math.pi, n, endpoint=False)
    return np.clip(0.15 + 0.02 * sum(w * np.cos((k + 1) * ang + k) for k, w in enumerate(c)), 0.02, None)


def _config(case, g):
    a, b = EOS_CONST[case["eos"]]
    rg, rl = _coexistence(case["eos"], case["t"])
    e = L.make_eos(case["eos"], a, b, 1.0, _temperature(case["eos"], case["t"]), OMEGA)
    shape = g["rho0"].shape
    return L.make_config("D2Q9" if len(shape) == 2 else "D3Q19", case["precision"], shape, e, sigma=SIGMA[case["eos"]],
                         rho_l=rl, rho_g=rg, rho_ref=rg, wall=case["wall"], kappa=g["kappa"], rho_w_const=g["rho_w"],
                         theta_a=g["theta"], body=g["body"], drop_hint=g["hint"], **RATES)


class _Batch:
    """An lbm_batch, released with the object."""

    def __init__(self, cfgs, masks, rho0s, stream):
        self.b = L.lbm_batch_init(cfgs, masks, rho0s, None, stream)

    def __del__(self):
        L.lbm_batch_destroy(self.b)


def prepare(case, seed):
    grids = _inputs(case, seed)
    cfgs = [_config(case, g) for g in grids]
    stream = torch.cuda.current_stream()
    st = {"case": case, "steps": case["steps"]}
    if case["kind"] == "adjoint":
        g = grids[0]
        sim = L.Simulation(cfgs[0], g["mask"], g["rho0"], stream=stream)
        st.update(sim=sim, f0=sim.get_state(), kappa=torch.tensor(_wall_kappa(len(sim.wall_nodes()), seed)),
                  target=torch.tensor(g["rho0"], device="cuda"))
        return st
    nodes = [g["mask"].size for g in grids]
    dim = grids[0]["rho0"].ndim
    if case["kind"] == "single":
        st["sim"] = L.Simulation(cfgs[0], grids[0]["mask"], grids[0]["rho0"], stream=stream)
        st["handles"] = [st["sim"].h]
    else:
        st["batch"] = _Batch(cfgs, [g["mask"] for g in grids], [g["rho0"] for g in grids], stream)
        st["handles"] = [L.lbm_batch_handle(st["batch"].b, i) for i in range(len(grids))]
    if case["kind"] != "observe":
        st["rho"] = torch.empty(sum(nodes), dtype=torch.float64, device="cuda")
        st["u"] = torch.empty(dim * sum(nodes), dtype=torch.float64, device="cuda")
        offs = np.cumsum([0] + nodes[:-1]).tolist()
        st["ptrs"] = [(h, st["rho"].data_ptr() + 8 * o, st["u"].data_ptr() + 8 * dim * o)
                      for h, o in zip(st["handles"], offs)]
    return st


# ---- one pass --------------------------------------------------------------------------------------

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "adjoint":
        kappa = st["kappa"].clone().requires_grad_(True)
        rho = DensityFromWettability.apply(kappa, st["sim"], st["f0"], case["steps"], case["every"])
        loss = 0.5 * ((rho - st["target"]) ** 2).sum()
        loss.backward()
        if case["precision"] == "fp32":
            return {"rho": rho.detach().float(), "grad": kappa.grad.float()}
        return {"rho": rho.detach(), "grad": kappa.grad}
    if kind == "single":
        st["sim"].step(st["steps"])
    else:
        L.lbm_batch_step(st["batch"].b, st["steps"])
    if kind == "observe":
        obs = L.lbm_batch_observables(st["batch"].b)
        keep = np.float32 if case["precision"] == "fp32" else np.float64
        return {"mass": np.array([o.mass for o in obs], keep),
                "extremes": np.array([(o.rho_max, o.rho_min) for o in obs], keep),
                "u_max": np.array([o.u_max for o in obs], keep),
                "theta": np.array([o.theta_deg for o in obs], keep),
                "drop": np.array([(o.drop_center[0], o.drop_center[1], o.drop_radius) for o in obs], keep)}
    for h, rho, u in st["ptrs"]:
        L.lbm_fields_device(h, rho, u)
    if case["precision"] == "fp32":
        return {"rho": st["rho"].float(), "u": st["u"].float()}
    return {"rho": st["rho"], "u": st["u"]}


def work(case):
    """Every step reads the distributions of its input state once and writes those of its output state
    once; the fields are written once.  Operations per node update: density, equation of state, force,
    velocity and collision (about 230 in 2D, 480 in 3D)."""
    size = 8 if case["precision"] == "fp64" else 4
    total_b = total_f = 0.0
    for nx, ny, nz in _shapes(case):
        n, q, ops = (nx * ny, 9, 230.0) if nz == 1 else (nx * ny * nz, 19, 480.0)
        step_b, step_f = 2.0 * q * size * n, ops * n
        if case["kind"] == "adjoint":
            # forward, recomputation, and the reverse step (state and adjoint read, adjoint written)
            total_b += case["steps"] * 3.5 * step_b
            total_f += case["steps"] * 4.0 * step_f
        else:
            total_b += case["steps"] * step_b + (q * size + 8.0 * (1 + (2 if nz == 1 else 3))) * n
            total_f += (case["steps"] + 0.5) * step_f
    return {"bytes": total_b, "flops": total_f}


# ---- the same in 64 bits, in plain torch -------------------------------------------------------------

def _lattice(d):
    if d == 2:
        E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        WF = [0.0] + [1 / 3] * 4 + [1 / 12] * 4

        def moments(x, y):
            n = x * x + y * y
            return [1, -4 + 3 * n, 4 - 21 * n / 2 + 9 * n * n / 2, x, (-5 + 3 * n) * x, y, (-5 + 3 * n) * y,
                    x * x - y * y, x * y]
        rates = ["s_rho", "s_e", "s_eps", "s_j", "s_q", "s_j", "s_q", "s_nu", "s_nu"]
    else:
        E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
             (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
             (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
        W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        WF = [0.0] + [1 / 6] * 6 + [1 / 12] * 12

        def moments(x, y, z):
            n = x * x + y * y + z * z
            pxx, pww = 3 * x * x - n, y * y - z * z
            return [1, 19 * n - 30, (21 * n * n - 53 * n + 24) / 2, x, (5 * n - 9) * x, y, (5 * n - 9) * y, z,
                    (5 * n - 9) * z, pxx, (3 * n - 5) * pxx, pww, (3 * n - 5) * pww, x * y, y * z, x * z,
                    pww * x, (z * z - x * x) * y, (x * x - y * y) * z]
        rates = ["s_rho", "s_e", "s_eps", "s_j", "s_q", "s_j", "s_q", "s_j", "s_q", "s_nu", "s_pi", "s_nu", "s_pi",
                 "s_nu", "s_nu", "s_nu", "s_m", "s_m", "s_m"]
    M = np.array([moments(*e) for e in E], dtype=np.float64).T
    opp = [E.index(tuple(-v for v in e)) for e in E]
    return E, W, WF, M, opp, [RATES[k] for k in rates]


class _Exact:
    """One grid in 64 bits: f holds the post-streaming distributions."""

    def __init__(self, case, g):
        self.case, self.g = case, g
        self.rg, self.rl = _coexistence(case["eos"], case["t"])
        self.T = _temperature(case["eos"], case["t"])
        dev = _device()
        self.solid = torch.tensor(g["mask"], device=dev) != 0
        self.fluid = ~self.solid
        self.d = self.solid.dim()
        self.E, self.W, self.WF, M, self.opp, rates = _lattice(self.d)
        self.q = len(self.E)
        self.M = torch.tensor(M, device=dev)
        self.Minv = torch.tensor(np.linalg.inv(M), device=dev)
        col = (self.q,) + (1,) * self.d
        self.lam = torch.tensor(rates, dtype=torch.float64, device=dev).reshape(col)
        s = self.fluid.to(torch.float64)
        self.den = sum(self.WF[a] * self.at(s, a) for a in range(1, self.q))
        self.wall = self.solid & (self.den > 0)
        self.src_fluid = [self.at(self.fluid, self.opp[a]) for a in range(self.q)]
        self.f = torch.stack([w * torch.tensor(g["rho0"], device=dev) for w in self.W]) * s
        self.kappa = g["kappa"]

    def at(self, x, a):
        """x at the neighbour in direction a."""
        return torch.roll(x, tuple(-c for c in self.E[a]), tuple(range(self.d - 1, -1, -1)))

    def psi(self, rho):
        rho = torch.where(rho > 0, rho, torch.full_like(rho, self.rg))
        return torch.sqrt(-2.0 * (_pressure(self.case["eos"], self.T, rho) - rho / 3.0))

    def fields(self):
        rho = self.f.sum(0)
        if self.case["wall"] == "VD":
            rw = torch.full_like(rho, self.g["rho_w"])
        else:
            num = sum(self.WF[a] * self.at(rho, a) for a in range(1, self.q))     # rho is 0 on solids
            ave = num / torch.where(self.wall, self.den, torch.ones_like(self.den))
            k = self.kappa
            if not torch.is_tensor(k):
                k = torch.full_like(rho, k)
            rw = torch.where(k >= 0, (1.0 + k) * ave, ave + k).clamp(self.rg, self.rl)
        psi = self.psi(torch.where(self.wall, rw, rho)) * (self.fluid | self.wall)
        Fm = [0.0] * self.d
        for a in range(1, self.q):
            pn = self.at(psi, a)
            for i in range(self.d):
                if self.E[a][i]:
                    Fm[i] = Fm[i] + (self.WF[a] * self.E[a][i]) * pn
        fl = self.fluid.to(torch.float64)
        Fm = [psi * x * fl for x in Fm]                                             # G = -1
        safe = torch.where(self.fluid, rho, torch.ones_like(rho))
        u = []
        for i in range(self.d):
            j = sum(self.E[a][i] * self.f[a] for a in range(self.q) if self.E[a][i])
            u.append((j + 0.5 * Fm[i]) / safe * fl)
        return rho, safe, psi, Fm, u

    def step(self):
        rho, safe, psi, F, u = self.fields()
        uu = sum(x * x for x in u)
        uF = sum(x * y for x, y in zip(u, F))
        feq, G = [], []
        for a in range(self.q):
            e = self.E[a]
            eu = sum(e[i] * u[i] for i in range(self.d))
            eF = sum(e[i] * F[i] for i in range(self.d))
            feq.append(self.W[a] * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu))
            G.append(self.W[a] * (3.0 * (eF - uF) + 9.0 * eu * eF))
        flat = (self.q, -1)
        m = (self.M @ self.f.reshape(flat)).reshape(self.f.shape)
        meq = (self.M @ torch.stack(feq).reshape(flat)).reshape(self.f.shape)
        S = (self.M @ torch.stack(G).reshape(flat)).reshape(self.f.shape)
        psafe = torch.where(psi > 0, psi, torch.ones_like(psi))
        X = SIGMA[self.case["eos"]] * sum(x * x for x in F) / psafe ** 2
        ce, cp = (12.0, 12.0) if self.d == 2 else (114.0, 33.0)
        add = torch.zeros((self.q,) + (1,) * self.d, dtype=torch.float64, device=X.device)
        add[1], add[2] = ce / (1.0 / RATES["s_e"] - 0.5), -cp / (1.0 / RATES["s_eps"] - 0.5)
        S = S + add * X
        ms = m - self.lam * (m - meq) + (1.0 - 0.5 * self.lam) * S
        fs = (self.Minv @ ms.reshape(flat)).reshape(self.f.shape)
        fl = self.fluid.to(torch.float64)
        self.f = torch.stack([torch.where(self.src_fluid[a], self.at(fs[a], self.opp[a]), fs[self.opp[a]]) * fl
                              for a in range(self.q)])


def _angle(x, rho, u):
    """Extremes, drop circle and contact angle from the interface points (link crossings of the mean
    density more than 3 nodes from a solid)."""
    g, fluid = x.g, x.fluid
    R, (cx, cy) = g["body"][2], g["body"][1]
    near = torch.zeros_like(fluid)
    for dx in range(-3, 4):
        for dy in range(-3, 4):
            if dx * dx + dy * dy <= 9:
                near |= torch.roll(x.solid, (dy, dx), (0, 1))
    mid = 0.5 * (x.rl + x.rg)
    pts = []
    for ax, (ex, ey) in ((1, (1, 0)), (0, (0, 1))):
        rn, ok = torch.roll(rho, -1, ax), fluid & ~near & torch.roll(fluid & ~near, -1, ax)
        cross = ok & ((rho - mid) * (rn - mid) < 0)
        yx = torch.nonzero(cross).to(torch.float64)
        t = ((mid - rho) / torch.where(cross, rn - rho, torch.ones_like(rho)))[cross]
        pts.append(torch.stack([yx[:, 1] + ex * t, yx[:, 0] + ey * t], 1))
    p = torch.cat(pts).cpu().numpy() - np.array(g["hint"])
    size = np.array(rho.shape[::-1], dtype=np.float64)
    p = p - size * np.round(p / size)
    um = float(torch.sqrt(u[0] ** 2 + u[1] ** 2)[fluid].max())
    head = (float(rho[fluid].sum()), float(rho[fluid].max()), float(rho[fluid].min()), um)
    A = np.concatenate([p, np.ones((len(p), 1))], 1)
    sol = np.linalg.lstsq(A, -(p ** 2).sum(1), rcond=None)[0]
    c = -0.5 * sol[:2]
    r = math.sqrt(float(c @ c - sol[2]))
    c = c + np.array(g["hint"])
    Rw = R + 0.5
    cth = (Rw * Rw + r * r - (c[0] - cx) ** 2 - (c[1] - cy) ** 2) / (2.0 * Rw * r)
    return head + (math.degrees(math.acos(min(1.0, max(-1.0, cth)))), float(c[0]), float(c[1]), r)


def exact(case, seed):
    if case["wall"] == "GF":
        return None
    grids = _inputs(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, grids[0], seed)
    rhos, us, rows = [], [], []
    with torch.no_grad():
        for g in grids:
            x = _Exact(case, g)
            for _ in range(case["steps"]):
                x.step()
            rho, _, _, _, u = x.fields()
            if case["kind"] == "observe":
                rows.append(_angle(x, rho, u))
            else:
                rhos.append(rho.reshape(-1))
                us.append(torch.stack(u).reshape(-1))
    if case["kind"] == "observe":
        v = np.array(rows)
        return {"mass": v[:, 0], "extremes": v[:, 1:3], "u_max": v[:, 3], "theta": v[:, 4], "drop": v[:, 5:8]}
    return {"rho": torch.cat(rhos), "u": torch.cat(us)}


def _exact_adjoint(case, g, seed):
    x = _Exact(case, g)
    n = int(x.wall.sum())
    kappa = torch.tensor(_wall_kappa(n, seed), device=x.f.device).requires_grad_(True)
    x.kappa = torch.zeros_like(x.f[0]).masked_scatter(x.wall, kappa)
    for _ in range(case["steps"]):
        x.step()
    rho = x.f.sum(0)
    loss = 0.5 * ((rho - torch.tensor(g["rho0"], device=rho.device)) ** 2).sum()
    loss.backward()
    return {"rho": rho.detach(), "grad": kappa.grad}
