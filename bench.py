"""Benchmark of the fused pseudopotential MRT-LB step with improved virtual-density walls.

Default workload: the 600 x 400 D2Q9 droplet-on-cylinder (cylinder R = 60, drop r = 70, C-S EOS at
0.6 Tc, improved virtual-density walls, FP32 deviation storage) over a sweep of 24 wall
parameters from hydrophilic to hydrophobic, stepped as one batch (one persistent kernel launch per
time step).  One bench step is one lattice Boltzmann time step of every grid.  Metric: MLUPS
(million lattice-node updates per second, all nodes counted).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--workload c2|c2single|c1|c3|c4] [--precision fp32|fp64]

Timing: W untimed steps, then K steps timed with CUDA events on the stream the step kernel is
launched on.  When the distributions of the workload fit in twice the L2 size, the L2 cache is
flushed (a 2 x L2-sized buffer is rewritten) before every timed step, outside the events that
bracket each step; larger workloads (the default sweep: 415 MB) run the K steps back to back
between one pair of events.  Under torchrun (N > 1) every rank runs an independent replica of the
workload (no data-path collective): value = N x nodes x K / the slowest rank's time.
--impl reference times the FP64 CPU oracle on the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import workloads as W  # noqa: E402

METRIC = "MLUPS (million lattice updates per second) of the fused time step"
UNIT = "MLUPS"

# DRAM bytes per launch of the step kernel measured by ncu on the workload below, keyed by a hash
# of the kernel code: when the code changes the figure is stale and reported as null.
NCU_TRAFFIC = {
    # pair_step_batched, 600 x 400 sweep of 24 grids: dram__bytes_read.sum + dram__bytes_write.sum of
    # one launch
    ("c2", "fp32", "6a403a0e20dafb8c"): 374299904,
    # ztma_step, 256^3 sphere: one launch
    ("c3", "fp32", "dacc8f5429e6fca9"): 2802910464,
}


# FP64 floating-point operations per node update of the FP64 batched kernel (step64_batched) on the
# 600 x 400 sweep, from ncu: (2 x DFMA + DADD + DMUL thread instructions of one launch) / nodes =
# (2 x 217,849,056 + 371,237,280 + 169,225,560) / 5,760,000; keyed by a hash of the kernel's code.
FP64_FLOPS_PER_NODE = {
    ("c2", "bb787547f4ebd7ba"): 169.47,
}
# FP64 peak of a GB300 from its unit counts and clock: 1.25 TFLOP/s nominal is 4 FP64 flops (2 FMA) per
# SM per clock at 2.07 GHz, so 152 SMs x 4 x 2.07 GHz = 1258.6 GFLOP/s.
FP64_PEAK_GFLOPS = 152 * 4 * 2.07
# GB300 HBM3e nominal bandwidth (the roofline fractions are against the measured copy rate; this is
# reported beside it)
NOMINAL_HBM_GBS = 7900.0


def _code_hash(files) -> str:
    """Hash of the code of the given csrc files, comments and whitespace removed (a comment edit does
    not make a measured figure stale; any code edit does)."""
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, "paper_1908_04443_gb300", "csrc", f)) as fh:
            src = fh.read()
        src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
        src = re.sub(r"//[^\n]*", " ", src)
        h.update(" ".join(src.split()).encode())
    return h.hexdigest()[:16]


def fp64_kernel_hash() -> str:
    return _code_hash(("step64.cu", "fp64.cuh", "tile_common.cuh", "lattice.cuh", "kernels.h"))   # the FP64 2D kernel's


def kernel_hash() -> str:
    return _code_hash(("step2p.cu", "pack2.cuh", "tile_common.cuh", "lattice.cuh", "kernels.h"))   # the pair kernel's


def ztma_kernel_hash() -> str:
    return _code_hash(("step3p.cu", "pack2.cuh", "tile_common.cuh", "lattice.cuh", "kernels.h"))   # the 3D kernel's


WORKLOADS = ("c2", "c2single", "c1", "c3", "c4")


def workload(name: str):
    """(list of instances, precision, label).  c2: the 600 x 400 cylinder workload over a sweep of
    24 wall parameters (hydrophilic to hydrophobic), run as one batch; c2single: one of them;
    c1: the 100 x 100 FP64 parity grid; c3: the 256^3 D3Q19 sphere; c4: 96 uneven 2D instances."""
    if name == "c1":
        return [W.c1_parity_cylinder()], "fp64", "c1_d2q9_fp64_100x100"
    if name == "c3":
        return [W.c3_sphere_256()], "fp32", "c3_d3q19_256cube_fp32"
    if name == "c4":
        return W.c4_batch(96), "fp32", "c4_batch96_d2q9_128to512_fp32"
    if name == "c2single":
        return [W.c2_cylinder_600x400(kappa=0.15)], "fp32", "c2_d2q9_600x400_fp32_single"
    return None, "fp32", "c2_d2q9_600x400_fp32_sweep24"


def c2_sweep(rho_l, rho_g):
    return [W.c2_cylinder_600x400(kappa=k) for k in W.c2_cylinder_sweep_kappas(rho_l, rho_g)]


def sigma_for(wl) -> float:
    return 0.12


def bytes_per_lu(lattice: str, precision: str) -> int:
    q = 9 if lattice == "D2Q9" else 19
    return 2 * q * (8 if precision == "fp64" else 4)


# ---------------------------------------------------------------------------------------------
# clocks sampled during the timed region
# ---------------------------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.thread.join(timeout=2)

    def summary(self):
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------------------------------------
# the CPU oracle (reported baseline and --impl reference)
# ---------------------------------------------------------------------------------------------

ORACLE_SNIPPET = r"""
import json, sys, time
sys.path.insert(0, {root!r})
import numpy as np
import workloads as W
from oracle import eos as E, lbm
wls = W.{ctor}
wls = wls if isinstance(wls, list) else [wls]
grids, nodes = [], 0
for wl in wls:
    e = (E.cs_config() if wl.eos == "CS" else E.pr_paper()).at_reduced_temperature(wl.t_over_tc)
    g, l = E.maxwell(e)
    if {scale_kappa} and wl.kappa < 0:   # drawn in units of (rho_l - rho_g)
        wl.kappa *= (l - g)
    mask, rho0 = wl.mask(), wl.rho0(l, g)
    crop = {crop}
    if crop:   # a window of the workload (mask and initial density) around the lower part of the body
        # and the gas below it: no liquid-gas interface crosses the window's (periodic) faces
        c = [int(round(v)) for v in wl.body_center[::-1]]
        c[0] -= 24
        win = tuple(slice(ci - crop // 2, ci + crop // 2) for ci in c)
        mask, rho0 = np.ascontiguousarray(mask[win]), np.ascontiguousarray(rho0[win])
    geo = lbm.Geometry(mask, wl.lattice)
    p = lbm.Params(wl.lattice, e, sigma={sigma}, rho_l=l, rho_g=g, kappa=wl.kappa)
    grids.append([geo, p, lbm.init_state(rho0, geo)])
    nodes += int(mask.size)
for _ in range({warmup}):
    for gr in grids:
        gr[2] = lbm.step(gr[2], gr[0], gr[1])
times = []
for _ in range({steps}):
    t = time.perf_counter()
    for gr in grids:
        gr[2] = lbm.step(gr[2], gr[0], gr[1])
    times.append(time.perf_counter() - t)
print(json.dumps({{"times": times, "nodes": nodes}}))
"""


# the 256^3 sphere's oracle sample: a 96^3 window of it around the sphere's lower half
C3_ORACLE_WINDOW = 96
# the 96-grid batch's oracle sample: its first instances, stepped in turn
C4_ORACLE_INSTANCES = 4


def run_oracle(wl_name: str, steps: int, warmup: int, procs: int = 1):
    """Step times of `procs` concurrent single-thread oracle processes (one list per process) and
    the grid's node count."""
    ctor = {"c1": "c1_parity_cylinder()", "c3": "c3_sphere_256()", "c4": f"c4_batch(96)[:{C4_ORACLE_INSTANCES}]"}.get(
        wl_name, "c2_cylinder_600x400(kappa=0.15)")
    crop = C3_ORACLE_WINDOW if wl_name == "c3" else 0
    code = ORACLE_SNIPPET.format(root=ROOT, ctor=ctor, sigma=0.12, warmup=warmup, steps=steps, crop=crop,
                                 scale_kappa=wl_name == "c4")
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1")
    ps = [subprocess.Popen([sys.executable, "-c", code], stdout=subprocess.PIPE, stderr=subprocess.PIPE, text=True,
                           env=env) for _ in range(procs)]
    outs = []
    for pr in ps:
        out, err = pr.communicate()
        if pr.returncode != 0:
            raise RuntimeError(err[-2000:])
        outs.append(json.loads(out.strip().splitlines()[-1]))
    return [d["times"] for d in outs], outs[0]["nodes"]


def cpu_baseline(wl_name: str, target_s: float = 15.0, all_cores: bool = True):
    # estimate the step time from one step, then take a sample of about target_s seconds
    (t1,), nodes = run_oracle(wl_name, 1, 0)
    n = max(1, min(2000, int(target_s / max(t1[0], 1e-4))))
    (times,), nodes = run_oracle(wl_name, n, 0)
    total = sum(times)
    what = (f"a {C3_ORACLE_WINDOW}^3 window of the 256^3 sphere workload (mask and initial density of "
            f"z 28..123 around the sphere's lower half, periodic)" if wl_name == "c3"
            else (f"the first {C4_ORACLE_INSTANCES} instances of the batch ({nodes} nodes), stepped in turn"
                  if wl_name == "c4" else f"one {nodes}-node grid of the workload"))
    res = {"value": round(nodes * n / total / 1e6, 4), "unit": UNIT, "cores": 1, "kind": "oracle",
           "sample": f"{n} FP64 oracle steps of {what}, one thread"}
    procs = os.cpu_count() or 1
    if all_cores and procs > 1:
        # every host core: the workload's grids are independent, so one single-thread oracle
        # process per core, each on a grid of the workload, all at once
        m = max(1, n // 2)
        runs, _ = run_oracle(wl_name, m, 0, procs)
        slowest = max(sum(t) for t in runs)
        res["all_cores"] = {"value": round(procs * nodes * m / slowest / 1e6, 4), "unit": UNIT, "cores": procs,
                            "sample": f"{procs} concurrent single-thread oracle processes, {m} steps each of one "
                                      f"{nodes}-node grid of the workload (rate over the slowest process)"}
    return res


# ---------------------------------------------------------------------------------------------
# error against the FP64 oracle: one step from the GPU's own state (the GPU steps once more; the
# oracle steps the same state), on a sampled instance or, for the 256^3 sphere, on windows around
# sampled nodes (one step's output at a node depends on the state within 3 nodes)
# ---------------------------------------------------------------------------------------------

def oracle_params(wl):
    from oracle import eos as E, lbm
    e = (E.cs_config() if wl.eos == "CS" else E.pr_paper()).at_reduced_temperature(wl.t_over_tc)
    g, l = E.maxwell(e)
    return lbm.Params(wl.lattice, e, sigma=sigma_for(wl), rho_l=l, rho_g=g, kappa=wl.kappa)


def err_one_step(L, h, wl, step_once, windows=0, seed=3):
    """max |f_gpu - f_oracle| / max |f_oracle| after one step from the GPU state of handle h (the
    step is taken by step_once(), which may step a whole batch)."""
    from oracle import lbm
    q = 9 if wl.lattice == "D2Q9" else 19
    before = L.lbm_get_state(h, q, wl.nodes).reshape((q,) + wl.shape)
    step_once()
    after = L.lbm_get_state(h, q, wl.nodes).reshape((q,) + wl.shape)
    p = oracle_params(wl)
    mask = wl.mask()
    if not windows:
        ref = lbm.step(before, lbm.Geometry(mask, wl.lattice), p)
        return {"max_rel": float(np.max(np.abs(after - ref)) / np.max(np.abs(ref))), "nodes": "all",
                "definition": "one step from a common state: max |f_gpu - f_oracle| / max |f_oracle|"}
    rng = np.random.default_rng(seed)
    fluid = np.argwhere(mask == 0)
    r = 7
    worst, ref_max, used = 0.0, 0.0, 0
    for z, y, x in fluid[rng.choice(len(fluid), windows, replace=False)]:
        win = np.ix_(*[np.arange(c - r, c + r + 1) % n for c, n in zip((z, y, x), wl.shape)])
        ref = lbm.step(before[(slice(None),) + win], lbm.Geometry(mask[win], wl.lattice), p)[:, r, r, r]
        worst = max(worst, float(np.max(np.abs(after[:, z, y, x] - ref))))
        ref_max = max(ref_max, float(np.max(np.abs(ref))))
        used += 1
    return {"max_rel": worst / ref_max, "nodes": f"{used} sampled fluid nodes (15^3 oracle windows)",
            "definition": "one step from a common state: max |f_gpu - f_oracle| / max |f_oracle|"}


# ---------------------------------------------------------------------------------------------
# our arm
# ---------------------------------------------------------------------------------------------

def slowest_rank_ms(local_ms, dist, torch, device):
    """The timed region's length on the slowest rank (max over ranks; the local value without a
    process group)."""
    if dist is None:
        return local_ms
    t = torch.tensor([local_ms], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_rate(world, nodes_per_rank, steps, total_ms):
    """Whole-job MLUPS of `world` replicas, each updating `nodes_per_rank` nodes `steps` times."""
    return world * nodes_per_rank * steps / (total_ms * 1e-3) / 1e6


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


STEP_KERNEL = "auto"   # --step-kernel


def make_cfg(L, wl, precision, rho_g, rho_l):
    e = L.make_eos(wl.eos, 0.25, 4.0, 1.0, 0.0)
    e.T = wl.t_over_tc * L.lbm_critical_temperature(e)
    return L.make_config(wl.lattice, precision, wl.shape, e, sigma=sigma_for(wl), rho_l=rho_l, rho_g=rho_g,
                         kappa=wl.kappa, rho_ref=rho_g, body=("ball", wl.body_center, wl.body_radius),
                         drop_hint=wl.drop_center, step_kernel=STEP_KERNEL)


class Runner:
    """One grid (lbm_handle) or several (lbm_batch) behind the same few calls."""

    def __init__(self, L, cfgs, masks, rho0s, stream):
        self.L = L
        self.batch = len(cfgs) > 1
        self.lattice3 = cfgs[0].lattice == 1
        self.fp64 = cfgs[0].precision == L.LBM_FP64
        if self.batch:
            self.b = L.lbm_batch_init(cfgs, masks, rho0s, None, stream)
            self.handles = [L.lbm_batch_handle(self.b, i) for i in range(len(cfgs))]
        else:
            self.b = None
            self.h = L.lbm_init(cfgs[0], masks[0], rho0s[0], None, None, stream)
            self.handles = [self.h]

    def enqueue(self, n):
        if self.batch:
            self.L.lbm_batch_enqueue_steps(self.b, n)
        else:
            self.L.lbm_enqueue_steps(self.h, n)

    def step(self, n):
        if self.batch:
            self.L.lbm_batch_step(self.b, n)
        else:
            self.L.lbm_step(self.h, n)

    def launches(self):
        return self.L.lbm_batch_kernel_launches(self.b) if self.batch else self.L.lbm_kernel_launches(self.h)

    def kernel_name(self):
        """Name of the step kernel this run launches."""
        k = self.L.lbm_batch_step_kernel_used(self.b) if self.batch else self.L.lbm_step_kernel_used(self.h)
        if k == "ztma":
            return "ztma_step"
        if self.lattice3:
            return "step3d64" if self.fp64 else "zpair_step" if k == "pair" else "zmarch_step"
        if k == "ymarch":
            return "ymarch_step"
        if k == "pair":
            return "pair_step_batched" if self.batch else "pair_step"
        if k == "tile":
            if self.fp64:
                return "step64_batched" if self.batch else "step64"
            return "fused_step_batched" if self.batch else "fused_step"
        return "zmarch_step"

    def close(self):
        if self.batch:
            self.L.lbm_batch_destroy(self.b)
        else:
            self.L.lbm_destroy(self.h)


def adjoint_c5(L, torch, stream, steps=2000, ckpt=100, n_fd=8, dk=1e-3):
    """The 256 x 256 adjoint workload as configured: per-wall-node wettability kappa_j on a cylinder of
    radius 40 (kappa = 0.1 everywhere), loss L = sum over fluid nodes of (rho_T - rho_target)^2 after
    2000 steps, where rho_target comes from the same run with kappa_j = 0.1 + a seeded smooth random
    function of the polar angle (4 modes, amplitude 0.2, seed 7).  The FP32 forward pass with
    checkpoints every 100 steps (lbm_record) and the gradient (lbm_adjoint: segment recomputation +
    reverse sweep) are timed with CUDA events; the gradient is checked against FP64 central finite
    differences of L at n_fd wall nodes spread around the cylinder."""
    wl = W.c5_adjoint_256()
    e = L.make_eos("CS", 0.25, 4.0, 1.0, 0.0)
    e.T = wl.t_over_tc * L.lbm_critical_temperature(e)
    rho_g, rho_l = L.lbm_coexistence(e)
    mask = wl.mask()
    fl = (mask.reshape(-1) == 0)
    rho0 = wl.rho0(rho_l, rho_g)
    h64 = L.lbm_init(make_cfg(L, wl, "fp64", rho_g, rho_l), mask, rho0, None, None, stream)
    idx = L.lbm_wall_nodes(h64)
    nw = len(idx)
    cx, cy = wl.body_center
    ang = np.arctan2(idx // wl.shape[1] - cy, idx % wl.shape[1] - cx)
    kap0 = np.full(nw, float(wl.kappa))
    kap_t = wl.kappa + W.smooth_polar_field(ang)
    f0 = L.lbm_get_state(h64, 9, wl.nodes)

    def rho_after(h, kap):
        L.lbm_set_kappa(h, kap)
        L.lbm_set_state(h, f0, 0)
        L.lbm_step(h, steps)
        rho = np.empty(wl.nodes)
        L.lbm_observables(h, rho, None)
        return rho

    rho_t = rho_after(h64, kap_t)

    def loss64(kap):
        d = (rho_after(h64, kap) - rho_t)[fl]
        return float(np.dot(d, d))

    # FP32 forward with checkpoints and the adjoint gradient at kappa0
    h32 = L.lbm_init(make_cfg(L, wl, "fp32", rho_g, rho_l), mask, rho0, None, None, stream)
    L.lbm_set_kappa(h32, kap0)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(4)]
    with torch.cuda.stream(stream):
        ev[0].record(stream)
        L.lbm_record(h32, steps, ckpt)
        ev[1].record(stream)
    rho = torch.empty(wl.nodes, dtype=torch.float64, device="cuda")
    L.lbm_fields_device(h32, rho.data_ptr(), None)
    torch.cuda.synchronize()
    target = torch.as_tensor(rho_t, device="cuda")
    drho = 2.0 * (rho - target) * torch.as_tensor(fl, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ev[2].record(stream)
        g32 = L.lbm_adjoint(h32, drho.data_ptr(), nw)
        ev[3].record(stream)
    torch.cuda.synchronize()
    fwd = ev[0].elapsed_time(ev[1])
    adj = ev[2].elapsed_time(ev[3])
    # FP64 central differences at wall nodes spread around the cylinder
    picks = [int(k) for k in np.linspace(0, nw - 1, n_fd).round()]
    g_fd = []
    for j in picks:
        kp, km = kap0.copy(), kap0.copy()
        kp[j] += dk
        km[j] -= dk
        g_fd.append((loss64(kp) - loss64(km)) / (2.0 * dk))
    g_fd = np.array(g_fd)
    g_ad = g32[picks]
    scale = float(np.max(np.abs(g_fd)))
    L.lbm_destroy(h32)
    L.lbm_destroy(h64)
    return {"workload": f"c5_adjoint_256x256_fp32 ({steps} steps, checkpoint every {ckpt}, {nw} wall nodes)",
            "loss": "sum over fluid nodes of (rho_T - rho_target)^2; target from kappa = 0.1 + smooth polar "
                    "field (4 modes, amplitude 0.2, seed 7)",
            "forward_ms": round(fwd, 3), "adjoint_ms": round(adj, 3), "ratio": round(adj / fwd, 3),
            "note": "adjoint = recomputation of each checkpoint segment + the reverse sweep; forward = "
                    "the checkpointed forward pass",
            "err_vs_oracle": {"max_rel": float(np.max(np.abs(g_ad - g_fd)) / scale) if scale > 0 else None,
                              "definition": f"FP32 adjoint dL/dkappa_j against FP64 central differences "
                                            f"(dkappa = {dk}) at {n_fd} wall nodes, max |diff| / max |FD|",
                              "fd": [float(v) for v in g_fd], "adjoint": [float(v) for v in g_ad]}}


def batched_vs_separate(L, torch, stream, run, cfgs, masks, rho0s, steps):
    """One batched launch per step against one launch per instance per step (no L2 flush)."""
    seps = [L.lbm_init(c, m, r, None, None, stream) for c, m, r in zip(cfgs, masks, rho0s)]

    def timed(fn):
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            fn(2)
            torch.cuda._sleep(int(2e6 + 4e5 * steps))
            ev0.record(stream)
            fn(steps)
            ev1.record(stream)
        torch.cuda.synchronize()
        return ev0.elapsed_time(ev1) / steps

    def sep(n):
        for _ in range(n):
            for h in seps:
                L.lbm_enqueue_steps(h, 1)

    ms_b = timed(run.enqueue)
    ms_s = timed(sep)
    for h in seps:
        L.lbm_destroy(h)
    return {"instances": len(cfgs), "steps": steps, "batched_ms_per_step": round(ms_b, 5),
            "separate_ms_per_step": round(ms_s, 5), "speedup": round(ms_s / ms_b, 3),
            "note": "one batched launch per step vs one launch per instance per step; L2 not flushed"}


GOLDEN_C2 = os.path.join(ROOT, "tests", "golden", "c2_600x400_kappa0.15_20000.npz")


def err_c2_golden(L, stream):
    """The 600 x 400 workload (kappa = 0.15, 0.6 Tc) run for its 20000 steps in FP32 on one grid with the
    bench's step kernel, against the FP64 oracle's stored result (tests/golden, written by a script
    that calls only the oracle): the density error split into bulk nodes (relative) and the interface
    band (in units of rho_l), and the contact angle."""
    from tests.fp32_bounds import split_errors
    ref = np.load(GOLDEN_C2)
    rho_g, rho_l = float(ref["rho_g"]), float(ref["rho_l"])
    wl = W.c2_cylinder_600x400(kappa=float(ref["kappa"]))
    cfg = make_cfg(L, wl, "fp32", rho_g, rho_l)
    t0 = time.perf_counter()
    with L.Simulation(cfg, wl.mask(), wl.rho0(rho_l, rho_g), None, None, stream) as sim:
        sim.step(int(ref["steps"]))
        o, rho, _ = sim.observables(fields=True)
        kernel = sim.step_kernel()
    sec = time.perf_counter() - t0
    bulk, band, nb, ni = split_errors(rho, ref["rho"], wl.mask(), rho_l, rho_g)
    return {"steps": int(ref["steps"]), "kernel": kernel, "bulk_max_rel": float(bulk), "bulk_nodes": int(nb),
            "band_max_over_rho_l": float(band), "band_nodes": int(ni),
            "theta_deg": round(o.theta_deg, 6), "theta_oracle_deg": round(float(ref["theta_deg"]), 6),
            "mass_rel": float(abs(o.mass / float(ref["mass"]) - 1)), "seconds": round(sec, 3),
            "definition": "FP32 GPU vs the stored FP64 oracle result after the workload's 20000 steps: max "
                          "|drho|/rho at bulk nodes (more than 3 nodes from the rho_mid contour and from solids), "
                          "max |drho|/rho_l in that interface band"}


GOLDEN_D3 = os.path.join(ROOT, "tests", "golden", "d3q19_sphere64_1000.npz")


def err_d3_golden(L, stream):
    """A 64^3 drop on a sphere (the 256^3 sphere scaled by 1/4, drop radius 16, 0.7 Tc, kappa = 0.2) run
    for 1000 steps in FP32 with the default D3Q19 step (the same TMA z-march as the 256^3 line), against
    the FP64 oracle's stored result: the split density errors and the contact angle."""
    from tests.fp32_bounds import split_errors
    ref = np.load(GOLDEN_D3)
    rho_g, rho_l = float(ref["rho_g"]), float(ref["rho_l"])
    wl = W.sphere_drop_64(int(ref["steps"]))
    cfg = make_cfg(L, wl, "fp32", rho_g, rho_l)
    t0 = time.perf_counter()
    with L.Simulation(cfg, wl.mask(), wl.rho0(rho_l, rho_g), None, None, stream) as sim:
        sim.step(int(ref["steps"]))
        o, rho, _ = sim.observables(fields=True)
        kernel = sim.step_kernel()
    sec = time.perf_counter() - t0
    bulk, band, nb, ni = split_errors(rho, ref["rho"], wl.mask(), rho_l, rho_g)
    return {"workload": wl.name, "steps": int(ref["steps"]), "kernel": kernel, "bulk_max_rel": float(bulk),
            "bulk_nodes": int(nb), "band_max_over_rho_l": float(band), "band_nodes": int(ni),
            "theta_deg": round(o.theta_deg, 6), "theta_oracle_deg": round(float(ref["theta_deg"]), 6),
            "mass_rel": float(abs(o.mass / float(ref["mass"]) - 1)), "seconds": round(sec, 3),
            "definition": "FP32 GPU vs the stored FP64 oracle result after 1000 steps of a 64^3 drop on a sphere "
                          "(the 256^3 grid is beyond the oracle): the split errors as for the 600 x 400 grid"}


def paper_context(L, stream, steps=30000):
    """The paper's own static contact angles for its improved scheme (Fig. 5) and its spurious-current
    level (Fig. 10), quoted beside the same runs here: the Sec. IV.A cylinder (300 x 350, PR at 0.86 Tc,
    R = 70 at (150, 130), drop r = 50 at (150, 230)), sigma = 0.11, FP32, 30000 steps.  Context, not
    parity: the paper prints neither sigma nor the relaxation rates."""
    e = L.make_eos("PR", 2.0 / 49.0, 2.0 / 21.0, 1.0, 0.0, omega=0.344)
    e.T = 0.86 * L.lbm_critical_temperature(e)
    g, l = L.lbm_coexistence(e)
    shape, c, R, d, r = (350, 300), (150.0, 130.0), 70.0, (150.0, 230.0), 50.0
    mask = W.ball_mask(shape, c, R)
    rho0 = np.where(mask != 0, g, W.tanh_drop_density(shape, d, r, l, g) + W.density_noise(shape))
    cases = []
    for kappa, label, paper in ((0.4, "phi = 1.4", 34.0), (0.0, "phi = 1", 88.0), (-0.5, "drho = 0.5", 125.0)):
        cfg = L.make_config("D2Q9", "fp32", shape, e, sigma=0.11, rho_l=l, rho_g=g, kappa=kappa, rho_ref=g,
                            body=("ball", c, R), drop_hint=d)
        with L.Simulation(cfg, mask, rho0, None, None, stream) as sim:
            sim.step(steps)
            o = sim.observables()[0]
        cases.append({"scheme": f"IVD, {label}", "theta_deg": round(o.theta_deg, 2), "paper_theta_deg": paper,
                      "u_max": round(o.u_max, 5), "rho_min": round(o.rho_min, 4), "rho_max": round(o.rho_max, 4)})
    return {"workload": "Sec. IV.A cylinder 300 x 350, PR 0.86 Tc, FP32, 30000 steps", "cases": cases,
            "coexistence": {"rho_g": round(g, 4), "rho_l": round(l, 4)},
            "paper_u_max": "Fig. 10: below 0.006 for the virtual-density schemes",
            "note": "context only: the paper does not print sigma or the relaxation rates (sigma = 0.11 here, "
                    "calibrated on a flat interface; sigma = 0.09 brings the three angles within 4 degrees)"}


def observables_rate(L, torch, run, wls, precision, stream, calls=20):
    """The observables (mass, density extremes, max |u|, contact angle: on demand, not per step)
    through the public call without fields, on every instance of the run: wall time per call after
    warm-up, against the minimum of one read of the distributions (Q values per node); with the
    fields pass of the first instance alone (device time) and its reductions through the
    allocation-free call (wall time: two kernels, an 18-double copy and a synchronisation)."""
    obs = (lambda: L.lbm_batch_observables(run.b)) if run.batch else (lambda: L.lbm_observables(run.handles[0]))
    for _ in range(3):
        obs()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(calls):
        obs()
    ms = (time.perf_counter() - t0) / calls * 1e3
    h, n0 = run.handles[0], wls[0].nodes
    d = 2 if wls[0].lattice == "D2Q9" else 3
    rho = torch.empty(n0, dtype=torch.float64, device="cuda")
    u = torch.empty(d * n0, dtype=torch.float64, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for _ in range(3):
        L.lbm_fields_device(h, rho.data_ptr(), u.data_ptr())
    torch.cuda.synchronize()
    ev[0].record(stream)     # the library's stream, on which the fields pass runs
    for _ in range(calls):
        L.lbm_fields_device(h, rho.data_ptr(), u.data_ptr())
    ev[1].record(stream)
    torch.cuda.synchronize()
    fields_ms = ev[0].elapsed_time(ev[1]) / calls
    for _ in range(3):
        L.lbm_observables_noalloc(h, rho.data_ptr(), u.data_ptr())
    t0 = time.perf_counter()
    for _ in range(calls):
        L.lbm_observables_noalloc(h, rho.data_ptr(), u.data_ptr())
    reduce_ms = (time.perf_counter() - t0) / calls * 1e3
    q = 9 if d == 2 else 19
    nodes = sum(wl.nodes for wl in wls)
    min_bytes = q * (8 if precision == "fp64" else 4) * nodes
    peak = 6800.0
    pk_path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pk_path):
        with open(pk_path) as fh:
            peak = json.load(fh).get("hbm_gbs", peak)
    gbs = min_bytes / (ms * 1e-3) / 1e9
    return {"call": "lbm_batch_observables" if run.batch else "lbm_observables", "instances": len(wls),
            "ms_per_call": round(ms, 4), "algorithmic_bytes": min_bytes, "achieved_gbs": round(gbs, 1),
            "frac_of_measured_hbm": round(gbs / peak, 4),
            "first_instance": {"nodes": n0, "fields_pass_ms": round(fields_ms, 4),
                               "reductions_noalloc_ms": round(reduce_ms, 4)},
            "definition": "wall time per call without fields (fields pass, reductions, contact-angle fit, one "
                          "synchronisation) over the minimum of one read of f (Q x 4 B per node in FP32)"}


def paper_context_3d(L, stream, steps=30000, samples=(20000, 25000, 30000)):
    """The paper's static contact angles on a sphere (Sec. IV.C, Fig. 14: phi = 1.2, phi = 1 and drho =
    0.55 give 53, 88 and 145 degrees) beside the same runs here: 200 x 200 x 280 D3Q19, sphere R = 50,
    drop r = 45, PR at 0.86 Tc, sigma = 0.11 as in 2D, FP32 with the default D3Q19 step, the angle
    read at a few late steps (the hydrophobic drop still moves).  Context, not parity."""
    e = L.make_eos("PR", 2.0 / 49.0, 2.0 / 21.0, 1.0, 0.0, omega=0.344)
    e.T = 0.86 * L.lbm_critical_temperature(e)
    g, l = L.lbm_coexistence(e)
    cases = []
    t0 = time.perf_counter()
    for kappa, label, paper in ((0.2, "phi = 1.2", 53.0), (0.0, "phi = 1", 88.0), (-0.55, "drho = 0.55", 145.0)):
        wl = W.sphere_fig14(kappa, steps)
        cfg = L.make_config("D3Q19", "fp32", wl.shape, e, sigma=0.11, rho_l=l, rho_g=g, kappa=kappa, rho_ref=g,
                            body=("ball", wl.body_center, wl.body_radius), drop_hint=wl.drop_center)
        th = []
        with L.Simulation(cfg, wl.mask(), wl.rho0(l, g), None, None, stream) as sim:
            done = 0
            for s_ in samples:
                sim.step(s_ - done)
                done = s_
                o = sim.observables()[0]
                th.append(o.theta_deg)
            kernel = sim.step_kernel()
        cases.append({"scheme": f"IVD, {label}", "theta_deg": round(th[-1], 2), "paper_theta_deg": paper,
                      "theta_range_deg": [round(min(th), 2), round(max(th), 2)], "at_steps": list(samples),
                      "u_max": round(o.u_max, 5), "rho_min": round(o.rho_min, 4), "rho_max": round(o.rho_max, 4),
                      "kernel": kernel})
    return {"workload": f"Sec. IV.C sphere 200 x 200 x 280, PR 0.86 Tc, FP32, {steps} steps", "cases": cases,
            "coexistence": {"rho_g": round(g, 4), "rho_l": round(l, 4)}, "seconds": round(time.perf_counter() - t0, 1),
            "note": "context only: sigma and the relaxation rates are the 2D readings; the drho = 0.55 drop keeps "
                    "moving on the sphere, its angle swinging by about 20 degrees between samples"}


def e2e_rate(L, cfgs, masks, rho0s, wls, steps, stream, world=1):
    """The metric end to end through the public API with host buffers: init from the host mask and
    initial density, `steps` calls of the stepping entry point with one step each (each reads back
    the 4-byte device status), then the observables with the host density and velocity fields of
    every instance.  The host buffers (inputs and outputs) are pinned and allocated before the timed
    region, as a caller streaming runs through the library would keep them."""
    import torch
    keep = []

    def pinned(a):
        t = torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
        keep.append(t)
        return t.numpy()

    dim = 2 if wls[0].lattice == "D2Q9" else 3
    masks_p = [pinned((np.asarray(m) != 0).astype(np.uint8)) for m in masks]
    rho0s_p = [pinned(np.asarray(r, dtype=np.float64)) for r in rho0s]
    outs = [(pinned(np.zeros(wl.nodes)), pinned(np.zeros(wl.nodes * dim))) for wl in wls]

    def once():
        t0 = time.perf_counter()
        r2 = Runner(L, cfgs, masks_p, rho0s_p, stream)
        t_init = time.perf_counter() - t0
        for _ in range(steps):
            r2.step(1)
        t_steps = time.perf_counter() - t0 - t_init
        if r2.batch:        # one call, one synchronisation for the whole batch
            L.lbm_batch_observables_fields(r2.b, [o[0] for o in outs], [o[1] for o in outs])
        else:
            L.lbm_observables(r2.h, outs[0][0], outs[0][1])
        r2.close()
        e2e_s = time.perf_counter() - t0
        return e2e_s, {"init": round(1e3 * t_init, 2), "steps": round(1e3 * t_steps, 2),
                       "observables_and_destroy": round(1e3 * (e2e_s - t_init - t_steps), 2)}

    nodes = sum(wl.nodes for wl in wls)
    rate = lambda sec: round(world * nodes * steps / sec / 1e6, 2)
    # cold: the library's device memory pool emptied first, so the set-up maps fresh memory
    L.lbm_release_cached_memory()
    cold_s, cold_parts = once()
    warm_s, warm_parts = once()
    d2h = 4 * steps + sum(r.nbytes + u.nbytes + 8 * 18 for r, u in outs)
    h2d = sum(m.size + r.size * 8 for m, r in zip(masks, rho0s))
    return {"value": rate(cold_s), "unit": UNIT,
            "h2d_bytes_per_step": round(h2d / steps, 1), "d2h_bytes_per_step": round(d2h / steps, 1),
            "seconds": round(cold_s, 4), "breakdown_ms": cold_parts,
            "warm_pool": {"value": rate(warm_s), "seconds": round(warm_s, 4), "breakdown_ms": warm_parts,
                          "note": "the same run again with the device memory pool holding the first run's memory"},
            "definition": "init from pinned host mask/rho0 + K x step(1) (4-byte status read each) + "
                          "observables with pinned host rho and u of every instance (one batched call) + destroy; "
                          "value: first run after the library's memory pool was emptied"}


def device_rate(L, torch, stream, name, steps, flush, precision=None, extras=None, autotune=False):
    """Device-timed MLUPS and HBM-roofline fraction of another workload (same protocol as the
    headline: L2 flushed before each timed step when the state fits in L2, else back-to-back steps
    between one pair of events); `precision` overrides the workload's.  Adds the fluid-only rate,
    the error against the FP64 oracle (one step from the GPU state of instance 0) and, through
    `extras(run, wls, cfgs, masks, rho0s)`, workload-specific fields."""
    wls, prec0, label = workload(name)
    precision = precision or prec0
    if precision != prec0:
        label = label.replace("_fp32", "") + "_" + precision
    e = L.make_eos("CS", 0.25, 4.0, 1.0, 0.0)
    e.T = (wls[0].t_over_tc if wls else 0.6) * L.lbm_critical_temperature(e)
    rho_g, rho_l = L.lbm_coexistence(e)
    if wls is None:
        wls = c2_sweep(rho_l, rho_g)
    if name == "c4":
        for wl in wls:
            if wl.kappa < 0:
                wl.kappa *= (rho_l - rho_g)
    cfgs = [make_cfg(L, wl, precision, rho_g, rho_l) for wl in wls]
    masks = [wl.mask() for wl in wls]
    rho0s = [wl.rho0(rho_l, rho_g) for wl in wls]
    run = Runner(L, cfgs, masks, rho0s, stream)
    nodes = sum(wl.nodes for wl in wls)
    fluid = int(sum(int((m == 0).sum()) for m in masks))
    tuning = None
    if autotune and run.batch:
        report = L.lbm_batch_autotune(run.b, 16)
        kinds = [L.lbm_batch_instance_kernel(run.b, i) for i in range(len(wls))]
        tuning = {"report": report.strip().splitlines(),
                  "instances_per_kernel": {k: kinds.count(k) for k in sorted(set(kinds))}}
    with torch.cuda.stream(stream):
        run.enqueue(3)
    run.step(0)
    l2 = torch.cuda.get_device_properties(torch.cuda.current_device()).L2_cache_size
    use_flush = bytes_per_lu(wls[0].lattice, precision) * nodes < 2 * l2
    st = [torch.cuda.Event(enable_timing=True) for _ in range(steps if use_flush else 1)]
    en = [torch.cuda.Event(enable_timing=True) for _ in range(steps if use_flush else 1)]
    with torch.cuda.stream(stream):
        torch.cuda._sleep(int(2e6 + 4e5 * steps))
        if use_flush:
            for k in range(steps):
                flush.zero_()
                st[k].record(stream)
                run.enqueue(1)
                en[k].record(stream)
        else:
            st[0].record(stream)
            run.enqueue(steps)
            en[0].record(stream)
    torch.cuda.synchronize()
    run.step(0)
    ms = sum(a.elapsed_time(b) for a, b in zip(st, en)) / steps
    kernel = run.kernel_name()
    err = err_one_step(L, run.handles[0], wls[0], lambda: run.step(1), windows=40 if wls[0].nodes > 4e6 else 0)
    more = extras(run, wls, cfgs, masks, rho0s) if extras else {}
    run.close()
    peak = 6800.0
    pk_path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pk_path):
        with open(pk_path) as fh:
            peak = json.load(fh).get("hbm_gbs", peak)
    gbs = bytes_per_lu(wls[0].lattice, precision) * nodes / (ms * 1e-3) / 1e9
    out = {"workload": label, "kernel": kernel, "nodes": nodes, "fluid_nodes": fluid, "steps": steps,
           "ms_per_step": round(ms, 5),
           "l2": "flushed before each timed step" if use_flush else "inputs larger than L2, no flush",
           "value": round(nodes / (ms * 1e-3) / 1e6, 1), "unit": UNIT,
           "fluid_only_value": round(fluid / (ms * 1e-3) / 1e6, 1), "achieved_gbs": round(gbs, 1),
           "frac_of_measured_hbm": round(gbs / peak, 4), "frac_of_measured_hbm_fluid_only": round(gbs * fluid / nodes / peak, 4),
           "frac_of_nominal_hbm": round(gbs / NOMINAL_HBM_GBS, 4), "bound": "hbm", "err_vs_oracle": err}
    if tuning:
        out["autotune"] = tuning
    out.update(more)
    if precision == "fp64":
        # GB300's FP64 rate is far below its FP32 rate: the FP64 step is bound by the FP64 pipe
        fpn = FP64_FLOPS_PER_NODE.get((name, fp64_kernel_hash()))
        fp64_peak = L.lbm_probe_fp64_rate(stream)
        out["bound"] = "alu"
        out["alu_roofline"] = {
            "flops_per_node": fpn, "unit": "GFLOP/s", "peak": round(fp64_peak, 1),
            "peak_source": "measured: lbm_probe_fp64_rate (independent FP64 FMA chains, 16 CTAs per SM)",
            "nominal_peak": round(FP64_PEAK_GFLOPS, 1),
            "achieved": None if fpn is None else round(fpn * nodes / (ms * 1e-3) / 1e9, 1),
            "frac": None if fpn is None else round(fpn * nodes / (ms * 1e-3) / 1e9 / fp64_peak, 4)}
    return out


def run_ours(args):
    import torch
    world, rank, local = dist_setup()
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group(backend="nccl", device_id=torch.device("cuda", local))
    from paper_1908_04443_gb300 import build as B
    if rank == 0 or world == 1:
        B.build()
    if dist is not None:
        dist.barrier()
    from paper_1908_04443_gb300 import lbmwet as L

    wls, precision, label = workload(args.workload)
    if args.precision:
        precision = args.precision
    e = L.make_eos("CS", 0.25, 4.0, 1.0, 0.0)
    tc = L.lbm_critical_temperature(e)
    t_over_tc = 0.6 if args.workload in ("c2", "c2single") else (wls[0].t_over_tc)
    e.T = t_over_tc * tc
    rho_g, rho_l = L.lbm_coexistence(e)
    if wls is None:
        wls = c2_sweep(rho_l, rho_g)
    if args.workload == "c4":
        # negative draws are drho in units of (rho_l - rho_g)
        for wl in wls:
            if wl.kappa < 0:
                wl.kappa *= (rho_l - rho_g)
    lattice = wls[0].lattice
    cfgs = [make_cfg(L, wl, precision, rho_g, rho_l) for wl in wls]
    masks = [wl.mask() for wl in wls]
    fluid = int(sum(int((m == 0).sum()) for m in masks))
    rho0s = [wl.rho0(rho_l, rho_g) for wl in wls]
    nodes = sum(wl.nodes for wl in wls)
    stream = torch.cuda.Stream()
    run = Runner(L, cfgs, masks, rho0s, stream)

    l2 = torch.cuda.get_device_properties(local).L2_cache_size
    flush = torch.empty(max(2 * l2, 256 << 20), dtype=torch.uint8, device="cuda")
    state_bytes = 2 * bytes_per_lu(lattice, precision) // 2 * nodes      # both distribution buffers
    use_flush = state_bytes < 2 * l2

    with torch.cuda.stream(stream):
        run.enqueue(args.warmup)
    run.step(0)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    launches0 = run.launches()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        t_wall = time.perf_counter()
        with torch.cuda.stream(stream):
            # a bounded spin (torch's sleep kernel) holds the stream while the host enqueues every
            # timed step, so that no event interval includes host launch latency
            torch.cuda._sleep(int(2e6 + 4e5 * args.steps))
            if use_flush:
                for k in range(args.steps):
                    flush.zero_()                  # evict the state from L2 (outside the events)
                    starts[k].record(stream)
                    run.enqueue(1)
                    ends[k].record(stream)
            else:
                # state larger than L2: the K steps run back to back between one pair of events,
                # enqueued by one call of the stepping entry point (its captured 16-step graphs)
                starts[0].record(stream)
                run.enqueue(args.steps)
                ends[0].record(stream)
        torch.cuda.synchronize()
        t_wall = time.perf_counter() - t_wall
    run.step(0)                                    # reads the device error flag
    if dist is not None:
        dist.barrier()
    if use_flush:
        total_ms = sum(s_.elapsed_time(e_) for s_, e_ in zip(starts, ends))
    else:
        total_ms = starts[0].elapsed_time(ends[0])
    launches = run.launches() - launches0
    total_ms = slowest_rank_ms(total_ms, dist, torch, "cuda")
    value = job_rate(world, nodes, args.steps, total_ms)
    ms_per_step = total_ms / args.steps

    # roofline of the step kernel: algorithmic bytes (read + write of every distribution once)
    bpl = bytes_per_lu(lattice, precision)
    alg_bytes = bpl * nodes
    achieved = alg_bytes / (ms_per_step * 1e-3) / 1e9
    peaks = {}
    pk_path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pk_path):
        with open(pk_path) as fh:
            peaks = json.load(fh)
    peak = peaks.get("hbm_gbs", 6800.0)
    khash = kernel_hash()
    traffic = NCU_TRAFFIC.get((args.workload, precision, khash))
    roofline = {"bound": "hbm", "achieved": round(achieved, 1), "peak": peak, "unit": "GB/s",
                "frac": round(achieved / peak, 4), "traffic": traffic,
                "peak_source": "measured (MEASURED_PEAKS.json hbm_gbs)" if "hbm_gbs" in peaks else "fallback",
                "algorithmic_bytes_per_launch": alg_bytes, "kernel": run.kernel_name(),
                "frac_fluid_only": round(achieved * fluid / nodes / peak, 4),
                "frac_of_nominal": round(achieved / NOMINAL_HBM_GBS, 4), "nominal_peak": NOMINAL_HBM_GBS,
                "bytes_per_lu": {"minimum": bytes_per_lu(lattice, precision),
                                 "measured_ncu": None if traffic is None else round(traffic / nodes, 2)}}

    # a sustained run of about one second (more clock samples than the K timed steps give)
    sustained = None
    if not args.no_extras:
        n_sus = max(args.steps, min(5000, int(1000.0 / max(ms_per_step, 1e-3))))
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with ClockSampler(local) as clk2:
            with torch.cuda.stream(stream):
                torch.cuda._sleep(int(2e6))
                e0.record(stream)
                run.enqueue(n_sus)
                e1.record(stream)
            torch.cuda.synchronize()
        run.step(0)
        ms_sus = e0.elapsed_time(e1) / n_sus
        cs = clk2.summary()
        sustained = {"steps": n_sus, "ms_per_step": round(ms_sus, 6), "value": round(nodes / (ms_sus * 1e-3) / 1e6, 1),
                     "unit": UNIT, "frac_of_measured_hbm": round(bpl * nodes / (ms_sus * 1e-3) / 1e9 / peak, 4),
                     "clocks": cs,
                     "ms_x_median_sm_ghz": None if not cs["sm_mhz"] else round(ms_sus * cs["sm_mhz"] / 1e3, 6),
                     "note": "the same step back to back for about one second (at most 5000 steps); time x "
                             "median SM clock is comparable across runs at different clocks"}

    # error against the FP64 oracle: one step from the GPU state of the first instance
    err = err_one_step(L, run.handles[0], wls[0], lambda: run.step(1))
    if args.workload == "c2" and precision == "fp32" and not args.no_extras:
        err = {"one_step": err, "after_20000_steps": err_c2_golden(L, stream)}

    observables = observables_rate(L, torch, run, wls, precision, stream)

    # batched launch vs one launch per instance (no L2 flush: back-to-back steps)
    bvs = None
    if run.batch and not args.no_extras:
        bvs = batched_vs_separate(L, torch, stream, run, cfgs, masks, rho0s, max(16, args.steps // 2))
    run.close()

    adjoint = None
    if not args.no_extras and args.workload in ("c2", "c5"):
        adjoint = adjoint_c5(L, torch, stream, steps=args.adjoint_steps)
    others = None
    if not args.no_extras and args.workload == "c2":
        def c3_extras(r, w, c, m, r0):
            tr = NCU_TRAFFIC.get(("c3", "fp32", ztma_kernel_hash()))
            out = {"traffic": tr,
                   "bytes_per_lu": {"minimum": bytes_per_lu("D3Q19", "fp32"),
                                    "measured_ncu": None if tr is None else round(tr / sum(x.nodes for x in w), 2)},
                   "e2e": e2e_rate(L, c, m, r0, w, args.steps, stream),
                   "observables": observables_rate(L, torch, r, w, "fp32", stream)}
            if rank == 0 and not args.no_cpu_baseline:
                try:
                    out["cpu_baseline"] = cpu_baseline("c3", target_s=10.0, all_cores=False)
                except Exception as exc:   # a reported baseline only
                    out["cpu_baseline"] = {"error": str(exc)[:200]}
            return out

        def c4_extras(r, w, c, m, r0):
            out = {"batched_vs_separate": batched_vs_separate(L, torch, stream, r, c, m, r0, max(16, args.steps // 2)),
                   "e2e": e2e_rate(L, c, m, r0, w, args.steps, stream)}
            if rank == 0 and not args.no_cpu_baseline:
                try:
                    out["cpu_baseline"] = cpu_baseline("c4", target_s=10.0, all_cores=False)
                except Exception as exc:   # a reported baseline only
                    out["cpu_baseline"] = {"error": str(exc)[:200]}
            return out

        others = {"c3": device_rate(L, torch, stream, "c3", max(100, args.steps), flush, extras=c3_extras),
                  "c4": device_rate(L, torch, stream, "c4", max(50, args.steps), flush, extras=c4_extras),
                  "c4_autotuned": device_rate(L, torch, stream, "c4", max(50, args.steps), flush, autotune=True),
                  "c2_fp64": device_rate(L, torch, stream, "c2", 10, flush, precision="fp64")}
        others["c3"]["err_vs_oracle"] = {"one_step": others["c3"]["err_vs_oracle"],
                                         "sphere_64cube_after_1000_steps": err_d3_golden(L, stream)}
        L.lbm_batch_autotune_forget()

    # end to end through the public API with host buffers
    torch.cuda.synchronize()
    e2e = e2e_rate(L, cfgs, masks, rho0s, wls, args.steps, stream, world)

    line = {"metric": METRIC, "value": round(value, 1), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(ms_per_step, 6), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32" if precision == "fp32" else "f64",
            "data": "synthetic (seeded drop-on-cylinder/sphere geometries shaped like the paper's Sec. IV)",
            "config": {"workload": label, "lattice": lattice, "instances": len(wls),
                       "grids": sorted(set(tuple(wl.shape[::-1]) for wl in wls))[:4], "nodes": nodes,
                       "precision": "fp32-deviation" if precision == "fp32" else "fp64",
                       "eos": f"C-S T={t_over_tc}Tc", "wall": "IVD", "kappas": [round(wl.kappa, 5) for wl in wls][:8],
                       "parallelism": f"replicas x{world}",
                       "l2": ("flushed before every timed step (2 x L2 buffer rewrite, outside the events)"
                              if use_flush else f"inputs larger than L2: {state_bytes / 1e6:.0f} MB of "
                              f"distributions vs {l2 / 1e6:.0f} MB of L2, no flush")},
            "fluid_only": {"value": round(value * fluid / nodes, 1), "unit": UNIT,
                           "note": "the same rate counting fluid nodes only (solid nodes are skipped)"},
            "roofline": roofline, "e2e": e2e, "gpu_launches": launches,
            "clocks": clk.summary(), "wall_s_timed_region": round(t_wall, 4),
            "kernel_hash": khash, "err_vs_oracle": err, "observables": observables}
    if sustained:
        line["sustained"] = sustained
    if bvs:
        line["batched_vs_separate"] = bvs
    if adjoint:
        line["adjoint_vs_forward"] = adjoint
    if others:
        line["other_workloads"] = others
    if not args.no_extras and args.workload == "c2":
        line["paper_context"] = paper_context(L, stream)
        line["paper_context_3d"] = paper_context_3d(L, stream)
    if rank == 0 and not args.no_cpu_baseline:
        try:
            line["cpu_baseline"] = cpu_baseline(args.workload)
        except Exception as exc:  # the oracle sample is a reported baseline only
            line["cpu_baseline"] = {"error": str(exc)[:200]}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()


def run_reference(args):
    world, rank, local = dist_setup()
    if rank != 0:
        return
    wls, precision, label = workload(args.workload)
    (times,), nodes = run_oracle(args.workload, args.steps, args.warmup)
    total = sum(times)
    value = nodes * args.steps / total / 1e6
    line = {"metric": METRIC, "value": round(value, 4), "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": round(1e3 * total / args.steps, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "impl": "reference",
            "config": {"workload": label, "per_step_sample": f"one {nodes}-node grid of the workload"},
            "cpu_baseline": {"value": round(value, 4), "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": f"{args.steps} FP64 oracle steps of one {nodes}-node grid of {label} "
                                       f"after {args.warmup} warm-up"},
            "e2e": {"value": round(value, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    global STEP_KERNEL
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c2", choices=list(WORKLOADS))
    ap.add_argument("--precision", default=None, choices=[None, "fp32", "fp64"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extras", action="store_true", help="skip the batched and adjoint side measurements")
    ap.add_argument("--adjoint-steps", type=int, default=2000)
    ap.add_argument("--step-kernel", default="auto", choices=["auto", "tile", "ymarch", "pair", "ztma"],
                    help="step kernel (auto: pair in D2Q9 FP32, ztma in D3Q19 FP32, tile in FP64)")
    args = ap.parse_args()
    STEP_KERNEL = args.step_kernel
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
