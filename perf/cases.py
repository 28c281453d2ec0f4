"""What is timed: the calls that users of the library make, over their range of sizes.

A case is one of
  run     one system: state in (device arrays), `steps` velocity-Verlet steps, state out
  batch   the same for many systems of uneven size stepped together
  sample  steps in blocks of ten with the observables read after each block
  nvt     Nose-Hoover steps (equilibration)
  forces  one force evaluation at new positions (a caller with its own integrator)
  noalloc the same through the allocation-free call

Positions are face-centred-cubic sites (the first n of the smallest lattice that holds
them) displaced uniformly by up to 0.1 per axis, velocities are Maxwell-Boltzmann with
zero net momentum: the state points, cutoffs, skin and time step are those of the
repository's own workloads (lj_inputs.py). Every pass sets its state first, so a pass
holds the binning and list build that new positions need.
"""
import math

import torch

from paper_1210_3450_gb300 import MD_FP32_FORCE, MD_FP64, LJBatch, LJSystem
from paper_1210_3450_gb300.ljmd import forces_noalloc

SKIN = 0.3
DT = 0.005
DEV = "cuda"


def listed():
    return [
        # the smallest served request: latency of a step counts
        dict(name="run_1000_fp32", kind="run", n=1000, rho=0.8442, temperature=0.722, rc=2.5, precision="fp32", steps=100),
        # the plain FP64 fluid of 4000 particles over its 200 steps
        dict(name="run_4000_fp64", kind="run", n=4000, rho=0.8442, temperature=0.722, rc=2.5, precision="fp64", steps=200),
        # the largest replica, one particle short of its lattice (ragged last tile)
        dict(name="run_31999_fp32", kind="run", n=31999, rho=0.75, temperature=1.0, rc=2.5, precision="fp32", steps=50),
        # the benchmark's fluid in both force forms
        dict(name="run_2048000_fp32", kind="run", n=2048000, rho=0.8442, temperature=0.722, rc=2.5, precision="fp32", steps=20),
        dict(name="run_2048000_fp64", kind="run", n=2048000, rho=0.8442, temperature=0.722, rc=2.5, precision="fp64", steps=10),
        # the cavitation liquid after its expansion, the longer cutoff
        dict(name="run_16384000_fp32", kind="run", n=16384000, rho=0.6047, temperature=0.9, rc=3.0, precision="fp32", steps=8),
        # replicas of uneven size stepped together
        dict(name="batch_256_fp32", kind="batch", sizes=1004, count=256, n_min=500, n_max=32000, precision="fp32", steps=20),
        # what a server holds at one time: few systems, sizes over three decades
        dict(name="batch_12_served", kind="batch", sizes=1005, count=12, n_min=1000, n_max=1000000, precision="fp32", steps=20),
        # production run with observables every ten steps
        dict(name="sample_864000_fp32", kind="sample", n=864000, rho=0.8442, temperature=0.722, rc=2.5, precision="fp32", blocks=2),
        # equilibration at constant temperature
        dict(name="nvt_16000_fp64", kind="nvt", n=16000, rho=0.70, temperature=0.90, rc=3.0, precision="fp64", steps=40),
        # forces of new positions, an odd size
        dict(name="forces_262143_fp64", kind="forces", n=262143, rho=0.8442, temperature=0.722, rc=2.5, precision="fp64"),
        # the allocation-free call at its largest size
        dict(name="noalloc_65536", kind="noalloc", n=65536, rho=0.8442, rc=2.5),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "sample", "nvt", "forces", "noalloc"])
    rho = round(rng.uniform(0.60, 0.85), 4)
    t = round(rng.uniform(0.7, 1.2), 3)
    rc = rng.choice([2.5, 2.5, 3.0])
    if kind == "noalloc":
        return dict(kind=kind, n=_log_uniform(rng, 500, 65536), rho=rho, rc=rc)
    if kind == "forces":
        return dict(kind=kind, n=_log_uniform(rng, 1000, 2000000), rho=rho, temperature=t, rc=rc,
                    precision=rng.choice(["fp64", "fp32"]))
    if kind == "batch":
        hi = rng.choice([4000, 32000, 200000])
        count = rng.randint(4, max(6, min(300, int(2.4e6 / hi))))
        return dict(kind=kind, sizes=rng.randrange(1 << 30), count=count, n_min=500, n_max=hi, precision=rng.choice(["fp32", "fp32", "fp64"]),
                    steps=rng.randint(10, 30))
    if kind == "sample":
        return dict(kind=kind, n=_log_uniform(rng, 4000, 1000000), rho=rho, temperature=t, rc=rc,
                    precision=rng.choice(["fp64", "fp32"]), blocks=rng.randint(1, 3))
    if kind == "nvt":
        return dict(kind=kind, n=_log_uniform(rng, 1000, 300000), rho=rho, temperature=t, rc=rc, precision="fp64",
                    steps=rng.randint(10, 40))
    precision = rng.choice(["fp64", "fp32", "fp32"])
    n = _log_uniform(rng, 500, 1500000 if precision == "fp64" else 4000000)
    steps = max(8, min(100, int(1.2e7 / n)))
    return dict(kind=kind, n=n, rho=rho, temperature=t, rc=rc, precision=precision, steps=steps)


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return g


def _positions(g, n, rho):
    box = (n / rho) ** (1.0 / 3.0)
    m = 1
    while 4 * m ** 3 < n:
        m += 1
    k = torch.arange(n, device=DEV)
    cell, b = k // 4, k % 4
    basis = torch.tensor([[0.0, 0.0, 0.0], [0.5, 0.5, 0.0], [0.5, 0.0, 0.5], [0.0, 0.5, 0.5]], dtype=torch.float64, device=DEV)
    x = torch.stack([cell // (m * m), cell // m % m, cell % m], 1).to(torch.float64)
    x = (x + basis[b]) * (box / m)
    x = x + (torch.rand(n, 3, dtype=torch.float64, device=DEV, generator=g) * 0.2 - 0.1)
    x = torch.remainder(x, box)
    x[x >= box] = 0.0
    return x.contiguous(), box


def _velocities(g, n, temperature):
    v = torch.randn(n, 3, dtype=torch.float64, device=DEV, generator=g)
    v = v - v.mean(0)
    return (v * torch.sqrt(temperature * 3.0 * (n - 1) / (v * v).sum())).contiguous()


def _inputs(case, seed):
    """The systems of a case: dicts of n, box, rc, x, v."""
    g = _generator(seed)
    if case["kind"] == "batch":
        # sizes and state points belong to the case, positions and velocities to the seed
        u = torch.rand(3, case["count"], dtype=torch.float64, device=DEV, generator=_generator(case["sizes"])).tolist()
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        specs = [(int(math.exp(lo + (hi - lo) * a)), 0.60 + 0.25 * b, 0.7 + 0.5 * c, 2.5) for a, b, c in zip(*u)]
    else:
        specs = [(case["n"], case["rho"], case.get("temperature", 1.0), case["rc"])]
    out = []
    for n, rho, t, rc in specs:
        x, box = _positions(g, n, rho)
        out.append(dict(n=n, box=box, rc=rc, x=x, v=_velocities(g, n, t)))
    return out


def _thermostat_mass(case):
    # thermostat period 0.5: Q = g T tau^2 / (4 pi^2)
    return 3.0 * (case["n"] - 1) * case["temperature"] * 0.25 / (4.0 * math.pi ** 2)


def _mode(case):
    return MD_FP32_FORCE if case["precision"] == "fp32" else MD_FP64


def prepare(case, seed):
    syss = _inputs(case, seed)
    st = dict(case=case, systems=syss)
    if case["kind"] == "batch":
        total = sum(s["n"] for s in syss)
        st["handle"] = LJBatch(systems=[(s["n"], s["box"], s["rc"], SKIN) for s in syss], precision=_mode(case))
        st["x"] = torch.empty(total, 3, dtype=torch.float64, device=DEV)
        st["v"] = torch.empty(total, 3, dtype=torch.float64, device=DEV)
        return st
    s = syss[0]
    if case["kind"] != "noalloc":
        st["handle"] = LJSystem(s["box"], s["n"], s["rc"], SKIN, _mode(case))
    if case["kind"] in ("forces", "noalloc"):
        st["f"] = torch.empty(s["n"], 3, dtype=torch.float64, device=DEV)
    else:
        st["x"] = torch.empty(s["n"], 3, dtype=torch.float64, device=DEV)
        st["v"] = torch.empty(s["n"], 3, dtype=torch.float64, device=DEV)
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "noalloc":
        s = st["systems"][0]
        forces_noalloc(s["x"], s["box"], s["rc"], st["f"])
        return {"f": st["f"]}
    h = st["handle"]
    if kind == "batch":
        for k, s in enumerate(st["systems"]):
            h.set_state_dev(k, s["x"], s["v"])
        h.step_async(case["steps"], DT)
        at = 0
        for k, s in enumerate(st["systems"]):
            h.get_state_dev(k, st["x"][at:at + s["n"]], st["v"][at:at + s["n"]])
            at += s["n"]
        return {"x": st["x"], "v": st["v"]}
    s = st["systems"][0]
    h.set_state_dev(s["x"], s["v"])
    if kind == "forces":
        h.forces_dev(st["f"])
        return {"f": st["f"]}
    out = {}
    if kind == "run":
        h.step_async(case["steps"], DT)
    elif kind == "nvt":
        out["zeta"], out["eta"] = h.step_nvt(case["steps"], DT, case["temperature"], _thermostat_mass(case))
    else:
        out["observables"] = []
        for _ in range(case["blocks"]):
            h.step_async(10, DT)
            out["observables"].append(h.observables())
    h.get_state_dev(st["x"], st["v"])
    return {"x": st["x"], "v": st["v"], **out}


# -------------------------------------------------------------------- work

def work(case):
    """Each pair inside the cutoff once per force evaluation (8 for the separation and the
    squared distance, 9 for the force factor, 12 to add it to both particles) and 18 per
    particle for the update; positions and velocities read and written once per step."""
    kind = case["kind"]
    rho, rc = case.get("rho", 0.725), case.get("rc", 2.5)
    if kind == "batch":
        lo, hi = case["n_min"], case["n_max"]
        n = case["count"] * (hi - lo) / math.log(hi / lo)  # mean of the log-uniform sizes
    else:
        n = case["n"]
    pairs = 0.5 * n * rho * 4.0 / 3.0 * math.pi * rc ** 3
    if kind in ("forces", "noalloc"):
        return {"bytes": 48.0 * n, "flops": 29.0 * pairs}
    steps = 10 * case["blocks"] if kind == "sample" else case["steps"]
    flops = steps * (29.0 * pairs + 18.0 * n)
    if kind == "sample":
        flops += case["blocks"] * 20.0 * pairs
    return {"bytes": 96.0 * n * steps, "flops": flops}


# --------------------------------------------- the same in plain 64-bit torch

class _Exact:
    """Forces of several periodic systems from a padded table of cells of side >= rc."""

    def __init__(self, syss):
        self.box = torch.cat([torch.full((s["n"],), s["box"], dtype=torch.float64, device=DEV) for s in syss])
        self.rc = syss[0]["rc"]
        nc = [max(1, int(s["box"] / self.rc)) for s in syss]
        if min(nc) < 3:
            raise ValueError("a box of fewer than three cells per axis")
        first = [0]
        for k in nc:
            first.append(first[-1] + k ** 3)
        self.ncell = first[-1]
        self.nc = torch.cat([torch.full((s["n"],), k, dtype=torch.int64, device=DEV) for s, k in zip(syss, nc)])
        self.first = torch.cat([torch.full((s["n"],), f, dtype=torch.int64, device=DEV) for s, f in zip(syss, first)])
        # neighbour cells and the shift of their particles, for each of the 27 directions
        self.near, self.shift = [], []
        axes = []
        for s, k, f in zip(syss, nc, first):
            c = torch.arange(k ** 3, device=DEV)
            axes.append((torch.stack([c % k, c // k % k, c // (k * k)], 1), k, f, s["box"]))
        for o in range(27):
            d = torch.tensor([o % 3 - 1, o // 3 % 3 - 1, o // 9 - 1], device=DEV)
            idx, sh = [], []
            for a, k, f, box in axes:
                q = a + d
                w = torch.div(q, k, rounding_mode="floor")
                q = q - w * k
                idx.append(f + q[:, 0] + k * (q[:, 1] + k * q[:, 2]))
                sh.append(w.to(torch.float64) * box)
            self.near.append(torch.cat(idx))
            self.shift.append(torch.cat(sh))
        r6 = self.rc ** -6
        self.c2 = 6.0 * r6 * r6 / self.rc ** 2 - 3.0 * r6 / self.rc ** 2
        self.c0 = 4.0 * r6 - 7.0 * r6 * r6

    def forces(self, x, energies=False):
        box = self.box[:, None]
        x = x - box * torch.floor(x / box)
        c = torch.clamp((x * (self.nc[:, None].to(torch.float64) / box)).to(torch.int64), min=0)
        c = torch.minimum(c, self.nc[:, None] - 1)
        cell = self.first + c[:, 0] + self.nc * (c[:, 1] + self.nc * c[:, 2])
        order = torch.argsort(cell)
        count = torch.bincount(cell, minlength=self.ncell)
        start = torch.cumsum(count, 0) - count
        m = int(count.max())
        slot = torch.arange(len(cell), device=DEV) - start[cell[order]]
        table = torch.full((self.ncell, m), -1, dtype=torch.int64, device=DEV)
        table[cell[order], slot] = order
        pos = x[table.clamp(min=0)].permute(2, 0, 1).contiguous()  # axis, cell, place
        pos = torch.where(table[None] < 0, torch.full_like(pos, 1e6), pos)
        f = torch.zeros(len(x), 3, dtype=torch.float64, device=DEV)
        pe = torch.zeros((), dtype=torch.float64, device=DEV)
        w = torch.zeros((), dtype=torch.float64, device=DEV)
        step = max(1, int(3e7) // (m * m))
        for a in range(0, self.ncell, step):
            here = pos[:, a:a + step]
            there = table[a:a + step]
            acc = torch.zeros_like(here)
            for near, shift in zip(self.near, self.shift):
                j = near[a:a + step]
                q, sh = pos[:, j], shift[a:a + step]
                d = [(q[k][:, None, :] - here[k][:, :, None]) + sh[:, k, None, None] for k in range(3)]
                r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
                inside = (r2 < self.rc * self.rc) & (table[j][:, None, :] != there[:, :, None]) & (there >= 0)[:, :, None]
                i2 = torch.where(inside, 1.0 / r2, torch.zeros_like(r2))
                i6 = i2 * i2 * i2
                g = i2 * i6 * (24.0 - 48.0 * i6) + (8.0 * self.c2) * inside.to(torch.float64)
                for k in range(3):
                    acc[k] += (g * d[k]).sum(2)
                if energies:
                    sr, nin = torch.where(inside, r2, 0.0).sum(), inside.sum()
                    pe += 0.5 * 4.0 * ((i6 * i6 - i6).sum() + self.c2 * sr + self.c0 * nin)
                    w += 0.5 * ((48.0 * i6 * i6 - 24.0 * i6).sum() - 8.0 * self.c2 * sr)
            real = there >= 0
            f[there[real]] = acc[:, real].T
        return (f, pe, w) if energies else f


def exact(case, seed):
    if case["kind"] == "batch":
        size = 20.0 * case["count"] * (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        size *= case["steps"] / 20.0
    else:
        size = case["n"] * float(case.get("steps", 10 * case.get("blocks", 0)) + 1) * (case["rc"] / 2.5) ** 3
    if size > 6e7:
        return None
    syss = _inputs(case, seed)
    try:
        e = _Exact(syss)
    except ValueError:
        return None
    x = torch.cat([s["x"] for s in syss])
    v = torch.cat([s["v"] for s in syss])
    if case["kind"] in ("forces", "noalloc"):
        f = e.forces(x)
        return {"f": f}
    out = {}
    f = e.forces(x)

    def verlet(x, v, f):
        v = v + 0.5 * DT * f
        x = x + DT * v
        f = e.forces(x)
        return x, v + 0.5 * DT * f, f

    if case["kind"] == "nvt":
        q, t, g = _thermostat_mass(case), case["temperature"], 3.0 * (case["n"] - 1)
        zeta = eta = 0.0

        def half(v, zeta, eta):
            k2 = float((v * v).sum())
            zeta += 0.25 * DT * (k2 - g * t) / q
            eta += 0.5 * DT * zeta
            s = math.exp(-0.5 * DT * zeta)
            zeta += 0.25 * DT * (k2 * s * s - g * t) / q
            return v * s, zeta, eta

        for _ in range(case["steps"]):
            v, zeta, eta = half(v, zeta, eta)
            x, v, f = verlet(x, v, f)
            v, zeta, eta = half(v, zeta, eta)
        out["zeta"], out["eta"] = zeta, eta
    elif case["kind"] == "sample":
        out["observables"] = []
        n, box = case["n"], syss[0]["box"]
        for _ in range(case["blocks"]):
            for _ in range(10):
                x, v, f = verlet(x, v, f)
            _, pe, w = e.forces(x, energies=True)
            ke = 0.5 * float((v * v).sum())
            out["observables"].append(dict(pe=float(pe), virial=float(w), ke=ke, temperature=2.0 * ke / (3.0 * (n - 1)),
                                           pressure=(2.0 * ke + float(w)) / (3.0 * box ** 3)))
    else:
        for _ in range(case["steps"]):
            x, v, f = verlet(x, v, f)
    box = e.box[:, None]
    x = x - box * torch.floor(x / box)
    return {"x": x, "v": v, **out}
