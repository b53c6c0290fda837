"""The calls that a user of this library makes, as cases that can be timed and compared.

listed() gives the fixed cases, draw() more of the same ranges; prepare() makes what a program has in hand before
the call (a context, its workspace and the particles on the GPU), run() makes the call once, work() says what the
call cannot do without, and exact() gives the outputs in 64 bits where plain numpy can form them.

Kinds of case:

* "steps": restart from a checkpoint's particles and clock, take `steps` time steps (regrid, collide, transport), and
  read the particles back on the device.  One disk, or several batched in one context; mixed or FP64; with or without
  the tracer, a fragmentation ramp, a tabulated gas and the adaptive step.  The mixed path's swarms per thread are
  pinned, as a resumed run has to do.
* "cell": the 0D constant-kernel cell, collided to t_end from its monomers.
* "transport": one transport step of a disk's particles, read back on the device.
* "regrid": the context-free regrid of one disk on the caller's arrays.
* "snapshot": the diagnostics of one output time (moments per radial bin and the sigma_d(m, r) map).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_21239_gb300 import mcd, workloads as W

AU, YR = W.AU, W.YR
CUDA = torch.device("cuda")


# ---- the cases -------------------------------------------------------------------------------------------------
def steps_case(name=None, *, n_r, n_z, per_cell, prec="mixed", disks=1, steps=1, dt_yr=1.0, alpha=1e-3, v_frag=1000.0,
               batch=False, features=False):
    c = dict(kind="steps", n_r=n_r, n_z=n_z, per_cell=per_cell, prec=prec, disks=disks, steps=steps, dt_yr=dt_yr,
             alpha=alpha, v_frag=v_frag, batch=batch, features=features)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one cell of the constant-kernel test problem (the method's analytic check), 1,500 events
        dict(name="cell_0d_200_fp64", kind="cell", n=200, prec="fp64", t_end=100.0),
        # a small disk stepped many times (seeds of a parameter study): launches and short chains
        steps_case("disk_16x4x100_mixed", n_r=16, n_z=4, per_cell=100, steps=8),
        # the same in the plain FP64 path (the reference precision)
        steps_case("disk_16x4x100_fp64", n_r=16, n_z=4, per_cell=100, steps=4, prec="fp64"),
        # the benchmark disk, the library's ordinary workload: 819,200 particles in 4,096 cells
        steps_case("disk_256x16x200_mixed", n_r=256, n_z=16, per_cell=200, steps=4),
        steps_case("disk_256x16x200_fp64", n_r=256, n_z=16, per_cell=200, prec="fp64"),
        # many disks of different size and physics in one context (a parameter grid), every cell class at once
        steps_case("batch_16_disks_mixed", n_r=0, n_z=8, per_cell=0, disks=16, batch=True),
        # the largest disk: 13.1 M particles, 400 per cell, fragmentation-dominated
        steps_case("stress_1024x32x400_mixed", n_r=1024, n_z=32, per_cell=400, alpha=1e-2, v_frag=100.0),
        # every option in one run on an odd-sized disk: ramp, tracer, gas table, adaptive step
        steps_case("features_61x7x157_mixed", n_r=61, n_z=7, per_cell=157, steps=2, features=True),
        # transport alone (a drift/diffusion run without collisions), both precisions
        dict(name="transport_819200_mixed", kind="transport", n_r=256, n_z=16, per_cell=200, prec="mixed", dt_yr=1.0),
        dict(name="transport_819200_fp64", kind="transport", n_r=256, n_z=16, per_cell=200, prec="fp64", dt_yr=1.0),
        # the regrid as a service on a caller's arrays, at its largest size
        dict(name="regrid_65536", kind="regrid", n_r=64, n_z=8, per_cell=128, dead=0.02),
        # an output time of the benchmark disk: radial moments and the sigma_d(m, r) map
        dict(name="snapshot_819200", kind="snapshot", n_r=256, n_z=16, per_cell=200, bins=32, map_r=64, map_m=96),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _disk(rng, n_hi, per_hi):
    """Odd and even sizes: zones over their logarithm, at most n_hi particles."""
    while True:
        n_r, n_z, per = _log(rng, 8, 1024), _log(rng, 1, 32), rng.randint(25, per_hi)
        if 2000 <= n_r * n_z * per <= n_hi and n_z * per <= 14336:  # (the largest zone the regrid takes)
            return n_r, n_z, per


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "fp64", "cell", "transport", "regrid", "snapshot"])
    if kind == "steps":
        n_r, n_z, per = _disk(rng, 3_000_000, 400)
        return steps_case(n_r=n_r, n_z=n_z, per_cell=per, steps=rng.randint(1, 2), dt_yr=round(rng.uniform(0.1, 0.75), 3),
                          alpha=rng.choice([1e-4, 1e-3, 1e-2]), v_frag=rng.choice([300.0, 1000.0, 3000.0]),
                          features=rng.random() < 0.25)
    if kind == "fp64":
        n_r, n_z, per = _disk(rng, 400_000, 250)
        return steps_case(n_r=n_r, n_z=n_z, per_cell=per, prec="fp64", dt_yr=round(rng.uniform(0.25, 1.0), 3))
    if kind == "cell":
        return dict(kind="cell", n=rng.randint(40, 400), prec=rng.choice(["mixed", "fp64"]),
                    t_end=round(rng.uniform(5.0, 100.0), 2))
    if kind == "transport":
        n_r, n_z, per = _disk(rng, 5_000_000, 450)
        return dict(kind="transport", n_r=n_r, n_z=n_z, per_cell=per, prec=rng.choice(["mixed", "mixed", "fp64"]),
                    dt_yr=round(rng.uniform(0.1, 3.0), 3))
    if kind == "regrid":
        while True:
            n_r, n_z, per = _log(rng, 4, 512), _log(rng, 1, 32), rng.randint(8, 400)
            if 1000 <= n_r * n_z * per <= 65536 and n_z * per <= 14336:
                return dict(kind="regrid", n_r=n_r, n_z=n_z, per_cell=per, dead=round(rng.uniform(0.0, 0.2), 3))
    n_r, n_z, per = _disk(rng, 4_000_000, 450)
    return dict(kind="snapshot", n_r=n_r, n_z=n_z, per_cell=per, bins=_log(rng, 8, 256), map_r=_log(rng, 8, 128),
                map_m=_log(rng, 8, 256))


# ---- inputs ----------------------------------------------------------------------------------------------------
def _uniform(gen, n):
    return torch.rand(n, dtype=torch.float64, device=CUDA, generator=gen)


def _midrun(P, n, seed):
    """A disk in growth/fragmentation balance (the recipe of workloads.midrun_state, drawn on the GPU)."""
    gen = torch.Generator(device=CUDA)
    gen.manual_seed(seed)
    r = P["r_in"] + _uniform(gen, n) * (P["r_out"] - P["r_in"])
    a0 = P["a_mono"]
    amax = torch.clamp(10.0 * AU / r, min=a0)
    a = (math.sqrt(a0) + _uniform(gen, n) * (torch.sqrt(amax) - math.sqrt(a0))) ** 2
    m = 4.0 / 3.0 * math.pi * P["rho_s"] * a**3
    h = 0.0334 * AU * (r / AU) ** 1.25 / torch.sqrt(1.0 + a / 1e-2)
    z = torch.randn(n, dtype=torch.float64, device=CUDA, generator=gen) * h
    return m, r, z


def _layout(case):
    """(parameters, grids) of the context's disks."""
    if case.get("batch"):
        disks = W.batched_disks()[:case["disks"]]
        return [d["params"] for d in disks], [(d["n_r"], d["n_z"], d["per_cell"]) for d in disks]
    over = dict(alpha=case.get("alpha", 1e-3), v_frag=case.get("v_frag", 1000.0))
    if case.get("features"):
        over["frag_ramp"] = 0.3
    P = W.benchmark_disk(**over)
    if case.get("features"):
        P["gas_table"] = W.gap_bump_gas_table(P)
    return [P], [(case["n_r"], case["n_z"], case["per_cell"])]


class Run:
    """A context, the particles it starts from and the columns its results are read into."""

    def __init__(self, case, seed):
        self.case = case
        params, grids = _layout(case)
        self.disk = mcd.Disk(params, grids, seed=seed, prec=case["prec"])
        if self.disk.prec == mcd.MCD_MIXED:
            mcd.mcd_set_option(self.disk.ctx, mcd.MCD_OPT_SWARMS_PER_THREAD, 1)
        self.start = []  # per disk: m, M, r, z, id
        self.sizes = [a * b * c for a, b, c in grids]
        for k, n in enumerate(self.sizes):
            p = self.disk.particles_device(k)
            m, r, z = _midrun(params[k], n, seed * 64 + k)
            ids = torch.arange(n, dtype=torch.int32, device=CUDA)
            self.start.append((m, p["M"], r, z, ids))
        n = sum(self.sizes)
        self.tracer = None
        if case.get("features"):
            gen = torch.Generator(device=CUDA)
            gen.manual_seed(seed + 1)
            self.tracer = _uniform(gen, n)
        self.out = {k: torch.empty(n, dtype=torch.float64, device=CUDA) for k in ("m", "M", "r", "z")}
        self.out["id"] = torch.empty(n, dtype=torch.int32, device=CUDA)
        if self.tracer is not None:
            self.out["q"] = torch.empty(n, dtype=torch.float64, device=CUDA)

    def restart(self):
        mcd.mcd_set_clock(self.disk.ctx, 0.0, 0)
        for k, cols in enumerate(self.start):
            mcd.mcd_set_particles(self.disk.ctx, k, *cols, where=mcd.MCD_DEVICE)
        if self.tracer is not None:
            mcd.mcd_set_tracer(self.disk.ctx, 0, self.tracer, mcd.MCD_DEVICE)

    def read(self):
        at = 0
        for k, n in enumerate(self.sizes):
            col = {key: v[at:at + n] for key, v in self.out.items()}
            mcd.mcd_get_particles(self.disk.ctx, k, col["m"], col["M"], col["r"], col["z"], col["id"], mcd.MCD_DEVICE)
            if self.tracer is not None:
                mcd.mcd_get_tracer(self.disk.ctx, k, col["q"], mcd.MCD_DEVICE)
            at += n
        return dict(self.out)


def _cell_positions(n, seed):
    P = W.constant_kernel_cell()
    gen = torch.Generator(device=CUDA)
    gen.manual_seed(seed)
    r = P["r_in"] + _uniform(gen, n) * (P["r_out"] - P["r_in"])
    return P, r, _uniform(gen, n) * AU


def _prepare_cell(case, seed):
    n = case["n"]
    P, r, z = _cell_positions(n, seed)
    d = mcd.Disk(P, (1, 1, n), seed=seed, prec=case["prec"])
    if d.prec == mcd.MCD_MIXED:
        mcd.mcd_set_option(d.ctx, mcd.MCD_OPT_SWARMS_PER_THREAD, 1)
    ids = torch.arange(n, dtype=torch.int32, device=CUDA)
    one = torch.ones(n, dtype=torch.float64, device=CUDA)
    return {"case": case, "disk": d, "start": (one, one / n, r, z, ids), "m": torch.empty_like(one),
            "id": torch.empty_like(ids)}


def _regrid_inputs(case, seed):
    """A disk's arrays as a transport step leaves them: cell order lost, some particles removed."""
    P = W.benchmark_disk()
    n = case["n_r"] * case["n_z"] * case["per_cell"]
    m, r, z = _midrun(P, n, seed)
    gen = torch.Generator(device=CUDA)
    gen.manual_seed(seed + 1)
    r = torch.where(_uniform(gen, n) < case["dead"], torch.full_like(r, math.inf), r)
    ids = torch.randperm(n, device=CUDA, generator=gen).to(torch.int32)
    M = torch.full_like(m, 1e24)
    return P, (m, M, r, z, ids)


def _prepare_regrid(case, seed):
    P, cols = _regrid_inputs(case, seed)
    n, C = cols[0].numel(), case["n_r"] * case["n_z"]
    new = lambda k, t: torch.empty(k, dtype=t, device=CUDA)  # noqa: E731
    f, i, l = torch.float64, torch.int32, torch.int64
    out = [new(n, f), new(n, f), new(n, f), new(n, f), new(n, i), new(C, l), new(C, i), new(6 * C, f), new(C, f),
           new(1, l), new(1, i)]
    return {"case": case, "P": P, "cols": cols, "out": out}


def _snapshot_edges(case):
    return (np.geomspace(1.0, 100.0, case["bins"] + 1) * AU, np.geomspace(1.0, 100.0, case["map_r"] + 1) * AU,
            np.geomspace(1e-12, 1e4, case["map_m"] + 1))


def _prepare_snapshot(case, seed):
    R = Run(dict(case, prec="mixed"), seed)
    R.restart()
    mcd.mcd_regrid(R.disk.ctx)
    return {"case": case, "run": R, "edges": _snapshot_edges(case)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "steps":
        return {"case": case, "run": Run(case, seed)}
    if kind == "cell":
        return _prepare_cell(case, seed)
    if kind == "transport":
        R = Run(case, seed)
        R.restart()
        return {"case": case, "run": R}
    if kind == "regrid":
        return _prepare_regrid(case, seed)
    return _prepare_snapshot(case, seed)


# ---- the calls -------------------------------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "steps":
        R = state["run"]
        R.restart()
        adaptive = case["features"]
        for _ in range(case["steps"]):
            R.disk.step(0.0 if adaptive else case["dt_yr"] * YR)
        out = R.read()
        if adaptive:
            out["t"] = R.disk.stats().t  # the clock that the chosen steps reached
        return out
    if kind == "cell":
        ctx = state["disk"].ctx
        mcd.mcd_set_clock(ctx, 0.0, 0)
        mcd.mcd_set_particles(ctx, 0, *state["start"], where=mcd.MCD_DEVICE)
        mcd.mcd_regrid(ctx)
        mcd.mcd_collide(ctx, case["t_end"])
        mcd.mcd_get_particles(ctx, 0, m=state["m"], id=state["id"], where=mcd.MCD_DEVICE)
        return {"m": state["m"], "id": state["id"]}
    if kind == "transport":
        R = state["run"]
        mcd.mcd_transport(R.disk.ctx, case["dt_yr"] * YR)
        return R.read()
    if kind == "regrid":
        mcd.mcd_regrid_noalloc(state["P"], (case["n_r"], case["n_z"], case["per_cell"]), state["cols"], state["out"])
        return list(state["out"])
    d, (edges, re, me) = state["run"].disk, state["edges"]
    return {"moments": d.moments(edges), "map": d.sigma_map(re, me)}


# ---- what a pass cannot do without -----------------------------------------------------------------------------
EVENTS = 0.13  # events per particle and year of the benchmark disk's mid-run state


def work(case):
    kind = case["kind"]
    if kind == "cell":
        n = case["n"]
        events = n * math.log(1.0 + case["t_end"]) * 1.6  # about 1,500 at n = 200, t = 100
        return {"bytes": 24.0 * n, "flops": 8.0 * n * (n + events)}
    if kind == "steps":
        _, grids = _layout(case)
        n = sum(a * b * c for a, b, c in grids)
        pairs = sum(a * b * c * (c + 1) / 2 for a, b, c in grids)
        events = sum(EVENTS * case["dt_yr"] * a * b * c * c for a, b, c in grids)
        # regrid reads three keys' columns and moves the record, the collide reads m, M and writes m, transport
        # reads r, z, m, id and writes r, z; 60 flops per kernel entry
        return {"bytes": case["steps"] * n * (92.0 + 24.0 + 44.0), "flops": case["steps"] * 60.0 * (pairs + events)}
    n = float(case["n_r"] * case["n_z"] * case["per_cell"])
    if kind == "transport":
        return {"bytes": 44.0 * n + 72.0 * n, "flops": 200.0 * n}  # the step, and the columns read back
    if kind == "regrid":
        return {"bytes": 72.0 * n, "flops": 0.0}
    return {"bytes": 24.0 * n + 40.0 * case["bins"] + 8.0 * case["map_r"] * case["map_m"], "flops": 10.0 * n}


# ---- the outputs in 64 bits ------------------------------------------------------------------------------------
def _mulhilo(a, b):
    """High and low words of the 64 x 64-bit product (numpy uint64 arrays)."""
    m32, s = np.uint64(0xFFFFFFFF), np.uint64(32)
    a0, a1, b0, b1 = a & m32, a >> s, b & m32, b >> s
    p00, p01, p10, p11 = a0 * b0, a0 * b1, a1 * b0, a1 * b1
    mid = (p00 >> s) + (p01 & m32) + (p10 & m32)
    return p11 + (p01 >> s) + (p10 >> s) + (mid >> s), a * b


def _philox(c, k):
    """Philox4x64-10 (Salmon et al. 2011): counters c (four uint64 arrays), key k (two ints)."""
    M0, M1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    W0, W1, mask = 0x9E3779B97F4A7C15, 0xBB67AE8584CAA73B, (1 << 64) - 1
    c = [np.asarray(x, np.uint64) for x in c]
    k0, k1 = k
    with np.errstate(over="ignore"):
        for _ in range(10):
            h0, l0 = _mulhilo(M0, c[0])
            h1, l1 = _mulhilo(M1, c[2])
            c = [h1 ^ c[1] ^ np.uint64(k0), l1, h0 ^ c[3] ^ np.uint64(k1), l0]
            k0, k1 = (k0 + W0) & mask, (k1 + W1) & mask
    return [((x >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0**-53 for x in c]


def _exact_cell(case, seed):
    """The event chain of the constant-kernel cell: every swarm's partner rate is sum_j M_j / m_j."""
    n, t_end = case["n"], case["t_end"]
    if case["prec"] != "fp64":  # FP32 choices may differ from the 64-bit ones now and then
        return None
    _, _, z = _cell_positions(n, seed)
    ids = np.argsort(z.cpu().numpy(), kind="stable").astype(np.int32)
    m, t, e = np.ones(n), 0.0, 0
    zero = np.zeros(4096, np.uint64)
    u = None
    while True:
        if e % 4096 == 0:
            at = np.arange(e, e + 4096, dtype=np.uint64)
            u = np.stack(_philox([at, zero, zero, zero + np.uint64(2)], (seed, 0)), 1)
        u0, u1, u2, _ = u[e % 4096]
        w = np.cumsum(1.0 / n / m)
        t -= math.log(u0) / (n * w[-1])
        if t >= t_end:
            return {"m": m, "id": ids}
        i = min(int(np.searchsorted(np.arange(1, n + 1) * w[-1], u1 * n * w[-1], side="right")), n - 1)
        j = min(int(np.searchsorted(w, u2 * w[-1], side="right")), n - 1)
        m[i] += m[j]
        e += 1


def _exact_transport(case, seed):
    """One drift/diffusion step of every particle in the power-law gas, vertically isothermal disk."""
    P = _layout(case)[0][0]
    n = case["n_r"] * case["n_z"] * case["per_cell"]
    m, r, z = (x.cpu().numpy() for x in _midrun(P, n, seed * 64))
    dt = case["dt_yr"] * YR
    zero = np.zeros(n, np.uint64)
    u = _philox([np.arange(n, dtype=np.uint64), zero, zero, zero + np.uint64(3)], (seed, 0))
    rad, ang = np.sqrt(-2.0 * np.log(u[0])), 2.0 * np.pi * u[1]
    kB, mp, GM = 1.380649e-16, 1.67262192e-24, 1.32712440018e26
    x = r / AU
    Sig, T = P["sigma0"] * x ** -P["p"], P["T0"] * x ** -P["q"]
    cs = np.sqrt(kB * T / (P["mu"] * mp))
    Om = np.sqrt(P["m_star"] * GM / r / r / r)
    H = cs / Om
    rho = Sig / (math.sqrt(2.0 * math.pi) * H) * np.exp(-0.5 * (z / H) ** 2)
    vth = math.sqrt(8.0 / math.pi) * cs
    lam = P["mu"] * mp / P["sigma_h2"] / rho
    nu = 0.5 * vth * lam
    eta = 0.5 * cs * cs / (Om * r) * (P["p"] + 0.5 * (3.0 + P["q"]))
    D = P["alpha"] * cs * H
    a = np.cbrt(3.0 * m / (4.0 * np.pi * P["rho_s"]))
    St = np.where(a < 2.25 * lam, P["rho_s"] * a / (rho * vth), 2.0 * P["rho_s"] * a * a / (9.0 * nu * rho)) * Om
    vr = -2.0 * eta * St / (1.0 + St * St)
    vD = D / r * (1.0 - P["p"] - 0.5 * P["q"] + (z / H) ** 2 * 0.5 * (3.0 - P["q"]))
    rn = r + (vr + vD) * dt + np.sqrt(2.0 * D * dt) * rad * np.cos(ang)
    k = Om * (St + P["alpha"])
    zn = z * np.exp(-k * dt) + np.sqrt(D * -np.expm1(-2.0 * k * dt) / k) * rad * np.sin(ang)
    rn = np.where(rn < P["r_in"], np.inf, np.where(rn > P["r_out"], 2.0 * P["r_out"] - rn, rn))
    return {"m": m, "M": None, "r": rn, "z": zn, "id": np.arange(n, dtype=np.int32)}


def _split(n, k):
    """Sizes of k consecutive parts of n, the first n mod k one larger, and their offsets."""
    size = np.full(k, n // k, np.int64)
    size[:n % k] += 1
    return size, np.concatenate([[0], np.cumsum(size)])


def _edges(x, at, size, k, K):
    """Part k's lower and upper edge: midpoints between parts, half a spacing beyond the ends."""
    lo = 0.5 * (x[at - 1] + x[at]) if k > 0 else x[at] - 0.5 * (x[1] - x[0])
    end = at + size
    hi = 0.5 * (x[end - 1] + x[end]) if k + 1 < K else x[-1] + 0.5 * (x[-1] - x[-2])
    return lo, hi


def _exact_regrid(case, seed):
    _, cols = _regrid_inputs(case, seed)
    m, M, r, z, ids = (x.cpu().numpy() for x in cols)
    n_r, n_z = case["n_r"], case["n_z"]
    order = np.lexsort((ids, r))
    alive = int(np.isfinite(r).sum())
    size, off = _split(alive, n_r)
    if size.min() < 2 * n_z:  # single-particle cells take the gas scale height
        return None
    start, num, bounds, V = [], [], [], []
    ranked = r[order[:alive]]
    for k in range(n_r):
        part = order[off[k]:off[k + 1]]
        rlo, rhi = _edges(ranked, off[k], size[k], k, n_r)
        part = part[np.lexsort((ids[part], z[part]))]
        order[off[k]:off[k + 1]] = part
        csize, coff = _split(size[k], n_z)
        for c in range(n_z):
            zlo, zhi = _edges(z[part], coff[c], csize[c], c, n_z)
            start.append(off[k] + coff[c])
            num.append(csize[c])
            bounds += [rlo, rhi, zlo, zhi, 0.5 * (rlo + rhi), 0.5 * (zlo + zhi)]
            V.append(math.pi * (rhi * rhi - rlo * rlo) * (zhi - zlo))
    return [m[order], M[order], r[order], z[order], ids[order], np.array(start), np.array(num, np.int32),
            np.array(bounds), np.array(V), np.array([alive]), np.array([0], np.int32)]


def _exact_snapshot(case, seed):
    edges, re, me = _snapshot_edges(case)
    P = _layout(case)[0][0]
    n = case["n_r"] * case["n_z"] * case["per_cell"]
    m, r, _ = (x.cpu().numpy() for x in _midrun(P, n, seed * 64))
    Mi = P["dust_to_gas"] * 2.0 * math.pi * P["sigma0"] * (P["r_out"] - P["r_in"]) / AU * AU * AU / n  # p = 1
    mom = np.zeros((len(edges) - 1, 5))
    b = np.searchsorted(edges, r, side="right") - 1
    for k in range(len(edges) - 1):
        x = m[b == k]
        mom[k] = [Mi * x.size] + [Mi * math.fsum(x**p) for p in (1, 2, 3)] + [x.size]
    br, bm = np.searchsorted(re, r, side="right") - 1, np.searchsorted(me, m, side="right") - 1
    ok = (br >= 0) & (br < len(re) - 1) & (bm >= 0) & (bm < len(me) - 1)
    nm = len(me) - 1
    cnt = np.bincount(br[ok] * nm + bm[ok], minlength=(len(re) - 1) * nm).reshape(len(re) - 1, nm)
    return {"moments": mom, "map": cnt * Mi}


def exact(case, seed):
    return {"cell": _exact_cell, "transport": _exact_transport, "regrid": _exact_regrid,
            "snapshot": _exact_snapshot}.get(case["kind"], lambda c, s: None)(case, seed)
