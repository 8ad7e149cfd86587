"""The runs whose speed counts, each through the package's public entry points.

A case is one avalanche run as a user's program makes it: a gas, a field and
primaries already uploaded (`prepare`), then `Avalanche.run` (or a replay of
its captured graph) and the endpoints that it wrote, in the order of their
electron ids: the slots of the new electrons depend on scheduling, the
electrons themselves only on the seed.  Sizes are those of the package's
workloads, tests and benchmark, and smaller and ragged ones of the same kinds.
"""
import math

import numpy as np
import torch

from paper_2509_15377_gb300 import avalanche as A
from paper_2509_15377_gb300 import workloads as W

FLOAT_KEYS = ("x0", "y0", "z0", "t0", "e0", "x1", "y1", "z1", "t1", "e1")
WHOLE_KEYS = ("status", "aval", "uid", "n_flight")
SIGNAL_BINS, SIGNAL_DT = 2000, 0.05     # 100 ns in bins of 50 ps

# One entry per option that a case may carry, with the value most runs use.
DEFAULTS = {
    "field": "plate",         # plate, coax, grid, mesh
    "gas": "basic",           # basic, physical (anisotropy, sharing, attachment)
    "precision": "mixed",     # mixed, fp64
    "mode": "batched",        # batched, plain, graph (a captured batched run)
    "majorant": "banded",     # banded, global
    "avalanches": 0,
    "e_lo": 40000.0, "e_hi": 40000.0,   # plate: V/cm, one field per avalanche
    "primaries": 1.0,         # plate: mean number per avalanche (Poisson above 1)
    "r_lo": 0.1, "r_hi": 0.1,           # coax, grid, mesh: start radius (cm)
    "voltage": 1500.0,
    "cells": 0,               # grid: nodes per axis; mesh: cubes per axis
    "signal": False, "crossing": False, "observables": False,
    "block": 0, "refill": 0, "phase": 0,  # launch shape, 0 = the library's choice
}


def _case(name, **kw):
    c = dict(DEFAULTS, name=name)
    c.update(kw)
    return c


def listed():
    return [
        # a handful of avalanches at a time: a program that looks at events one by one;
        # few electrons are alive, so one electron's chain of flights sets the time
        _case("plate_few", avalanches=8),
        # the parallel-plate configuration: 1000 avalanches, gain 1e3, and its observables
        _case("plate_1000", avalanches=1000, observables=True),
        # the benchmark's step: 4096 avalanches replayed as a graph, at its launch shape
        _case("plate_batched_4096", avalanches=4096, e_lo=30000.0, e_hi=50000.0, primaries=3.0,
              mode="graph", block=1024, refill=32, phase=1),
        # RunOptions as they stand: the global majorant, every flight tested against nu_max
        _case("plate_global", avalanches=500, majorant="global"),
        # the general gas: anisotropic scattering, ionisation sharing, attachment
        _case("plate_physical", avalanches=767, gas="physical", e_lo=30000.0, e_hi=50000.0,
              primaries=3.0),
        # induced anode signals in 2000 bins; signals and crossings with the general gas,
        # whose runs give the same electrons again
        _case("plate_signal", avalanches=500, gas="physical", e_lo=30000.0, e_hi=50000.0,
              primaries=3.0, signal=True),
        # endpoints at the exact boundary crossing
        _case("plate_crossing", avalanches=1000, gas="physical", crossing=True),
        # the tube with 1 T axial field: a long drift, then the avalanche at the wire
        _case("coax_b", field="coax", avalanches=512, r_lo=0.05, r_hi=0.11),
        # the regular field map of the benchmark
        _case("grid_256", field="grid", avalanches=128, voltage=1810.0, cells=256),
        # the tetrahedral field map, graded towards the wire
        _case("mesh_32", field="mesh", avalanches=48, r_lo=0.05, r_hi=0.05, voltage=1810.0,
              cells=32),
        # double precision throughout
        _case("fp64_batched", avalanches=300, precision="fp64"),
        # one avalanche at a time, one launch per generation
        _case("fp64_plain", avalanches=2, precision="fp64", mode="plain"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["plate", "plate", "options", "map", "fp64"])
    c = dict(DEFAULTS)
    if kind == "plate":
        e = round(rng.uniform(3.0e4, 4.2e4), 1)
        c.update(avalanches=log(4, 2000), e_lo=e, e_hi=round(e + rng.uniform(0.0, 8.0e3), 1),
                 primaries=rng.choice([1.0, 3.0]), observables=rng.random() < 0.5,
                 mode=rng.choice(["batched", "graph"]))
        if rng.random() < 0.4:
            c.update(block=rng.choice([768, 896, 1024]), refill=32, phase=1)
    elif kind == "options":
        c.update(avalanches=log(20, 1000), signal=rng.random() < 0.4, crossing=rng.random() < 0.4,
                 majorant=rng.choice(["banded", "banded", "global"]))
        c["gas"] = "physical" if c["signal"] or c["crossing"] else rng.choice(["basic", "physical"])
        if c["majorant"] == "global":
            c["avalanches"] = min(c["avalanches"], 400)
    elif kind == "map":
        f = rng.choice(["coax", "grid", "mesh"])
        r = round(rng.uniform(0.03, 0.07), 4)
        c.update(field=f, avalanches=log(24, 120), r_lo=r, r_hi=round(r * rng.uniform(1.0, 1.3), 4),
                 voltage=1500.0 if f == "coax" else round(rng.uniform(1700.0, 1810.0), 1),
                 cells={"coax": 0, "grid": log(65, 256), "mesh": log(12, 32)}[f])
    else:
        c.update(precision="fp64", e_lo=round(rng.uniform(3.0e4, 4.0e4), 1),
                 majorant=rng.choice(["banded", "banded", "global"]))
        c["e_hi"] = c["e_lo"]
        if rng.random() < 0.3:
            c.update(mode="plain", avalanches=1, majorant="banded")
        else:
            c.update(avalanches=log(20, 300))
            if c["majorant"] == "global":
                c["avalanches"] = min(c["avalanches"], 100)
    return c


# ------------------------------------------------------------------ inputs
def _gas(case):
    return W.argon_like_physical_gas() if case["gas"] == "physical" else W.argon_like_gas()


def _workload(case, seed):
    """Gas, field and primaries of the case from the seed."""
    n, f = case["avalanches"], case["field"]
    if f == "plate":
        if case["primaries"] > 1.0 or case["e_hi"] > case["e_lo"]:
            w = W.plate_batched(n, case["e_lo"], case["e_hi"], case["primaries"], seed=seed)
        else:
            w = W.plate(n, case["e_lo"], seed=seed)
        w.gas = _gas(case)
        return w
    # the tube's primaries; on a map they start half-way along it
    w = W.coax(n, voltage=case["voltage"], b_axial=1.0 if f == "coax" else 0.0,
               r_lo=case["r_lo"], r_hi=case["r_hi"], seed=seed)
    w.gas = _gas(case)
    if f == "grid":
        w.field = W.coax_grid_map(n=case["cells"], voltage=case["voltage"])
    elif f == "mesh":
        w.field = W.coax_mesh_map(cells=case["cells"], voltage=case["voltage"], seed=seed,
                                  grading=4.0)
    if f != "coax":
        w.primaries.z[:] = 0.5
        w.t_max = 1000.0
    return w


def _electrons(case):
    """Mean number of electrons of one primary: the plate's gain is
    exponential in the field (97, 996 and 9150 at 30, 40 and 50 kV/cm), the
    tube's and the maps' depend on the voltage alone."""
    if case["field"] == "plate":
        lo, hi = (4.575 + 0.2275e-3 * (e - 3.0e4) for e in (case["e_lo"], case["e_hi"]))
        return math.exp(lo) if hi - lo < 1e-6 else (math.exp(hi) - math.exp(lo)) / (hi - lo)
    return 6376.0 if case["field"] == "coax" else 1.1e5 * math.exp((case["voltage"] - 1810.0) / 95.0)


def _capacity(case):
    """Room for the run: its mean size and half as much, and more where few
    avalanches spread widely."""
    primaries = case["avalanches"] * case["primaries"]
    mean = _electrons(case) * primaries
    return int(1.5 * mean + 10.0 * mean / math.sqrt(primaries)) + 4096


def prepare(case, seed):
    w = _workload(case, seed)
    av = A.Avalanche(0)
    av.set_gas(w.gas)
    av.set_field(w.field)
    opt = A.RunOptions(
        seed=seed, t_max=w.t_max,
        precision=A.GT_FP64 if case["precision"] == "fp64" else A.GT_MIXED,
        mode=A.GT_PLAIN if case["mode"] == "plain" else A.GT_BATCHED,
        majorant=A.GT_MAJORANT_BANDED if case["majorant"] == "banded" else A.GT_MAJORANT_GLOBAL,
        block=case["block"], refill_period=case["refill"], flights_per_phase=case["phase"],
        crossing=int(case["crossing"]))
    if case["signal"]:
        opt.signal_kind, opt.signal_bins, opt.signal_dt = W.W_PLATE, SIGNAL_BINS, SIGNAL_DT
    capacity = _capacity(case)
    prim = av.primaries_device(w.primaries)
    out = {k: torch.zeros(capacity, dtype=torch.float64, device="cuda") for k in FLOAT_KEYS}
    out.update({k: torch.zeros(capacity, dtype=torch.int64 if k == "uid" else torch.int32,
                               device="cuda") for k in WHOLE_KEYS})
    return {"av": av, "opt": opt, "prim": prim, "capacity": capacity, "primaries": w.primaries,
            "gap": w.field.gap, "signal": case["signal"], "observables": case["observables"],
            "out": out,
            "graph": av.graph(prim, opt, capacity) if case["mode"] == "graph" else None}


def run(s):
    av = s["av"]
    if s["graph"] is not None:
        s["graph"].launch(s["opt"].seed)
        st = s["graph"].stats(allow=(A.GT_OK,))
    else:
        st = av.run(s["prim"], s["opt"], s["capacity"], allow=(A.GT_OK,))
    # the electrons in the order of their ids, zeros after the last
    n, ep, out = st["n_endpoints"], av.ep, dict(s["out"])
    order = torch.argsort(ep["uid"][:n])
    for k in FLOAT_KEYS + WHOLE_KEYS:
        torch.index_select(ep[k][:n], 0, order, out=out[k][:n])
    out["electrons"], out["tallies"] = ep["electrons"], ep["tallies"]
    out["counts"] = [n, st["real_collisions"], st["null_collisions"], st["flights"]]
    if s["signal"]:
        out["signal"] = ep["signal"]
    if s["observables"]:
        out["observables"] = av.observables(n, s["primaries"], W.ANODE, W.ANODE, s["gap"])
    return out


def work(case):
    """A primary's or new electron's record and endpoint once (76 and 112
    bytes), and about 190 operations for each of its flights (one random
    block, the majorant, the motion, the rate and the scattering)."""
    electrons = _electrons(case) * case["avalanches"] * case["primaries"]
    flights = 330.0 * electrons
    if case["field"] == "plate":
        if case["majorant"] == "global":
            flights *= 5.6
    else:  # the drift to the wire
        r = 0.5 * (case["r_lo"] + case["r_hi"])
        flights += case["avalanches"] * 8.0e6 * r * r * 1500.0 / case["voltage"]
    nbytes = 188.0 * electrons
    if case["signal"]:
        nbytes += 8.0 * SIGNAL_BINS * case["avalanches"]
    return {"bytes": nbytes, "flops": 190.0 * flights}


# ----------------------------------------------------- the method in 64 bits
M32 = 0xFFFFFFFF


def _s64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., 2011) on int64 tensors of 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * _s64(0xCD9E8D57)
        c0, c1, c2, c3 = (((b >> 32) & M32) ^ c1 ^ k0, b & M32,
                          ((a >> 32) & M32) ^ c3 ^ k1, a & M32)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _child_id(parent, flight):
    """SplitMix64's output (Steele, Lea, Flood, 2014) of the flight-th step."""
    def shr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)

    z = parent + (flight + 1) * _s64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * _s64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _s64(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _direction(u, v):
    ct = 1.0 - 2.0 * u
    st = torch.sqrt(torch.clamp(1.0 - ct * ct, min=0.0))
    return st * torch.cos(2.0 * math.pi * v), st * torch.sin(2.0 * math.pi * v), ct


def exact(case, seed):
    """The plate runs in double precision, flight by flight over all living
    electrons at once.  The mixed-precision step rounds its way to other
    trajectories, which have no value in 64 bits."""
    if case["precision"] != "fp64" or case["field"] != "plate" or case["gas"] != "basic" \
            or case["majorant"] != "banded" or case["e_hi"] > case["e_lo"]:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    w = _workload(case, seed)
    g, p, L = w.gas, w.primaries, w.gas.n_levels
    acc, efield, gap = 1.75882001076e-3, w.field.e0, w.field.gap
    f64 = torch.float64

    def on(a, dt=f64):
        return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device=dev)

    cum = on(np.cumsum(g.rate, axis=1))
    thr, kind = on(g.threshold), on(g.level_type, torch.int64)
    per = int(round(g.band_width / g.d_eps))
    n_bands = -(-(g.n_nodes - 1) // per)
    total = np.cumsum(g.rate, axis=1)[:, -1]
    band = on([total[b * per:(b + 1) * per + 1].max() for b in range(n_bands)])

    def band_of(eps):
        return band[torch.clamp((eps / (per * g.d_eps)).floor().long(), 0, n_bands - 1)]

    def u01(word):
        return (word.to(f64) + 0.5) / 4294967296.0

    # the living electrons: position, time, velocity; id, avalanche, flights; row
    s0 = np.sqrt(2.0 * acc * p.e)
    F = torch.stack([on(a) for a in (p.x, p.y, p.z, p.t, s0 * p.dx, s0 * p.dy, s0 * p.dz)])
    I = torch.stack([on(p.uid.view(np.int64), torch.int64), on(p.aval, torch.int64),
                     torch.zeros(p.n, dtype=torch.int64, device=dev),
                     torch.arange(p.n, device=dev)])
    starts = [torch.stack([on(a) for a in (p.x, p.y, p.z, p.t, p.e)])]
    ids = [I[:2]]
    rows, ends, whole = [], [], []
    n_all = p.n
    tallies = torch.zeros(p.n_avalanches * (L + 1), dtype=torch.int64, device=dev)
    while F.shape[1]:
        x, y, z, t, vx, vy, vz = F
        uid, av, nf, row = I
        w0, w1, w2, w3 = _philox(nf, 2 * av, uid & M32, (uid >> 32) & M32, seed)
        eps = (vx * vx + vy * vy + vz * vz) / (2.0 * acc)
        tau = 2.0 / band_of(eps)
        gain = vz * efield * tau + 0.5 * acc * efield * efield * tau * tau
        nu = band_of(eps + torch.clamp(gain, min=0.0))
        dt = -torch.log(u01(w0)) / nu
        stop = dt >= tau
        dt = torch.where(stop, tau, dt)
        timed = t + dt > w.t_max
        dt = torch.where(timed, w.t_max - t, dt)
        az = acc * efield
        x, y, z = x + vx * dt, y + vy * dt, z + vz * dt + 0.5 * az * dt * dt
        vz = vz + az * dt
        t = torch.where(timed, torch.full_like(t, w.t_max), t + dt)
        nf = nf + 1
        status = torch.where(z >= gap, W.ANODE, torch.where(z < 0.0, W.CATHODE,
                                                            torch.where(timed, W.TIME, 0)))
        eps = (vx * vx + vy * vy + vz * vz) / (2.0 * acc)
        xk = torch.clamp(eps / g.d_eps, max=g.n_nodes - 1.0)
        k = torch.clamp(xk.long(), max=g.n_nodes - 2)
        c0, c1 = cum[k], cum[k + 1]
        c = c0 + (xk - k).unsqueeze(1) * (c1 - c0)
        R = u01(w1) * nu
        lvl = torch.clamp((c <= R.unsqueeze(1)).sum(1), max=L - 1)
        test = (status == 0) & ~stop
        real = test & (R < c[:, -1]) & ((kind[lvl] == W.ELASTIC) | (eps >= thr[lvl]))
        tallies.index_add_(0, av * (L + 1) + torch.where(real, lvl, L), test.long())
        nx, ny, nz = _direction(u01(w2), u01(w3))
        sp = torch.sqrt(vx * vx + vy * vy + vz * vz)
        cchi = torch.where(sp > 0.0, (vx * nx + vy * ny + vz * nz) / sp, 0.0)
        new = torch.where(kind[lvl] == W.ELASTIC, eps * (1.0 - g.recoil * (1.0 - cchi)),
                          eps - thr[lvl])
        ion = (real & (kind[lvl] == W.IONISATION)).nonzero()[:, 0]
        if len(ion):
            a0, a1, a2, _ = _philox(nf[ion] - 1, 2 * av[ion] + 1, uid[ion] & M32,
                                    (uid[ion] >> 32) & M32, seed)
            share = u01(a0) * new[ion]
            new[ion] = new[ion] - share
            sx, sy, sz = _direction(u01(a1), u01(a2))
            ss = torch.sqrt(2.0 * acc * share)
            born = torch.stack([x[ion], y[ion], z[ion], t[ion], ss * sx, ss * sy, ss * sz])
            tags = torch.stack([_child_id(uid[ion], nf[ion] - 1), av[ion],
                                torch.zeros_like(ion), n_all + torch.arange(len(ion), device=dev)])
            starts.append(torch.cat([born[:4], share.unsqueeze(0)]))
            ids.append(tags[:2])
            n_all += len(ion)
        sp = torch.sqrt(2.0 * acc * torch.clamp(new, min=0.0))
        vx, vy, vz = (torch.where(real, sp * d, v) for d, v in ((nx, vx), (ny, vy), (nz, vz)))
        F, I = torch.stack([x, y, z, t, vx, vy, vz]), torch.stack([uid, av, nf, row])
        gone = status != 0
        if bool(gone.any()):
            G = F[:, gone]
            ends.append(torch.cat([G[:4], ((G[4:] ** 2).sum(0) / (2.0 * acc)).unsqueeze(0)]))
            whole.append(torch.stack([status[gone], nf[gone]]))
            rows.append(row[gone])
            F, I = F[:, ~gone], I[:, ~gone]
        if len(ion):
            F, I = torch.cat([F, born], 1), torch.cat([I, tags], 1)
    start, tag = torch.cat(starts, 1), torch.cat(ids, 1)
    row = torch.cat(rows)
    end, fin = torch.empty_like(start), torch.empty_like(tag)
    end[:, row], fin[:, row] = torch.cat(ends, 1), torch.cat(whole, 1)
    order = torch.argsort(tag[0])

    def padded(a):  # run()'s arrays have a slot for every electron there is room for
        return torch.nn.functional.pad(a[:, order], (0, _capacity(case) - n_all))

    electrons = torch.bincount(tag[1], minlength=p.n_avalanches)
    start, end, tag, fin = padded(start), padded(end), padded(tag), padded(fin)
    out = dict(zip(FLOAT_KEYS, list(start) + list(end)))
    out.update(status=fin[0].int(), aval=tag[1].int(), uid=tag[0], n_flight=fin[1].int(),
               electrons=electrons, tallies=tallies.view(-1, L + 1))
    out["counts"] = [n_all, int(tallies.view(-1, L + 1)[:, :L].sum()),
                     int(tallies.view(-1, L + 1)[:, L].sum()), int(fin[1].sum())]
    return out
