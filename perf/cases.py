"""What this library is used for, as cases that can be timed and compared.

A case is a dict of plain values.  Its "kind" is the call that a program makes:

  window      advance an ensemble to the end of an observation window, then read the clocks, the
              gauges and every member's state (and the running maxima where they are tracked)
  assimilate  sample the gauges and let the particle filter weigh and resample the ensemble
  maps        exceedance and percentile maps of the running maximum depth
  adjoint     a window's gauge misfit and its gradients
  batch       advance an uneven batch of scenarios by a window, then read clocks and states

Everything runs through the package's public binding (`capi`).  Inputs are made on the GPU from
the seed: terrain of the kind `synth.make_terrain` makes (3 m cells, a 0.5 % slope to the eastern
outflow edge, hills, 10 m buildings, smoother roads), a thin layer of water that leaves some cells
dry, the triangular 60 mm/h storm, and the prior's rain multipliers and Manning scales.  `exact`
is the same scheme, filter and maps in plain torch and numpy, in 64 bits.
"""
import math

import numpy as np
import torch

from paper_2302_08341_gb300 import capi, synth

DEV = "cuda"
G = 9.81
DX = 3.0
BLOCK = 300.0          # rain blocks (s)
SLOPE = 0.005          # bed slope past the outflow edge
WALL = 1.0e6           # bed of the cells outside a land-cover domain
L2_BYTES = 126e6       # a state that fits stays on the chip between the steps of a window
LEVELS = (0.1, 0.5, 0.9)
THRESHOLD = 0.2


def listed():
    w, a = {"kind": "window"}, {"kind": "adjoint"}
    return [
        # one small deterministic model: the shortest steps, where launches and latency count
        dict(w, name="window_256_single", ny=256, nx=256, members=1, seconds=300.0, h0=0.05),
        # the paper's share of one of its devices (12 members) at its fixed 0.25 s step, on a
        # ragged grid with a river entering in the west and the running maxima tracked
        dict(w, name="window_river_12_tracked", ny=777, nx=1013, members=12, seconds=20.0, h0=0.05,
             dt_fixed=0.25, track=True, inflow=True),
        # the benchmark's ensemble: the largest work, bound by memory
        dict(w, name="window_ensemble_96", ny=2000, nx=2000, members=96, seconds=30.0, h0=0.05),
        # deep water: every member at its own step length (Eq. 4 binds)
        dict(w, name="window_deep_16", ny=1000, nx=1000, members=16, seconds=30.0, h0=1.0),
        # land cover with drainage on an irregular domain, per-member class roughness
        dict(w, name="window_land_32", ny=1200, nx=1310, members=32, seconds=30.0, h0=0.03, land=True),
        # risk maps: between two resamplings the weights are unequal, right after one equal
        dict(kind="maps", name="maps_unequal_96", ny=2000, nx=2000, members=96, equal=False),
        dict(kind="maps", name="maps_equal_20", ny=517, nx=1003, members=20, equal=True),
        # one assimilation with resampling: the filter and the copies of the duplicated members
        dict(kind="assimilate", name="assimilate_96", ny=1000, nx=1000, members=96, gauges=6),
        # gradients of one model's window, and of an ensemble's with and without land cover
        dict(a, name="adjoint_1024_single", ny=1024, nx=1024, members=1, samples=5, sample_dt=60.0,
             gauges=8, h0=0.08, grad_h0=True),
        dict(a, name="adjoint_ensemble_24", ny=1000, nx=1000, members=24, samples=1, sample_dt=60.0,
             gauges=6, h0=0.08),
        dict(a, name="adjoint_land_8", ny=600, nx=707, members=8, samples=2, sample_dt=20.0, gauges=6,
             h0=0.05, land=True),
        # many towns at once, each with its own size and storm
        dict(kind="batch", name="batch_16_uneven", scenarios=16, side_lo=256, side_hi=1024, members=1,
             seconds=60.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["window", "window", "window", "assimilate", "maps", "adjoint", "adjoint", "batch"])
    if kind == "window":
        ny, nx, m = _log(rng, 64, 2000), _log(rng, 64, 2000), _log(rng, 1, 96)
        steps = max(4, min(300, int(3e9 / (ny * nx * m))))
        c = dict(kind=kind, ny=ny, nx=nx, members=m, seconds=float(steps), h0=rng.choice([0.03, 0.05, 1.0]))
        form = rng.choice(["plain", "plain", "fixed", "land", "track", "river"])
        if form == "fixed":
            c.update(dt_fixed=0.25, seconds=max(1.0, steps // 4 * 1.0))
        elif form == "land":
            c.update(land=True, h0=0.03)
        elif form == "track":
            c.update(track=True)
        elif form == "river":
            c.update(inflow=True)
        return c
    if kind == "assimilate":
        return dict(kind=kind, ny=_log(rng, 100, 1000), nx=_log(rng, 100, 1000), members=_log(rng, 4, 96),
                    gauges=rng.randint(1, 40))
    if kind == "maps":
        return dict(kind=kind, ny=_log(rng, 100, 1500), nx=_log(rng, 100, 1500), members=_log(rng, 4, 128),
                    equal=rng.random() < 0.5)
    if kind == "adjoint":
        ny, nx, m = _log(rng, 64, 1000), _log(rng, 64, 1000), _log(rng, 1, 24)
        n = max(6, min(200, int(1.2e9 / (ny * nx * m))))
        return dict(kind=kind, ny=ny, nx=nx, members=m, samples=2, sample_dt=float(n // 2),
                    gauges=rng.randint(1, 12), h0=rng.choice([0.05, 0.08]), land=rng.random() < 0.3,
                    grad_h0=rng.random() < 0.3)
    return dict(kind=kind, scenarios=_log(rng, 4, 24), side_lo=rng.randint(100, 300),
                side_hi=rng.randint(400, 1024), members=rng.choice([1, 1, 2, 4]), seconds=float(rng.randint(20, 60)))


# ---- inputs ------------------------------------------------------------------------------------

class _Rand:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed)

    def uniform(self, lo, hi, *shape):
        return torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64) * (hi - lo) + lo

    def integers(self, lo, hi, *shape):
        return torch.randint(lo, hi + 1, shape, generator=self.g, device=DEV)


def _terrain(rand, ny, nx):
    """Bed, Manning n and the building and road masks, as synth.make_terrain describes them."""
    r = torch.arange(ny, device=DEV)
    c = torch.arange(nx, device=DEV)
    z = (SLOPE * DX * (nx - 1 - c).double())[None, :].expand(ny, nx).clone()
    cy, cx = rand.uniform(0, ny * DX, 40), rand.uniform(0, nx * DX, 40)
    amp, sig = rand.uniform(0, 1.0, 40), rand.uniform(10.0, 40.0, 40)
    gy = torch.exp(-(((r + 0.5) * DX)[:, None] - cy) ** 2 / (2 * sig * sig)) * amp
    gx = torch.exp(-(((c + 0.5) * DX)[:, None] - cx) ** 2 / (2 * sig * sig))
    z += gy @ gx.T
    road = ((r % 41) < 3)[:, None] | ((c % 37) < 2)[None, :]
    by, bx = ny // 16 + 1, nx // 16 + 1
    put = rand.uniform(0, 1, by, bx) < 0.22
    h, w = rand.integers(4, 12, by, bx), rand.integers(4, 12, by, bx)
    oy, ox = rand.integers(0, 4, by, bx), rand.integers(0, 4, by, bx)
    at = lambda v: v[(r // 16)[:, None], (c // 16)[None, :]]  # noqa: E731
    ly, lx = (r % 16)[:, None], (c % 16)[None, :]
    b = at(put) & (ly >= at(oy)) & (ly < at(oy + h)) & (lx >= at(ox)) & (lx < at(ox + w)) & ~road
    z = torch.where(b, z + 10.0, z)
    z -= z.min()
    n = torch.where(road, 0.03, 0.05)
    return z.float(), n.float(), b, road


def _depths(rand, ny, nx, members, h0, building):
    """Initial depths [members][ny][nx]: a layer around h0 (deeper by member and place), one cell
    in eight dry, and no water on one roof in two."""
    f = rand.uniform(0.5, 1.5, ny, nx)
    f = torch.where(rand.uniform(0, 1, ny, nx) < 0.125, torch.zeros_like(f), f)
    if h0 < 0.5:
        f = torch.where(building & (rand.uniform(0, 1, ny, nx) < 0.5), torch.zeros_like(f), f)
    else:
        f = 0.8 + 0.2 * f       # deep water everywhere
    out = torch.empty(members, ny, nx, device=DEV)
    for m, s in enumerate(rand.uniform(0.7, 1.3, members).tolist()):
        out[m] = (f * (h0 * s)).float()
    return out


def _land(rand, ny, nx, building, road):
    """Class per cell: roads and buildings hardened, ponds, green land; outside a disc-like domain
    that reaches the eastern edge (about a tenth to a third of the box lies outside)."""
    cls = torch.zeros(ny, nx, dtype=torch.uint8, device=DEV)
    cls[building | road] = 2
    for y, x in zip(rand.integers(0, ny - 1, 6).tolist(), rand.integers(0, nx - 1, 6).tolist()):
        blk = cls[y:y + 20, x:x + 24]
        blk[blk == 0] = 1
    y = (torch.arange(ny, device=DEV)[:, None] - 0.5 * ny) / (0.5 * ny)
    x = (torch.arange(nx, device=DEV)[None, :] - 0.62 * nx) / (0.5 * nx)
    cls[torch.hypot(x, y) > 1.08] = 3
    return cls.cpu().numpy()


def _prior(rand, members):
    rm = torch.exp(0.3 * torch.randn(members, generator=rand.g, device=DEV, dtype=torch.float64))
    return rm.float().cpu().numpy(), rand.uniform(0.6, 1.4, members).float().cpu().numpy()


def _land_prior(rand, members):
    n = torch.stack([rand.uniform(lo, hi, members) for lo, hi in synth.N_RANGES], 1)
    d = rand.uniform(0.5, 1.5, members) * (synth.I_DRN_MM_H * synth.MM_PER_H)
    return n.float().cpu().numpy(), d.float().cpu().numpy()


def _cells(rand, ny, nx, n):
    return rand.integers(0, ny * nx - 1, n).int().cpu().numpy()


def _sides(case):
    """The scenarios' sides, spread over [side_lo, side_hi] in no order."""
    lo, hi = case["side_lo"], case["side_hi"]
    return [lo + int((hi - lo + 1) * ((0.37 + 0.6180339887 * i) % 1.0)) for i in range(case["scenarios"])]


def _inputs(case, seed):
    """What a program has in hand: the arrays of the case."""
    rand = _Rand(seed)
    if case["kind"] == "batch":
        sides = _sides(case)
        x = {"sides": sides, "terr": [_terrain(rand, s, s)[:2] for s in sides]}
        k = case["scenarios"] * case["members"]
        x["rm"], x["sc"] = _prior(rand, k)
        x["rain"] = rand.uniform(20.0, 100.0, case["scenarios"]).tolist()
        x["hy"] = [synth.hyetograph_constant(v, 900.0) for v in x["rain"]]
        return x
    ny, nx, m = case["ny"], case["nx"], case["members"]
    x = {}
    x["z"], x["n"], building, road = _terrain(rand, ny, nx)
    x["rm"], x["sc"] = _prior(rand, m)
    x["hy"] = synth.hyetograph_triangular(60.0, 1200.0, 3600.0)
    if case["kind"] in ("window", "adjoint"):
        x["h0"] = _depths(rand, ny, nx, m, case["h0"], building)
        x["cells"] = _cells(rand, ny, nx, case.get("gauges", 6))
        if case.get("land"):
            x["cls"] = _land(rand, ny, nx, building, road)
            x["lc_n"], x["lc_d"] = _land_prior(rand, m)
            x["sc"] = np.ones(m, np.float32)
        if case.get("inflow"):
            x["inflow"] = (ny // 3, ny // 3 + max(1, ny // 20), np.array([4.0, 6.0, 9.0] * 4, np.float32))
        if case["kind"] == "adjoint":
            x["d"] = rand.uniform(0.0, 3.0 * case["h0"], case["samples"], case["gauges"]).cpu().numpy()
    elif case["kind"] == "assimilate":
        x["h0"] = _depths(rand, ny, nx, m, 0.05, building)
        x["cells"] = _cells(rand, ny, nx, case["gauges"])
        # what the observation operator gave for every member, and what was observed
        x["y"] = rand.uniform(0.05, 0.15, m, case["gauges"]).float().cpu().numpy()
        x["d"] = rand.uniform(0.08, 0.12, case["gauges"]).cpu().numpy()
        x["u"], x["beta"] = synth.pf_draws(seed, 1, m)
    else:  # maps: depths that follow the members' rain; on roofs thin films from 1e-6 m up
        base = rand.uniform(0.02, 0.45, ny, nx)
        x["h0"] = torch.empty(m, ny, nx, device=DEV)
        for i, v in enumerate(x["rm"].tolist()):
            h = base * v ** 1.2 * rand.uniform(0.9, 1.1, ny, nx)
            film = torch.exp(rand.uniform(math.log(1e-6), math.log(1e-2), ny, nx))
            x["h0"][i] = torch.where(building, film, h).float()
        w = rand.uniform(0.2, 1.0, m).cpu().numpy()
        x["w"] = w / w.sum()
    return x


# ---- the library's side ------------------------------------------------------------------------

def prepare(case, seed):
    x = _inputs(case, seed)
    if case["kind"] == "batch":
        k = case["members"]
        b = capi.Batch([z.cpu().numpy() for z, _ in x["terr"]], [n.cpu().numpy() for _, n in x["terr"]])
        counts = np.full(case["scenarios"], k, np.int32)
        b.init(x["hy"], x["rm"], x["sc"], np.full(case["scenarios"], 1.0e7), members=counts if k > 1 else None)
        out = [torch.empty(k, 3, s, s, device=DEV) for s in x["sides"]]
        return {"case": case, "batch": b, "t": 0.0, "out": out}
    p = capi.Params.default(dt_fixed=case.get("dt_fixed", 0.0))
    m = case["members"]
    g = capi.Grid(x["z"], x["n"], p)
    if "cls" in x:
        g.set_land_cover(x["cls"], synth.LAND_CLASSES)
    g.ensemble_init(m, x["rm"], x["sc"], x["hy"], h0=x["h0"])
    s = {"case": case, "grid": g, "t": 0.0, "cells": x.get("cells")}
    if "cls" in x:
        g.set_land_params(x["lc_n"], x["lc_d"])
    if "inflow" in x:
        g.set_inflow(*x["inflow"])
    if case["kind"] == "window":
        s["out"] = torch.empty(m, 3, case["ny"], case["nx"], device=DEV)
        if case.get("track"):
            g.track_max_depth(True)
            s["hmax"] = torch.empty(m, case["ny"], case["nx"], device=DEV)
    elif case["kind"] == "maps":
        g.track_max_depth(True)
        if not case["equal"]:
            g.set_members(weights=x["w"])
        s["out"] = (torch.empty(case["ny"], case["nx"], device=DEV),
                    torch.empty(len(LEVELS), case["ny"], case["nx"], device=DEV))
    elif case["kind"] == "assimilate":
        s.update({k: x[k] for k in ("y", "d", "u", "beta")})
        s["out"] = torch.empty(2, 3, case["ny"], case["nx"], device=DEV)
    else:
        s["d"] = x["d"]
    torch.cuda.synchronize()
    return s


def _ok(rc):
    if rc != capi.FLOOD_OK:
        raise RuntimeError("libflood.so returned %d" % rc)


def _read_states(g, members, out):
    """The members' states into a device buffer of the caller's."""
    s = capi.stream_handle(None)
    for k, m in enumerate(members):
        _ok(capi.lib().flood_get_state(g.h, m, capi.ptr(out[k, 0]), capi.ptr(out[k, 1]), capi.ptr(out[k, 2]), s))


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        b = s["batch"]
        s["t"] += case["seconds"]
        b.step(s["t"])
        mem = b.members()
        h = capi.stream_handle(None)
        for i, o in enumerate(s["out"]):
            for m in range(case["members"]):
                _ok(capi.lib().flood_batch_get_member_state(b.h, i, m, capi.ptr(o[m, 0]), capi.ptr(o[m, 1]),
                                                            capi.ptr(o[m, 2]), h))
        return {"t": mem["t"], "steps": mem["steps"], "storage": mem["storage"], "states": s["out"]}
    g = s["grid"]
    if case["kind"] == "window":
        s["t"] += case["seconds"]
        g.advance_to(s["t"])
        y = g.gauge_sample(s["cells"])
        mem = g.members()
        _read_states(g, range(case["members"]), s["out"])
        out = {"t": mem["t"], "steps": mem["steps"], "hmax": mem["hmax"], "gauges": y, "states": s["out"]}
        if case.get("track"):
            h = capi.stream_handle(None)
            for m in range(case["members"]):
                _ok(capi.lib().flood_get_max_depth(g.h, m, capi.ptr(s["hmax"][m]), h))
            out["maxima"] = s["hmax"]
        return out
    if case["kind"] == "assimilate":
        y = g.gauge_sample(s["cells"])
        pf = g.pf_assimilate(s["d"], 0.05, s["u"], s["beta"], y=s["y"], force=True)
        mem = g.members()
        _read_states(g, (0, case["members"] - 1), s["out"])
        # (the rain multipliers walk on with every pass, so a later pass has other ones)
        return {"gauges": y, "weights": pf["weights"], "idx": pf["idx"], "neff": pf["neff"],
                "resampled": int(pf["resampled"]), "rain_mult": mem["rain_mult"], "scale": mem["scale"],
                "weights_after": mem["weights"], "first_last": s["out"]}
    if case["kind"] == "maps":
        g.ensemble_products(THRESHOLD, LEVELS, out=s["out"])
        return {"exceedance": s["out"][0], "percentiles": s["out"][1]}
    o = g.adjoint(s["cells"], s["d"], case["sample_dt"], grad_h0=bool(case.get("grad_h0")))
    out = {k: o[k] for k in ("loss", "grad_rain", "grad_scale", "grad_n")}
    if case.get("grad_h0"):
        out["grad_h0"] = o["grad_h0"]
    if case.get("land"):
        out["grad_class"], out["grad_drain"] = g.adjoint_land_grad()
    return out


def _steps(case):
    """Steps of one pass: the cap of 1 s, the fixed step, or in deep water about half a second."""
    secs = case["samples"] * case["sample_dt"] if case["kind"] == "adjoint" else case["seconds"]
    if case.get("dt_fixed"):
        return secs / case["dt_fixed"]
    return secs / (0.55 if case.get("h0", 0.05) >= 0.5 else 1.0)


def work(case):
    """Bytes: inputs once, outputs once; between the steps of a window (and of an adjoint) the
    state and what the reverse pass needs of it once per step, where they cannot stay on the chip.
    Flops: about 60 per cell for a step's two links and its depth, 130 for their reverse."""
    k = case["kind"]
    if k == "batch":
        cells = sum(v * v for v in _sides(case))
        m, n = case["members"], _steps(case)
        fits = cells * (24 * m + 8) < L2_BYTES
        return {"bytes": cells * (24 * m + 8 + 12 * m) if fits else cells * (24 * m + 8) * n + cells * 12 * m,
                "flops": 60.0 * cells * m * n}
    cells, m = case["ny"] * case["nx"], case["members"]
    if k == "maps":
        return {"bytes": 4.0 * cells * (m + 1 + len(LEVELS)), "flops": float(cells) * m * math.log2(m + 1)}
    if k == "assimilate":
        return {"bytes": 24.0 * cells * 0.4 * m, "flops": 100.0 * m * case["gauges"]}
    n = _steps(case)
    if k == "window":
        per = 24 + (8 if case.get("track") else 0)
        fits = cells * (per * m + 8) < L2_BYTES
        once = cells * (12 * m * 2 + 8)
        return {"bytes": once if fits else cells * (per * m + 8) * n + once, "flops": 60.0 * cells * m * n}
    # adjoint: forward 24 B, recomputation 12 B written, reverse 16 B of states and 24 B of lambda
    fits = cells * m * 36 + cells * 8 < L2_BYTES
    per_step = cells * m * (12 + 16) if fits else cells * (m * (24 + 12 + 16 + 24) + 3 * 8)
    return {"bytes": per_step * n + cells * 12, "flops": 250.0 * cells * m * n}


# ---- the same in 64 bits -----------------------------------------------------------------------

def _link(h1, z1, h2, z2, q, nl, gdt_dx, gdt, lim):
    """Eq. 3, Eq. 2 and the quarter-volume limiter on interior links, with the branch taken made
    explicit (so that its derivative is the branch's)."""
    dz = z2 - z1
    a1, a2 = h1 - dz.clamp(min=0), h2 + dz.clamp(max=0)
    hf = torch.where(a1 >= a2, a1, a2)
    wet = hf > 0
    hs = torch.where(wet, hf, torch.ones_like(hf))
    num = q - gdt_dx * hs * (dz + (h2 - h1))
    qn = num / (1 + gdt * nl * nl * q.abs() * hs.pow(-7.0 / 3.0).clamp(max=1e30))
    up, dn = h1 * lim, -h2 * lim
    qn = torch.where(qn > up, up, torch.where(qn < dn, dn, qn))
    return torch.where(wet, qn, torch.zeros_like(qn))


def _outflow(h, q, nc, gdt_dx, gdt, lim):
    wet = h > 0
    hs = torch.where(wet, h, torch.ones_like(h))
    qn = (q + gdt_dx * hs * (SLOPE * DX)) / (1 + gdt * nc * nc * q.abs() * hs.pow(-7.0 / 3.0).clamp(max=1e30))
    qn = torch.where(qn > hs * lim, hs * lim, qn)
    return torch.where(wet & (qn > 0), qn, torch.zeros_like(qn))


def _step64(h, qx, qy, z, n, sc, rain, dt, drain=None, q_in=None, rows=None):
    """One step of [m][ny][nx] members; dt [m][1][1]; rain: depth added per cell; drain: depth the
    pipes could take."""
    gdt_dx, gdt, lim = G * dt / DX, G * dt, DX / (4 * dt)
    e = _link(h[..., :-1], z[..., :-1], h[..., 1:], z[..., 1:], qx[..., :-1],
              0.5 * sc * (n[..., :-1] + n[..., 1:]), gdt_dx, gdt, lim)
    last = _outflow(h[..., -1:], qx[..., -1:], sc * n[..., -1:], gdt_dx, gdt, lim)
    s = _link(h[:, :-1], z[..., :-1, :], h[:, 1:], z[..., 1:, :], qy[:, :-1],
              0.5 * sc * (n[..., :-1, :] + n[..., 1:, :]), gdt_dx, gdt, lim)
    qx2 = torch.cat([e, last], 2)
    qy2 = torch.cat([s, torch.zeros_like(h[:, :1])], 1)
    west = torch.zeros_like(h[..., :1])
    if q_in is not None:
        west = west.clone()
        west[:, rows[0]:rows[1]] = q_in
    net = torch.cat([west, qx2[..., :-1]], 2) - qx2 + torch.cat([torch.zeros_like(h[:, :1]), s], 1) - qy2
    hn = h + (dt / DX * net + rain)
    if drain is not None:
        sink = torch.minimum(drain.expand_as(hn), hn.clamp(min=0))
        empty = (hn > 0) & (sink >= hn)
        hn = torch.where(empty, torch.zeros_like(hn), hn - sink)
    return torch.where(hn < 0, torch.zeros_like(hn), hn), qx2, qy2


class _Model64:
    """Some members of a case in 64 bits."""

    def __init__(self, case, x, who):
        d = lambda v: torch.as_tensor(np.asarray(v), device=DEV).double()  # noqa: E731
        self.case, self.fixed = case, case.get("dt_fixed", 0.0)
        self.z = x["z"].double()[None]
        self.rm, self.sc = d(x["rm"])[who][:, None, None], d(x["sc"])[who][:, None, None]
        self.hy = np.asarray(x["hy"], np.float64)
        self.h = x["h0"][who].double() if "h0" in x else torch.zeros(len(who), *x["z"].shape, device=DEV).double()
        self.n, self.runoff, self.drains, self.rate = x["n"].double()[None], None, None, None
        if "cls" in x:
            cls = torch.as_tensor(x["cls"], device=DEV).long()
            out = torch.tensor([bool(c[3]) for c in synth.LAND_CLASSES], device=DEV)
            ro = torch.tensor([0.0 if c[3] else c[1] for c in synth.LAND_CLASSES], device=DEV)
            dr = torch.tensor([0.0 if c[3] else float(c[2]) for c in synth.LAND_CLASSES], device=DEV)
            self.cls, self.runoff, self.drains = cls, ro.float().double()[cls][None], dr.double()[cls][None]
            self.z = torch.where(out[cls], torch.full_like(self.z[0], WALL), self.z[0])[None]
            self.n = d(x["lc_n"])[who][:, cls]
            self.rate = d(x["lc_d"])[who][:, None, None]
            self.h = torch.where(out[cls], torch.zeros_like(self.h), self.h)
        self.qx, self.qy = torch.zeros_like(self.h), torch.zeros_like(self.h)
        self.inflow = x.get("inflow")
        m = len(who)
        self.t, self.steps = np.zeros(m), np.zeros(m, np.int64)
        self.top = self.h.clone() if case.get("track") else None

    def plan(self, t_end):
        """Eq. 4 with its cap, landing on rain blocks and the end: step and rain rate by member."""
        hm = np.maximum(self.h.amax((1, 2)).cpu().numpy(), 1e-6)
        dt = np.full(len(hm), self.fixed) if self.fixed else np.minimum(0.7 * DX / np.sqrt(G * hm), 1.0)
        blk = np.floor(self.t / BLOCK)
        stop = np.minimum((blk + 1) * BLOCK, t_end)
        land = self.t + dt >= stop
        dt = np.where(land, stop - self.t, dt)
        nxt = np.where(land, stop, self.t + dt)
        rate = np.array([self.hy[int(b)] if b < len(self.hy) else 0.0 for b in blk])
        q_in = None
        if self.inflow is not None:
            r0, r1, q = self.inflow
            q_in = torch.as_tensor([float(q[int(b)]) / (DX * (r1 - r0)) if b < len(q) else 0.0 for b in blk],
                                   device=DEV).double()[:, None, None]
        return self.t < t_end, dt, nxt, rate, q_in

    def rain(self, dt, rate, rm):
        v = dt * rate * rm
        return v if self.runoff is None else v * self.runoff

    def advance(self, t_end):
        """To t_end, each member with its own steps; yields (dt, rate) of every round."""
        while True:
            on, dt, nxt, rate, q_in = self.plan(t_end)
            if not on.any():
                return
            tt = lambda v: torch.as_tensor(v, device=DEV)[:, None, None]  # noqa: E731
            d, act = tt(np.where(on, dt, 1.0)), tt(on)
            new = _step64(self.h, self.qx, self.qy, self.z, self.n, self.sc, self.rain(d, tt(rate), self.rm), d,
                          None if self.rate is None else self.rate * self.drains * d, q_in,
                          None if self.inflow is None else self.inflow[:2])
            new = [torch.where(act, a, b) for a, b in zip(new, (self.h, self.qx, self.qy))] if not on.all() else new
            self.h, self.qx, self.qy = new
            self.t, self.steps = np.where(on, nxt, self.t), self.steps + on
            if self.top is not None:
                self.top = torch.maximum(self.top, self.h)
            yield d, tt(rate)


def _exact_window(case, x):
    m, cells = case["members"], torch.as_tensor(x["cells"], device=DEV).long()
    out = {"t": [], "steps": [], "hmax": [], "gauges": [], "states": [], "maxima": []}
    group = max(1, int(4e7 // (case["ny"] * case["nx"])))
    for a in range(0, m, group):
        w = _Model64(case, x, list(range(a, min(m, a + group))))
        for _ in w.advance(case["seconds"]):
            pass
        out["t"].append(torch.as_tensor(w.t))
        out["steps"].append(torch.as_tensor(w.steps))
        out["hmax"].append(w.h.amax((1, 2)))
        out["gauges"].append(w.h.flatten(1)[:, cells])
        out["states"].append(torch.stack([w.h, w.qx, w.qy], 1))
        if w.top is not None:
            out["maxima"].append(w.top)
    return {k: torch.cat(v) for k, v in out.items() if v}


def _exact_batch(case, x):
    k, out = case["members"], {"t": [], "steps": [], "storage": [], "states": []}
    for i, (z, n) in enumerate(x["terr"]):
        one = {"z": z, "n": n, "hy": x["hy"][i], "rm": x["rm"][i * k:(i + 1) * k], "sc": x["sc"][i * k:(i + 1) * k]}
        w = _Model64(case, one, list(range(k)))
        for _ in w.advance(case["seconds"]):
            pass
        out["t"].append(w.t)
        out["steps"].append(w.steps)
        out["storage"].append((w.h.sum((1, 2)) * DX * DX).cpu().numpy())
        out["states"].append(torch.stack([w.h, w.qx, w.qy], 1))
    return {j: v if j == "states" else np.concatenate(v) for j, v in out.items()}


def _exact_adjoint(case, x):
    """Reverse mode step by step with the recorded step lengths, by torch's autograd."""
    res = {"loss": [], "grad_rain": [], "grad_scale": [], "grad_h0": [], "grad_class": [], "grad_drain": []}
    grad_n = torch.zeros(case["ny"], case["nx"], device=DEV, dtype=torch.float64)
    cells, obs = torch.as_tensor(x["cells"], device=DEV).long(), torch.as_tensor(x["d"], device=DEV)
    for i in range(case["members"]):
        w = _Model64(case, x, [i])
        tape, loss, seeds = [], 0.0, {}
        before = (w.h, w.qx, w.qy)
        for k in range(case["samples"]):
            for d, rate in w.advance((k + 1) * case["sample_dt"]):
                tape.append((before, d, rate))
                before = (w.h, w.qx, w.qy)
            off = w.h.flatten()[cells] - obs[k]
            loss = loss + float((off * off).sum())
            seeds[len(tape)] = 2 * off
        lam = [torch.zeros_like(w.h) for _ in range(3)]
        leaf = [v.clone().requires_grad_() for v in (w.n, w.rm, w.sc) + ((w.rate,) if w.rate is not None else ())]
        total = [torch.zeros_like(v) for v in leaf]
        for j in range(len(tape), 0, -1):
            if j in seeds:
                lam[0] = lam[0].flatten().index_add(0, cells, seeds[j]).view_as(lam[0])
            (h, qx, qy), d, rate = tape[j - 1]
            tape[j - 1] = None
            v = [a.detach().requires_grad_() for a in (h, qx, qy)]
            n, rm, sc = leaf[:3]
            new = _step64(*v, w.z, n, sc, w.rain(d, rate, rm), d, leaf[3] * w.drains * d if w.rate is not None else None)
            got = torch.autograd.grad(new, v + leaf, lam)
            lam = list(got[:3])
            for a, b in zip(total, got[3:]):
                a += b
        grad_n += total[0][0]
        res["loss"].append(loss)
        res["grad_rain"].append(float(total[1]))
        res["grad_scale"].append(float(total[2]))
        if case.get("grad_h0"):
            res["grad_h0"].append(lam[0][0])
        if w.rate is not None:
            res["grad_class"].append([float(total[0][0][w.cls == q].sum()) for q in range(len(synth.LAND_CLASSES))])
            res["grad_drain"].append(float(total[3]))
    out = {k: np.array(v) for k, v in res.items() if v and k != "grad_h0"}
    out["grad_n"] = grad_n
    if case.get("grad_h0"):
        out["grad_h0"] = torch.stack(res["grad_h0"])
    return out


def _exact_assimilate(case, x):
    m = case["members"]
    lw = -0.5 * (((x["y"].astype(np.float64) - x["d"]) / 0.05) ** 2).sum(1) - math.log(m)
    w = np.exp(lw - lw.max())
    w /= w.sum()
    c = np.cumsum(w)
    c[-1] = 1.0
    idx = np.minimum(np.searchsorted(c, (x["u"] + np.arange(m)) / m, "right"), m - 1)
    # survivors keep their slot; further copies fill the dropped slots in order
    cnt = np.bincount(idx, minlength=m)
    src = np.arange(m)
    extra = iter([p for p in range(m) for _ in range(max(0, cnt[p] - 1))])
    for s in range(m):
        if cnt[s] == 0:
            src[s] = next(extra)
    h = x["h0"].double()
    zero = torch.zeros_like(h[0])
    return {"gauges": h.flatten(1)[:, torch.as_tensor(x["cells"], device=DEV).long()], "weights": w,
            "idx": idx.astype(np.int32), "neff": float(1.0 / (w * w).sum()), "resampled": 1,
            "rain_mult": x["rm"].astype(np.float64)[src] * x["beta"], "scale": x["sc"].astype(np.float64)[src],
            "weights_after": np.full(m, 1.0 / m),
            "first_last": torch.stack([torch.stack([h[int(src[s])], zero, zero]) for s in (0, m - 1)])}


def _exact_maps(case, x):
    m = case["members"]
    w = np.full(m, 1.0 / m) if case["equal"] else x["w"]
    u = torch.as_tensor(np.rint(np.ldexp(w, 60)).astype(np.int64), device=DEV)
    ex = torch.empty(case["ny"], case["nx"], device=DEV, dtype=torch.float64)
    pct = torch.empty(len(LEVELS), case["ny"], case["nx"], device=DEV, dtype=torch.float64)
    thr = float(np.float32(THRESHOLD))
    for r in range(0, case["ny"], 256):
        h = x["h0"][:, r:r + 256]
        ex[r:r + 256] = ((h >= thr) * u[:, None, None]).sum(0).double() * 2.0 ** -60
        v, order = h.sort(0)
        cum = u[order].cumsum(0)
        for q, a in enumerate(LEVELS):
            k = (cum < math.ceil(math.ldexp(a, 60))).sum(0).clamp(max=m - 1)
            pct[q, r:r + 256] = v.gather(0, k[None])[0].double()
    return {"exceedance": ex, "percentiles": pct}


def exact(case, seed):
    f = {"window": _exact_window, "batch": _exact_batch, "adjoint": _exact_adjoint,
         "assimilate": _exact_assimilate, "maps": _exact_maps}[case["kind"]]
    return f(case, _inputs(case, seed))
