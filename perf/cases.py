"""What the library's speed is measured on: calls that a program using it makes, over the range of sizes it is
used at.  Lens fields are seeded random discs (unit masses or Salpeter masses in [0.1, 1], a disc covering the shooting
region 1.5 times), the geometry of the paper's experiments; grids, maps and lens counts are those of the repository's
workloads and tests, or lie between them.

Kinds of case (a case's "kind"):
  map     one magnification map: zero the counts, shoot the grid (or its rows [row0, row1)), normalise
  frames  a moving field stepped through a few times, one map per step (a time series)
  staged  a map's row block through a field held as several lens partitions
  batch   a planned batch of independent fields, one launch
  zoom    a culled re-shoot of a part of a map at higher resolution
  trace   source positions of listed rays (float32 with deflections and error bands, or certified)
  curves  light curves of source tracks across maps (a plan launched again, or a single call)
"""
import math

import numpy as np
import torch

import paper_0905_2453_gb300 as rs

SLOPE, M_LO, M_HI = 2.35, 0.1, 1.0


# ---------------------------------------------------------------------------------------------- cases

def listed():
    return [
        # a quick look at a small field: launches and latency are all of it
        {"name": "map-300-quick", "kind": "map", "n": 300, "salpeter": True, "kstar": 0.5, "kc": 0.1, "gamma": 0.3,
         "n0": 384, "n1": 384, "row0": 0, "row1": 384, "np0": 64, "np1": 64},
        # the smallest workload (100 lenses, 1000^2 rays, 256^2 map) as a time series of moving lenses
        {"name": "frames-100", "kind": "frames", "n": 100, "salpeter": False, "kstar": 0.69, "kc": 0.0, "gamma": 0.0,
         "n0": 1000, "n1": 1000, "np0": 256, "np1": 256, "frames": 4},
        # the ordinary map: 1e4 equal masses, 4096^2 rays, 1024^2 pixels
        {"name": "map-1e4", "kind": "map", "n": 10000, "salpeter": False, "kstar": 0.45, "kc": 0.0, "gamma": 0.4,
         "n0": 4096, "n1": 4096, "row0": 0, "row1": 4096, "np0": 1024, "np1": 1024},
        # a field with a mass spectrum on a grid that fits no tile
        {"name": "map-30011-ragged", "kind": "map", "n": 30011, "salpeter": True, "kstar": 0.6, "kc": 0.1,
         "gamma": 0.3, "n0": 1777, "n1": 1301, "row0": 0, "row1": 1301, "np0": 501, "np1": 640},
        # 1e6 Salpeter lenses resident as four partitions, a block of rows of the 16384^2 grid
        {"name": "staged-1e6", "kind": "staged", "n": 1000000, "salpeter": True, "kstar": 0.6, "kc": 0.1, "gamma": 0.3,
         "n0": 16384, "n1": 16384, "row0": 8160, "row1": 8224, "np0": 2048, "np1": 2048, "parts": 4},
        # the largest fields are shot in blocks of a few rows (checkpoints): 1e7 equal masses, 32 rows of 8192^2
        {"name": "rows-1e7", "kind": "map", "n": 10000000, "salpeter": False, "kstar": 0.5, "kc": 0.0, "gamma": 0.5,
         "n0": 8192, "n1": 8192, "row0": 4080, "row1": 4112, "np0": 4096, "np1": 4096},
        # many small maps in one launch
        {"name": "batch-60x100", "kind": "batch", "fields": 60, "n_lo": 100, "n_hi": 100, "side_lo": 1000,
         "side_hi": 1000, "np_lo": 256, "np_hi": 256, "salpeter": False},
        # realisations of uneven size with a mass spectrum in one launch
        {"name": "batch-16-uneven", "kind": "batch", "fields": 16, "n_lo": 100, "n_hi": 30000, "side_lo": 1024,
         "side_hi": 2048, "np_lo": 512, "np_hi": 1024, "salpeter": True},
        # the central quarter of the ordinary map at four times the resolution
        {"name": "zoom-1e4-x4", "kind": "zoom", "n": 10000, "salpeter": False, "kstar": 0.45, "kc": 0.0, "gamma": 0.4,
         "n0": 4096, "n1": 4096, "np0": 1024, "np1": 1024, "factor": 4, "part": 0.25},
        # source positions, deflections and error bands of a list of rays through a large field
        {"name": "trace-4096-1e5", "kind": "trace", "n": 100000, "salpeter": True, "kstar": 0.6, "kc": 0.1,
         "gamma": 0.3, "n0": 8192, "n1": 8192, "rays": 4096, "certified": False},
        # light curves of a small Gaussian source over many maps, the plan launched again for each set of maps
        {"name": "curves-gauss-plan", "kind": "curves", "maps": 64, "np_lo": 512, "np_hi": 1024, "tracks": 16,
         "samples": 2048, "gauss": True, "s_px": 2.0, "step_px": 0.25, "plan": True},
        # light curves of a resolved disc over a few maps, one call
        {"name": "curves-disc-call", "kind": "curves", "maps": 5, "np_lo": 700, "np_hi": 1100, "tracks": 7,
         "samples": 1501, "gauss": False, "s_px": 17.3, "step_px": 0.8, "plan": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _middle(rng, n, rows):
    """First row of a block about the middle of a grid of n rows (the part that the window sees)."""
    return min(max(0, (n - rows) // 2 + rng.randint(-n // 20, n // 20)), n - rows)


def draw(rng):
    kind = rng.choice(["map", "map", "map", "frames", "staged", "batch", "zoom", "trace", "curves"])
    macro = {"kstar": round(rng.uniform(0.2, 0.7), 3), "kc": rng.choice([0.0, 0.1]),
             "gamma": round(rng.uniform(0.0, 0.5), 3)}
    salpeter = rng.random() < 0.5
    if kind == "map":
        n = _log(rng, 100, 4000000)
        n0, n1 = _log(rng, 200, 8192), _log(rng, 200, 8192)
        rows = max(1, min(n1, int(2.0e11 / (float(n) * n0)), _log(rng, 100, 4096)))
        row0 = _middle(rng, n1, rows)
        return {"kind": kind, "n": n, "salpeter": salpeter, **macro, "n0": n0, "n1": n1, "row0": row0,
                "row1": row0 + rows, "np0": _log(rng, 64, 2048), "np1": _log(rng, 64, 2048)}
    if kind == "frames":
        return {"kind": kind, "n": _log(rng, 50, 3000), "salpeter": salpeter, **macro, "n0": _log(rng, 200, 1500),
                "n1": _log(rng, 200, 1500), "np0": _log(rng, 64, 512), "np1": _log(rng, 64, 512),
                "frames": rng.randrange(1, 7)}
    if kind == "staged":
        n0 = _log(rng, 300, 16384)
        n = _log(rng, 3000, 1000000)
        # blocks of whole groups of 64 rows, as row blocks under a state budget are cut
        rows = max(1, min(n0, int(2.0e11 / (float(n) * n0)), 1000) // 64) * 64
        row0 = _middle(rng, n0, rows)
        return {"kind": kind, "n": n, "salpeter": salpeter, **macro, "n0": n0, "n1": n0, "row0": row0,
                "row1": row0 + rows, "np0": _log(rng, 128, 2048), "np1": _log(rng, 128, 2048),
                "parts": rng.randrange(2, 7)}
    if kind == "batch":
        lo = _log(rng, 50, 2000)
        side = _log(rng, 200, 1500)
        return {"kind": kind, "fields": rng.randrange(2, 49), "n_lo": lo, "n_hi": lo * rng.choice([1, 3, 8]),
                "side_lo": side, "side_hi": min(2000, side * rng.choice([1, 2])), "np_lo": 100, "np_hi": 700,
                "salpeter": salpeter}
    if kind == "zoom":
        n0 = _log(rng, 500, 3000)
        return {"kind": kind, "n": _log(rng, 100, 10000), "salpeter": salpeter, **macro, "n0": n0, "n1": n0,
                "np0": _log(rng, 128, 1024), "np1": _log(rng, 128, 1024), "factor": rng.randrange(1, 5),
                "part": round(rng.uniform(0.1, 0.9), 2)}
    if kind == "trace":
        n = _log(rng, 100, 1000000)
        return {"kind": kind, "n": n, "salpeter": salpeter, **macro, "n0": 8192, "n1": 8192,
                "rays": max(1, min(_log(rng, 1, 200000), int(2.0e9 / n))), "certified": rng.random() < 0.5}
    lo = _log(rng, 200, 1000)
    gauss = rng.random() < 0.5
    return {"kind": kind, "maps": rng.randrange(1, 33), "np_lo": lo, "np_hi": lo + rng.randrange(0, 400),
            "tracks": rng.randrange(1, 17), "samples": _log(rng, 100, 2048), "gauss": gauss,
            "s_px": round(rng.uniform(0.4, 4.0) if gauss else rng.uniform(0.7, 24.0), 2),
            "step_px": round(rng.uniform(0.1, 1.5), 2), "plan": rng.random() < 0.5}


# ---------------------------------------------------------------------------------------------- inputs

def _mean_mass(salpeter):
    if not salpeter:
        return 1.0
    a, b = 1.0 - SLOPE, 2.0 - SLOPE
    return ((M_HI ** b - M_LO ** b) / b) / ((M_HI ** a - M_LO ** a) / a)


def _geometry(n, kstar, salpeter):
    """Disc radius, half side of the shooting region, half side of the source window."""
    radius = math.sqrt(n * _mean_mass(salpeter) / kstar)
    half = radius / (1.5 * math.sqrt(2.0))
    return radius, half, half / 5.0


def _lenses(n, radius, salpeter, gen):
    """float32 positions [n, 2] and masses [n] (None: all 1) on the GPU."""
    u = torch.rand(3, n, dtype=torch.float64, device="cuda", generator=gen)
    r, th = radius * u[0].sqrt(), 2.0 * math.pi * u[1]
    xy = torch.stack([r * th.cos(), r * th.sin()], 1).float().contiguous()
    if not salpeter:
        return xy, None
    a = 1.0 - SLOPE
    lo, hi = M_LO ** a, M_HI ** a
    return xy, ((lo + u[2] * (hi - lo)) ** (1.0 / a)).float()


def _grid(half, n0, n1):
    d = (2.0 * half / n0, 2.0 * half / n1)
    return rs.RayGrid((-half + 0.5 * d[0], -half + 0.5 * d[1]), d, (n0, n1))


def _window(s, np0, np1):
    return rs.Window((-s, -s), (s, s), (np0, np1))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _field_inputs(case, seed):
    radius, half, s = _geometry(case["n"], case["kstar"], case["salpeter"])
    gen = _gen(seed)
    xy, m = _lenses(case["n"], radius, case["salpeter"], gen)
    return gen, xy, m, half, s


def _velocities(case, gen):
    return 0.3 * torch.randn(case["n"], 2, device="cuda", generator=gen)


def _times(case):
    return [0.5 * k for k in range(case["frames"])]


def _zoom_box(case, s):
    q = s * case["part"]
    return (-q, -q), (q, q)


def _rays(case, gen):
    i = torch.randint(0, case["n0"], (case["rays"],), device="cuda", generator=gen)
    j = torch.randint(0, case["n1"], (case["rays"],), device="cuda", generator=gen)
    return torch.stack([i, j], 1).contiguous()


def _batch_inputs(case, seed):
    rng = np.random.default_rng([int(seed), 5])
    gen = _gen(seed)
    out = []
    for k in range(case["fields"]):
        # sizes belong to the case, not to the seed: every seed's batch is the same work
        size = np.random.default_rng([k, 11])
        n = int(round(math.exp(size.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        side = int(size.integers(case["side_lo"], case["side_hi"] + 1))
        npix = int(size.integers(case["np_lo"], case["np_hi"] + 1))
        kstar, gamma = float(rng.uniform(0.1, 0.8)), float(rng.uniform(0.0, 0.6))
        radius, half, s = _geometry(n, kstar, case["salpeter"])
        xy, m = _lenses(n, radius, case["salpeter"], gen)
        out.append((xy, m, gamma, _grid(half, side, side), _window(s, npix, npix)))
    return out


def _curve_inputs(case, seed):
    """Maps with the structure of magnification maps (a lognormal background and fold caustics outside of which mu
    rises as 1 / sqrt(distance)), their windows, the tracks and the source size."""
    gen = _gen(seed)
    rng = np.random.default_rng([int(seed), 3])
    maps, wins, tracks = [], [], []
    px = 2.0 / case["np_hi"]
    for k in range(case["maps"]):
        npix = int(np.random.default_rng([k, 13]).integers(case["np_lo"], case["np_hi"] + 1))
        mu = torch.exp(0.25 * torch.randn(npix, npix, device="cuda", generator=gen))
        ax = torch.arange(npix, device="cuda", dtype=torch.float32)
        for _ in range(6):
            cx, cy = rng.uniform(0, npix, 2)
            r = rng.uniform(0.05, 0.4) * npix
            d = torch.hypot(ax[None, :] - cx, ax[:, None] - cy) - r
            mu += torch.where((d > 0) & (d < 15), rng.uniform(1.0, 4.0) * torch.rsqrt(d.clamp(min=1e-3)), 0.0)
        maps.append(mu.clamp_(max=500.0).contiguous())
        wins.append(rs.Window((-1.0, -1.0), (1.0, 1.0), (npix, npix)))
        for _ in range(case["tracks"]):
            y0 = rng.uniform(-0.9, 0.9, 2)
            th = rng.uniform(0.0, 2.0 * math.pi)
            step = case["step_px"] * px
            tracks.append(rs.Track(k, (float(y0[0]), float(y0[1])), (step * math.cos(th), step * math.sin(th)),
                                   case["samples"]))
    return maps, wins, tracks, case["s_px"] * px


def _counts(window):
    return torch.zeros((window.npix[1], window.npix[0]), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "oow": torch.zeros(1, dtype=torch.int64, device="cuda")}
    if kind == "batch":
        inp = _batch_inputs(case, seed)
        st["fields"] = [rs.Field(xy, m, 0.0, gamma) for xy, m, gamma, _, _ in inp]
        st["batch"] = rs.Batch(st["fields"], [i[3] for i in inp], [i[4] for i in inp])
        return st
    if kind == "curves":
        st["maps"], st["wins"], st["tracks"], st["s"] = _curve_inputs(case, seed)
        st["profile"] = rs.RS_PROFILE_GAUSSIAN if case["gauss"] else rs.RS_PROFILE_DISC
        if case["plan"]:
            st["plan"] = rs.LightCurvePlan(st["maps"], st["wins"], st["tracks"], st["profile"], st["s"])
        return st
    gen, xy, m, half, s = _field_inputs(case, seed)
    st["grid"] = _grid(half, case["n0"], case["n1"])
    if kind == "trace":
        st["field"] = rs.Field(xy, m, case["kc"], case["gamma"])
        st["rays"] = _rays(case, gen)
        return st
    st["window"] = _window(s, case["np0"], case["np1"])
    if kind == "frames":
        st["field"] = rs.Field(xy, m, case["kc"], case["gamma"], velocities=_velocities(case, gen))
        st["counts"] = [_counts(st["window"]) for _ in range(case["frames"])]
    elif kind == "staged":
        n = case["n"]
        size = -(-n // case["parts"]) // 256 * 256 + 256
        st["fields"] = [rs.Field(xy[a:a + size], None if m is None else m[a:a + size], case["kc"], case["gamma"])
                        for a in range(0, n, size)]
        st["counts"] = _counts(st["window"])
    else:
        st["field"] = rs.Field(xy, m, case["kc"], case["gamma"])
        if kind == "map":
            st["counts"] = _counts(st["window"])
        else:
            st["lo"], st["hi"] = _zoom_box(case, s)
    return st


# ---------------------------------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].launch()
        return {"counts": state["batch"].counts, "oow": state["batch"].out_of_window}
    if kind == "curves":
        if case["plan"]:
            state["plan"].launch()
            return {"mu": state["plan"].mu, "dm": state["plan"].dm}
        mu, dm = rs.light_curves(state["maps"], state["wins"], state["tracks"], state["profile"], state["s"])
        return {"mu": mu, "dm": dm}
    grid = state["grid"]
    if kind == "trace":
        if case["certified"]:
            y, alpha = state["field"].trace(grid, state["rays"], with_alpha=True, certified=True)
            return {"y": y, "alpha": alpha}
        y, alpha, err = state["field"].trace(grid, state["rays"], with_alpha=True, with_err=True)
        return {"y": y, "alpha": alpha, "err": err}
    window, oow = state.get("window"), state["oow"]
    if kind == "zoom":
        counts, g, w = state["field"].zoom(grid, window, state["lo"], state["hi"], case["factor"])
        return {"counts": counts, "mu": rs.magnification(counts, g, w)}
    oow.zero_()
    if kind == "frames":
        mu = []
        for t, counts in zip(_times(case), state["counts"]):
            state["field"].set_time(t)
            counts.zero_()
            state["field"].shoot(grid, window, counts, oow)
            mu.append(rs.magnification(counts, grid, window))
        return {"counts": state["counts"], "oow": oow, "mu": mu}
    counts = state["counts"].zero_()
    if kind == "staged":
        rs.rs_shoot_staged([f.handle for f in state["fields"]], grid, case["row0"], case["row1"], window, counts, oow)
    elif case["row0"] == 0 and case["row1"] == case["n1"]:
        state["field"].shoot(grid, window, counts, oow)
    else:
        state["field"].shoot(grid, window, counts, oow, rows=(case["row0"], case["row1"]))
    return {"counts": counts, "oow": oow, "mu": rs.magnification(counts, grid, window)}


# ---------------------------------------------------------------------------------------------- work

def _batch_sizes(case):
    for k in range(case["fields"]):
        size = np.random.default_rng([k, 11])
        n = int(round(math.exp(size.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        yield n, int(size.integers(case["side_lo"], case["side_hi"] + 1)), int(size.integers(case["np_lo"],
                                                                                             case["np_hi"] + 1))


def work(case):
    """Ten flops per lens-ray pair (the paper's count, a division as one); lenses read once (8 bytes, 12 with a
    mass), counts written and read once and mu written once (12 bytes a pixel)."""
    kind = case["kind"]
    if kind == "batch":
        lens = 12 if case["salpeter"] else 8
        return {"bytes": sum(lens * n + 4.0 * p * p for n, _, p in _batch_sizes(case)),
                "flops": sum(10.0 * n * side * side for n, side, _ in _batch_sizes(case))}
    if kind == "curves":
        # a multiply-add and the weight's exponent per covered pixel; the maps read once, two doubles a sample
        samples = case["maps"] * case["tracks"] * case["samples"]
        side = 0.5 * (case["np_lo"] + case["np_hi"])
        radius = case["s_px"] * (6.0 if case["gauss"] else 1.0) * side / case["np_hi"]
        return {"bytes": 16.0 * samples + 4.0 * case["maps"] * side * side,
                "flops": samples * math.pi * radius * radius * (4.0 if case["gauss"] else 1.0)}
    lenses = (12.0 if case["salpeter"] else 8.0) * case["n"]
    if kind == "trace":
        return {"bytes": lenses + case["rays"] * (48.0 if case["certified"] else 64.0),
                "flops": 10.0 * case["n"] * case["rays"]}
    pixels = float(case["np0"] * case["np1"])
    if kind == "frames":
        return {"bytes": case["frames"] * (2 * lenses + 12.0 * pixels),
                "flops": 10.0 * case["frames"] * case["n"] * case["n0"] * case["n1"]}
    if kind == "zoom":
        # the rays that land in the region: its area times the mean magnification, at the finer density
        lam = [abs(1.0 - case["kstar"] - case["kc"] + g) for g in (-case["gamma"], case["gamma"])]
        share = min(1.0, case["part"] / 5.0 / max(lam[0], 0.1)) * min(1.0, case["part"] / 5.0 / max(lam[1], 0.1))
        rays = share * case["n0"] * case["n1"] * case["factor"] ** 2
        fine = pixels * (case["part"] * case["factor"]) ** 2
        return {"bytes": lenses + 12.0 * fine, "flops": 10.0 * case["n"] * rays}
    return {"bytes": lenses + 12.0 * pixels, "flops": 10.0 * case["n"] * case["n0"] * (case["row1"] - case["row0"])}


def tolerance(case):
    # Counts are those of the float64 definition (rays too close to a pixel edge for float32 are decided in
    # float-float), and mu is a count times one float32 factor: whole numbers stay the same.
    if case["kind"] == "trace":
        # float32 sums of 64 lenses folded into pairs of floats, 2e-8 from exact() here (more through few lenses); the
        # certified path keeps 2^-44 of each term
        return {"rel": 1e-12, "max": 1e-10} if case["certified"] else {"rel": 4e-7, "max": 4e-5}
    # curves: float32 row sums and weights, 3e-7 from exact()
    return {"rel": 1.5e-6, "max": 2e-5} if case["kind"] == "curves" else {"rel": 2e-7, "max": 1e-6}


# ---------------------------------------------------------------------------------------------- 64 bits

def _coords(grid, k):
    """Ray coordinates along axis k: the float64 position rounded to float32 is the ray's position."""
    i = torch.arange(grid.n[k], dtype=torch.float64, device="cuda")
    return (i * grid.spacing[k] + grid.origin[k]).float().double()


def _alpha(x1, x2, xy, m):
    """Deflection of rays (x1, x2) (float64 vectors) by all lenses, in float64."""
    a1, a2 = torch.zeros_like(x1), torch.zeros_like(x2)
    lens = xy.double()
    step = max(1, (1 << 25) // max(1, x1.numel()))
    for b in range(0, lens.shape[0], step):
        d1 = x1[:, None] - lens[None, b:b + step, 0]
        d2 = x2[:, None] - lens[None, b:b + step, 1]
        w = (d1 * d1 + d2 * d2).reciprocal_()
        if m is not None:
            w *= m[None, b:b + step].double()
        a1 += (w * d1).sum(1)
        a2 += (w * d2).sum(1)
    return a1, a2


def _map(xy, m, kc, gamma, grid, window, rows):
    """Counts, out-of-window count and mu of grid rows [rows) in float64."""
    x1, x2 = _coords(grid, 0), _coords(grid, 1)[rows[0]:rows[1]]
    n0 = x1.numel()
    npx = window.npix[0] * window.npix[1]
    counts = torch.zeros(npx, dtype=torch.int64, device="cuda")
    per = max(1, (1 << 18) // n0)
    for r in range(0, x2.numel(), per):
        b2 = x2[r:r + per].repeat_interleave(n0)
        b1 = x1.repeat(min(per, x2.numel() - r))
        a1, a2 = _alpha(b1, b2, xy, m)
        u = [((1.0 - kc) - gamma) * b1 - a1, ((1.0 - kc) + gamma) * b2 - a2]
        u = [(u[k] - window.lo[k]) * (window.npix[k] / (window.hi[k] - window.lo[k])) for k in (0, 1)]
        ok = (u[0] >= 0) & (u[0] < window.npix[0]) & (u[1] >= 0) & (u[1] < window.npix[1])
        pix = u[1][ok].floor().long() * window.npix[0] + u[0][ok].floor().long()
        counts += torch.bincount(pix, minlength=npx)
    nav = 1.0
    for k in (0, 1):
        nav *= (window.hi[k] - window.lo[k]) / window.npix[k] / grid.spacing[k]
    counts = counts.reshape(window.npix[1], window.npix[0])
    return counts.int(), n0 * x2.numel() - int(counts.sum()), counts.double() / nav


def _exact_curves(case, seed):
    maps, wins, tracks, s = _curve_inputs(case, seed)
    cut2 = (6.0 * s) * (6.0 * s) if case["gauss"] else s * s
    reach = 6.0 * s if case["gauss"] else s
    out = []
    for k, (mu, w) in enumerate(zip(maps, wins)):
        own = [t for t in tracks if t.map == k]
        ks = torch.arange(case["samples"], dtype=torch.float64, device="cuda")
        y = [torch.cat([t.y0[a] + ks * t.step[a] for t in own]) for a in (0, 1)]
        pix = [(w.hi[a] - w.lo[a]) / w.npix[a] for a in (0, 1)]
        c0 = [((y[a] - w.lo[a]) / pix[a]).floor().long() for a in (0, 1)]
        r = int(reach / min(pix)) + 2
        num, den, flat = torch.zeros_like(y[0]), torch.zeros_like(y[0]), mu.double().reshape(-1)
        for j in range(-r, r + 1):
            jj = c0[1] + j
            dy2 = (w.lo[1] + (jj.double() + 0.5) * pix[1] - y[1]) ** 2
            for i in range(-r, r + 1):
                ii = c0[0] + i
                d2 = (w.lo[0] + (ii.double() + 0.5) * pix[0] - y[0]) ** 2 + dy2
                ok = (d2 <= cut2) & (ii >= 0) & (ii < w.npix[0]) & (jj >= 0) & (jj < w.npix[1])
                wt = ok * (torch.exp(-d2 / (2.0 * s * s)) if case["gauss"] else 1.0)
                den += wt
                num += wt * flat[(jj * w.npix[0] + ii).clamp(0, flat.numel() - 1)]
        out.append(num / den)
    mu = torch.cat(out)
    return {"mu": mu, "dm": -2.5 * torch.log10(mu)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "curves":
        side = 2.0 * case["s_px"] * (6.0 if case["gauss"] else 1.0) + 5.0
        if case["maps"] * side * side * (200.0 + case["tracks"] * case["samples"] / 100.0) > 3e7:
            return None
        return _exact_curves(case, seed)
    if work(case)["flops"] > 2e11:
        return None
    if kind == "batch":
        parts = [_map(xy, m, 0.0, gamma, g, w, (0, g.n[1])) for xy, m, gamma, g, w in _batch_inputs(case, seed)]
        return {"counts": [p[0] for p in parts], "oow": torch.tensor([p[1] for p in parts])}
    gen, xy, m, half, s = _field_inputs(case, seed)
    grid = _grid(half, case["n0"], case["n1"])
    if kind == "trace":
        ij = _rays(case, gen)
        x1, x2 = _coords(grid, 0)[ij[:, 0]], _coords(grid, 1)[ij[:, 1]]
        a1, a2 = _alpha(x1, x2, xy, m)
        y = torch.stack([((1.0 - case["kc"]) - case["gamma"]) * x1 - a1,
                         ((1.0 - case["kc"]) + case["gamma"]) * x2 - a2], 1)
        return {"y": y, "alpha": torch.stack([a1, a2], 1)}
    window = _window(s, case["np0"], case["np1"])
    if kind == "zoom":
        if float(case["n"]) * case["n0"] * case["n1"] * case["factor"] ** 2 > 2e10:
            return None
        lo, hi = _zoom_box(case, s)
        f = case["factor"]
        sp = [v / f for v in grid.spacing]
        fine = rs.RayGrid(tuple(grid.origin[k] - 0.5 * grid.spacing[k] + 0.5 * sp[k] for k in (0, 1)), tuple(sp),
                          (case["n0"] * f, case["n1"] * f))
        npix = [max(1, int(round((hi[k] - lo[k]) / ((window.hi[k] - window.lo[k]) / window.npix[k] / f))))
                for k in (0, 1)]
        counts, _, mu = _map(xy, m, case["kc"], case["gamma"], fine, rs.Window(lo, hi, tuple(npix)), (0, fine.n[1]))
        return {"counts": counts, "mu": mu}
    if kind == "frames":
        vel = _velocities(case, gen)
        maps = [_map((xy.double() + vel.double() * t).float(), m, case["kc"], case["gamma"], grid, window,
                     (0, case["n1"])) for t in _times(case)]
        return {"counts": [c for c, _, _ in maps], "oow": torch.tensor([sum(o for _, o, _ in maps)]),
                "mu": [v for _, _, v in maps]}
    counts, oow, mu = _map(xy, m, case["kc"], case["gamma"], grid, window, (case["row0"], case["row1"]))
    return {"counts": counts, "oow": torch.tensor([oow]), "mu": mu}
