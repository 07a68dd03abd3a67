"""Performance cases of the fire-growth library: the calls a user's program makes, over the sizes,
directions and options in which they are made.

A case is a dict of plain values; ``prepare`` makes what a program has in hand (a context, landscapes on the
device, weather streams, parameters), ``run`` is one pass through the public entry points, and its outputs
are what the program would read: burn counts, counters, scars, ignition steps, comparison metrics, rates.
All inputs are synthetic and seeded, shaped like the repository's workloads: 100 m cells, clustered FBP fuels
with a tenth of non-fuel, fractal terrain with slopes up to 40 %, hourly weather with wind N(20, 5) km/h,
uniform random ignitions and a lognormal(0, sigma) perturbation of the rates of spread.
"""
import math

import numpy as np
import torch

import paper_1905_09317_gb300 as c2f

FUELS = (1, 2, 3, 4, 6, 7, 8, 9, 11, 13)   # C1 C2 C3 C4 C6 C7 D1 M1 O1a S1

KINDS = {
    # one deterministic fire under new weather: what an interactive program asks for
    "single": dict(rows=40, cols=40, hours=10),
    # Monte-Carlo replicas on one landscape; `weather`: "new" (a new stream comes with every pass, so the rates
    # are tabulated in the pass), "kept" (a stream that earlier runs used), "scenarios" (several new streams with
    # probabilities); `lazy`: rates tabulated where fires go
    "mc": dict(rows=512, cols=512, replicas=1000, hours=24, weather="new", scenarios=1, lazy=False, minutes=1,
               sigma=0.1, threshold=0.0, delta=0.0, ellipse=0, burn_min=0, burn_max=0, shift=0, steps=False),
    # many landscapes of uneven sizes, new weather on each, in one batched call
    "batch": dict(landscapes=24, lo=64, hi=1024, reps_lo=16, reps_hi=1024, hours=24, sizes=3),
    # requests that are all waiting, on landscapes whose rates are already tabulated
    "serve": dict(requests=48, pool=6, lo=128, hi=1024, reps_lo=32, reps_hi=2048, hours_lo=12, hours_hi=48, sizes=5),
    # hourly MSE / SSIM and final norm between two runs' scars
    "compare": dict(rows=512, cols=512, replicas=500, hours=24),
    # burn grids, ignition steps and a mid-run scar of every replica, to the host
    "export": dict(rows=300, cols=400, replicas=100, hours=12),
    # a landscape that was not seen before: loaded, given its weather, and its rates of one hour read back
    "rates": dict(rows=501, cols=700, hours=24, ellipse=0),
}


def _case(kind, name=None, **kw):
    c = {**KINDS[kind], **kw, "kind": kind}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a 40 x 40 single-fuel grid, one fire for 10 hours
        _case("single", "single_40x40"),
        # a small ragged landscape with every option of the method that changes the loops: 5-minute periods, a
        # receive threshold, burn-out by rate, the centre-offset ellipse, 6 to 12 burning hours a day
        _case("mc", "options_130x97", rows=130, cols=97, replicas=64, hours=36, minutes=5, sigma=0.2, threshold=1.0,
              delta=0.5, ellipse=1, burn_min=6, burn_max=12),
        # the standard burn-probability map: a new day's weather on a landscape that is loaded
        _case("mc", "forecast_512x512"),
        # more replicas under a stream that is tabulated already, ignition steps kept
        _case("mc", "rerun_517x389", rows=517, cols=389, replicas=300, weather="kept", steps=True),
        # weather uncertainty: eight streams with probabilities, each replica draws one
        _case("mc", "scenarios_512x512", weather="scenarios", scenarios=8),
        # the largest landscape, a wind shift half way
        _case("mc", "large_4096x4096", rows=4096, cols=4096, replicas=256, hours=36, shift=18),
        # few fires on a large landscape, with the table mode meant for them
        _case("mc", "few_fires_4096x4096", rows=4096, cols=4096, replicas=8, hours=24, lazy=True),
        # a study over a region's landscapes
        _case("batch", "batch_24"),
        # a server's backlog
        _case("serve", "serve_48"),
        # two fire models or settings against each other
        _case("compare", "compare_512x512"),
        # scars for plotting and post-processing
        _case("export", "export_300x400"),
        # a new landscape's map of rates
        _case("rates", "rates_501x700"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("single", "mc", "mc", "mc", "mc", "mc", "batch", "serve", "compare", "export", "rates"))
    if kind == "single":
        return _case(kind, rows=_log(rng, 20, 300), cols=_log(rng, 20, 300), hours=rng.randint(2, 24))
    if kind == "mc":
        rows = _log(rng, 30, 2500)
        cols = max(20, min(3000, int(rows * rng.uniform(0.6, 1.5))))
        weather = rng.choice(("new", "new", "new", "kept", "scenarios"))
        scen = rng.randint(2, 12) if weather == "scenarios" else 1
        hours = max(2, min(rng.randint(4, 36), int(2.5e8 / (rows * cols * scen))))
        lazy = rng.random() < 0.15
        over = dict(rows=rows, cols=cols, hours=hours, weather=weather, scenarios=scen, lazy=lazy,
                    replicas=_log(rng, 1, 60 if lazy else 1200), shift=hours // 2 if rng.random() < 0.3 else 0,
                    sigma=rng.choice((0.0, 0.1, 0.1, 0.3)))
        over["steps"] = rows * cols * over["replicas"] < 2e8 and rng.random() < 0.3
        if rng.random() < 0.35:
            lo = rng.randint(1, 24)
            over.update(minutes=rng.choice((1, 2, 5, 10, 15)), threshold=rng.choice((-1.0, 0.0, 1.0, 2.5)),
                        delta=rng.choice((0.0, 0.5, 1.5)), ellipse=rng.randint(0, 1), burn_min=lo,
                        burn_max=rng.randint(lo, 24))
        return _case(kind, **over)
    if kind == "batch":
        return _case(kind, landscapes=rng.randint(2, 24), lo=rng.randint(40, 100), hi=rng.randint(200, 1024),
                     reps_hi=_log(rng, 32, 1024), hours=rng.randint(6, 24), sizes=rng.randint(0, 1 << 20))
    if kind == "serve":
        return _case(kind, requests=rng.randint(2, 48), pool=rng.randint(1, 6), hi=rng.randint(200, 1024),
                     reps_hi=_log(rng, 64, 2048), sizes=rng.randint(0, 1 << 20))
    if kind == "compare":
        return _case(kind, rows=_log(rng, 50, 700), cols=_log(rng, 50, 700), replicas=_log(rng, 10, 500),
                     hours=rng.randint(2, 48))
    if kind == "export":
        return _case(kind, rows=_log(rng, 50, 500), cols=_log(rng, 50, 500), replicas=_log(rng, 1, 100),
                     hours=rng.randint(2, 24))
    return _case(kind, rows=_log(rng, 40, 1000), cols=_log(rng, 40, 1000), hours=rng.randint(1, 24),
                 ellipse=rng.randint(0, 1))


# ------------------------------------------------------------------ inputs
def _noise(rng, rows, cols, period):
    """Lattice noise of the given period, bilinearly interpolated (float64 on the GPU)."""
    ny, nx = int(math.ceil(rows / period)) + 1, int(math.ceil(cols / period)) + 1
    lat = torch.from_numpy(rng.random((ny, nx))).cuda()
    y = (torch.arange(rows, device="cuda", dtype=torch.float64) + 0.5) / period
    x = (torch.arange(cols, device="cuda", dtype=torch.float64) + 0.5) / period
    y0, x0 = y.floor().long(), x.floor().long()
    fy, fx = (y - y0)[:, None], (x - x0)[None, :]
    top = lat[y0] * (1 - fy) + lat[y0 + 1] * fy
    return top[:, x0] * (1 - fx) + top[:, x0 + 1] * fx


def _kth(v, q):
    v = v.reshape(-1)
    return torch.sort(v).values[min(v.numel() - 1, int(q * v.numel()))]


def _landscape(seed, rows, cols):
    """Fuel codes, slope (percent) and aspect (degrees) on the host: clustered fuels (the largest of ten noise
    fields), the lowest tenth of another field without fuel, six octaves of fractal elevation, Horn's slope and
    aspect scaled to a 99th percentile of 40 percent."""
    rng = np.random.default_rng(seed)
    best = _noise(rng, rows, cols, 8.0)
    fuel = torch.full((rows, cols), FUELS[0], dtype=torch.uint8, device="cuda")
    for code in FUELS[1:]:
        v = _noise(rng, rows, cols, 8.0)
        fuel[v > best] = code
        best = torch.maximum(best, v)
    v = _noise(rng, rows, cols, 8.0)
    fuel[v <= _kth(v, 0.1)] = 0
    z, amp = torch.zeros((rows, cols), dtype=torch.float64, device="cuda"), 1.0
    for octave in range(6):
        z += amp * _noise(rng, rows, cols, 256.0 / 2 ** octave)
        amp *= 0.5
    p = torch.nn.functional.pad(z[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    a, b, c = p[:-2, :-2], p[:-2, 1:-1], p[:-2, 2:]
    d, f = p[1:-1, :-2], p[1:-1, 2:]
    g, h, i = p[2:, :-2], p[2:, 1:-1], p[2:, 2:]
    dx, dy = (c + 2 * f + i) - (a + 2 * d + g), (a + 2 * b + c) - (g + 2 * h + i)
    slope = torch.hypot(dx, dy)
    slope = torch.clamp(slope * (40.0 / _kth(slope, 0.99)), max=40.0).float()
    aspect = (torch.rad2deg(torch.atan2(-dx, -dy)) % 360.0).float()
    return fuel.cpu().numpy(), slope.cpu().numpy(), aspect.cpu().numpy()


def _weather(rng, hours, mean=20.0, wd0=270.0, shift=0):
    ws = np.clip(rng.normal(mean, 5.0, hours), 0.0, None)
    step = rng.normal(0.0, 15.0, hours)
    if shift:
        step[shift] += 90.0
    wd = (wd0 + np.cumsum(step)) % 360.0
    return np.stack([ws, wd, rng.uniform(85.0, 93.0, hours), np.full(hours, rng.uniform(40.0, 120.0))], axis=1)


def _params(rng, hours, replicas, **kw):
    return c2f.default_params(seed=int(rng.integers(1 << 62)), hours=hours, n_replicas=replicas,
                              **dict(dict(ignition_mode=1, ros_sigma=0.1), **kw))


def _batch_sizes(case):
    rng = np.random.default_rng(case["sizes"])
    u = rng.random((case["landscapes"], 2))
    span = lambda x, lo, hi: int(round(lo * (hi / lo) ** x))  # noqa: E731
    return [(span(a, case["lo"], case["hi"]), span(b, case["reps_lo"], case["reps_hi"])) for a, b in u]


def _serve_sizes(case):
    rng = np.random.default_rng(case["sizes"])
    span = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))  # noqa: E731
    sides = [span(case["lo"], case["hi"]) for _ in range(case["pool"])]
    reqs = [(int(rng.integers(case["pool"])), span(case["reps_lo"], case["reps_hi"]),
             int(rng.integers(case["hours_lo"], case["hours_hi"] + 1))) for _ in range(case["requests"])]
    return sides, reqs


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([seed, 1905])
    s = dict(case=case, ctx=c2f.Context(0))
    ctx = s["ctx"]

    def land(rows, cols):
        fuel, slope, aspect = _landscape(int(rng.integers(1 << 30)), rows, cols)
        return ctx.load_landscape(fuel, slope, aspect)

    if kind == "single":
        rows, cols, hours = case["rows"], case["cols"], case["hours"]
        s["lid"] = ctx.load_landscape(np.full((rows, cols), 1, dtype=np.uint8))
        day = (rng.uniform(15.0, 25.0), rng.uniform(0.0, 360.0), rng.uniform(88.0, 92.0), rng.uniform(60.0, 100.0))
        s["weather"] = np.tile(np.array([day]), (hours, 1))
        s["params"] = _params(rng, hours, 1, ignition_mode=0, ignition_cell=(rows // 2) * cols + cols // 2,
                              ros_sigma=0.0, outputs=c2f.OUT_SCARS | c2f.OUT_COUNTERS | c2f.OUT_IGN_STEPS)
    elif kind == "mc":
        s["lid"] = land(case["rows"], case["cols"])
        hours, n = case["hours"], case["scenarios"]
        if case["weather"] == "scenarios":   # calm to strong wind from several directions, the middle ones likelier
            s["weather"] = np.stack([_weather(rng, hours, 8.0 + 28.0 * i / max(n - 1, 1), (270.0 + 20.0 * i) % 360.0,
                                              case["shift"]) for i in range(n)])
            s["prob"] = np.minimum(np.arange(1, n + 1), np.arange(n, 0, -1)).astype(np.float64)
        else:
            s["weather"] = _weather(rng, hours, shift=case["shift"])
        s["params"] = _params(rng, hours, case["replicas"], ros_sigma=case["sigma"], minutes_per_step=case["minutes"],
                              ros_threshold=case["threshold"], burnout_delta=case["delta"],
                              ellipse_mode=case["ellipse"], burn_hours_min=case["burn_min"],
                              burn_hours_max=case["burn_max"],
                              outputs=c2f.OUT_SCARS | c2f.OUT_COUNTERS | (c2f.OUT_IGN_STEPS if case["steps"] else 0))
        ctx.set_table_mode(not case["lazy"])
        if case["weather"] == "kept":
            ctx.set_weather(s["lid"], s["weather"])
            ctx.build_ros(s["lid"], s["params"], 2 if case["lazy"] else 0)
            if case["lazy"]:
                ctx.release(ctx.simulate(s["lid"], s["params"]))
    elif kind == "batch":
        sizes = _batch_sizes(case)
        s["lids"] = [land(side, side) for side, _ in sizes]
        s["cells"] = [side * side for side, _ in sizes]
        s["weather"] = [_weather(rng, case["hours"]) for _ in sizes]
        s["params"] = [_params(rng, case["hours"], reps) for _, reps in sizes]
    elif kind == "serve":
        sides, reqs = _serve_sizes(case)
        s["lids"] = [land(side, side) for side in sides]
        s["cells"] = [side * side for side in sides]
        for lid in s["lids"]:
            ctx.set_weather(lid, _weather(rng, case["hours_hi"]))
            ctx.build_ros(lid, _params(rng, case["hours_hi"], 1), 0)
        s["requests"] = [(k, _params(rng, hours, reps)) for k, reps, hours in reqs]
    elif kind in ("compare", "export"):
        lid = land(case["rows"], case["cols"])
        p = _params(rng, case["hours"], case["replicas"],
                    outputs=c2f.OUT_SCARS | c2f.OUT_COUNTERS | c2f.OUT_IGN_STEPS)
        s["sims"] = []
        for _ in range(2 if kind == "compare" else 1):   # compared: the same replicas under two weather streams
            ctx.set_weather(lid, _weather(rng, case["hours"]))
            s["sims"].append(ctx.simulate(lid, p))
        ctx.release(lid)
    else:
        s["land"] = _landscape(int(rng.integers(1 << 30)), case["rows"], case["cols"])
        s["weather"] = _weather(rng, case["hours"])
        s["params"] = _params(rng, case["hours"], 1, ellipse_mode=case["ellipse"])
        s["hour"] = case["hours"] // 2
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "single":
        n = case["rows"] * case["cols"]
        ctx.set_weather(s["lid"], s["weather"])
        sid = ctx.simulate(s["lid"], s["params"])
        scar, steps = ctx.get_replica_scar(sid, 0, n, ign_steps=True)
        out = dict(scar=scar, steps=steps, counters=ctx.get_counters(sid, 1))
        ctx.release(sid)
        return out
    if kind == "mc":
        n, reps = case["rows"] * case["cols"], case["replicas"]
        if case["weather"] == "new":
            ctx.set_weather(s["lid"], s["weather"])
        elif case["weather"] == "scenarios":
            ctx.set_weather_scenarios(s["lid"], s["weather"], s["prob"])
        sid = ctx.simulate(s["lid"], s["params"])
        out = dict(counts=ctx.burn_prob(sid, n).view(np.int32), counters=ctx.get_counters(sid, reps))
        if case["weather"] == "scenarios":
            out["scenario"] = ctx.get_scenarios(sid, reps)
        if case["steps"]:
            _, out["steps"] = ctx.get_replica_scar(sid, reps // 2, n, ign_steps=True)
        ctx.release(sid)
        return out
    if kind == "batch":
        for lid, w in zip(s["lids"], s["weather"]):
            ctx.set_weather(lid, w)
        sids = ctx.simulate_batch(s["lids"], s["params"])
        out = dict(counts=[ctx.burn_prob(sid, n).view(np.int32) for sid, n in zip(sids, s["cells"])],
                   work=[ctx.get_counters(sid, p.n_replicas)[0] for sid, p in zip(sids, s["params"])])
        for sid in sids:
            ctx.release(sid)
        return out
    if kind == "serve":
        sids = [ctx.submit(s["lids"][k], p) for k, p in s["requests"]]
        counts, work = [], []
        for sid, (k, p) in zip(sids, s["requests"]):
            ctx.wait(sid)
            counts.append(ctx.burn_prob(sid, s["cells"][k]).view(np.int32))
            work.append(ctx.get_counters(sid, p.n_replicas)[0])
            ctx.release(sid)
        return dict(counts=counts, work=np.concatenate(work))
    if kind == "compare":
        mse, ssim, norm = ctx.compare_scars(s["sims"][0], s["sims"][1], case["replicas"], case["hours"])
        return dict(mse=mse, ssim=ssim, norm=norm)
    if kind == "export":
        n, reps = case["rows"] * case["cols"], case["replicas"]
        scars, steps = ctx.get_scars(s["sims"][0], reps, n, ign_steps=True)
        return dict(scars=scars, steps=steps,
                    midway=ctx.get_scars_at_hour(s["sims"][0], case["hours"] // 2, reps, n))
    lid = ctx.load_landscape(*s["land"])
    ctx.set_weather(lid, s["weather"])
    ros8, hros, base = ctx.get_ros(lid, s["params"], s["hour"], s["land"][0].size)
    ctx.release(lid)
    return dict(ros8=ros8, hros=hros, base=base)


# ------------------------------------------------------------------ what a pass cannot do without
FLOPS_PER_RATE = 300   # binary64 operations of one cell and hour: FBP rates, ellipse, eight axes


def work(case):
    kind = case["kind"]
    if kind in ("single", "mc"):
        n, reps = case["rows"] * case["cols"], case.get("replicas", 1)
        new = case.get("weather", "new") != "kept"
        rates = case.get("scenarios", 1) * case["hours"] * n
        if case.get("lazy"):   # only the cells that fires reach need rates: here up to a few thousand a fire
            rates = min(rates, reps * case["hours"] * 4000)
        out = 4 * n + 16 * reps + (4 * n if case.get("steps") else 0) + (5 * n if kind == "single" else 0)
        return dict(bytes=9 * n + 32 * case["hours"] * case.get("scenarios", 1) + out,
                    flops=FLOPS_PER_RATE * rates if new else 0)
    if kind == "batch":
        n = sum(side * side for side, _ in _batch_sizes(case))
        return dict(bytes=13 * n + 16 * sum(r for _, r in _batch_sizes(case)), flops=FLOPS_PER_RATE * n * case["hours"])
    if kind == "serve":
        sides, reqs = _serve_sizes(case)
        return dict(bytes=sum(9 * x * x for x in sides) + sum(4 * sides[k] ** 2 + 16 * r for k, r, _ in reqs), flops=0)
    n, hours = case["rows"] * case["cols"], case["hours"]
    if kind == "compare":
        return dict(bytes=case["replicas"] * (8 * n + 16 * hours + 8), flops=0)
    if kind == "export":   # a bit and a step per cell and replica in, two bytes and a step out
        return dict(bytes=case["replicas"] * n * (4.125 + 6), flops=0)
    return dict(bytes=9 * n + 136 * n, flops=FLOPS_PER_RATE * n)


# ------------------------------------------------------------------ what the rates are in 64 bits
COEF = {1: (90.0, 0.0649, 4.5, 0.90, 72.0), 2: (110.0, 0.0282, 1.5, 0.70, 64.0), 3: (110.0, 0.0444, 3.0, 0.75, 62.0),
        4: (110.0, 0.0293, 1.5, 0.80, 66.0), 6: (30.0, 0.0800, 3.0, 0.80, 62.0), 7: (45.0, 0.0305, 2.0, 0.85, 106.0),
        8: (30.0, 0.0232, 1.6, 0.90, 32.0), 9: (None, None, None, 0.80, 50.0), 11: (190.0, 0.0310, 1.4, 1.0, 1.0),
        13: (75.0, 0.0297, 1.3, 0.75, 38.0)}


def _exact_rates(fuel, slope, aspect, weather, ellipse):
    """The eight axis rates and the head rate (m/min) of every cell in one hour, the FBP surface-spread equations
    and the ellipse written the plain way (curing 60 %, M1 half conifer)."""
    ws, wd, ffmc, bui = (float(v) for v in weather)
    m = 147.2 * (101.0 - ffmc) / (59.5 + ffmc)
    isz = 0.208 * 91.9 * math.exp(-0.1386 * m) * (1.0 + m ** 5.31 / 4.93e7)
    cure = 0.176 + 0.02 * (60.0 - 58.8)
    ros8, hros_all = np.zeros((fuel.size, 8)), np.zeros(fuel.size)
    fuel, slope, aspect = fuel.ravel(), slope.ravel().astype(np.float64), aspect.ravel().astype(np.float64)

    def curve(code, isi):
        a, b, c = COEF[code][:3]
        return a * (1.0 - np.exp(-b * isi)) ** c

    def rsi(code, isi):
        if code == 9:
            return 0.5 * curve(2, isi) + 0.5 * curve(8, isi)
        return curve(code, isi) * (cure if code == 11 else 1.0)

    def isf_of(code, mult, sf):
        a, b, c = COEF[code][:3]
        return np.log(np.maximum(1.0 - (curve(code, isz) * sf / a) ** (1.0 / c), 0.01)) / -b

    for code in np.unique(fuel):
        if code == 0:
            continue
        at = np.nonzero(fuel == code)[0]
        gs = slope[at]
        sf = np.exp(3.533 * (np.minimum(gs, 60.0) / 100.0) ** 1.2)
        isf = 0.5 * isf_of(2, 1.0, sf) + 0.5 * isf_of(8, 1.0, sf) if code == 9 else isf_of(code, 1.0, sf)
        ff = isz / 0.208
        wse = np.log(isf / isz) / 0.05039
        high = np.where(isf < 0.999 * 2.496 * ff,
                        28.0 - np.log(np.maximum(1.0 - isf / (2.496 * ff), 1e-300)) / 0.0818, 112.45)
        wse = np.where(gs > 0, np.where(wse > 40.0, high, wse), 0.0)
        up, to = np.radians(aspect[at] + 180.0), math.radians(wd + 180.0)
        wx, wy = ws * math.sin(to) + wse * np.sin(up), ws * math.cos(to) + wse * np.cos(up)
        wsv = np.sqrt(wx * wx + wy * wy)
        calm = wsv == 0
        ux, uy = np.where(calm, 1.0, wx / np.where(calm, 1.0, wsv)), np.where(calm, 0.0, wy / np.where(calm, 1.0, wsv))
        fw = np.where(wsv <= 40.0, np.exp(0.05039 * wsv), 12.0 * (1.0 - np.exp(-0.0818 * (wsv - 28.0))))
        q, bui0 = COEF[code][3:]
        be = 1.0 if code == 11 else math.exp(50.0 * math.log(q) * (1.0 / bui - 1.0 / bui0))
        hros, bros = rsi(code, isz * fw) * be, rsi(code, isz * np.exp(-0.05039 * wsv)) * be
        if code == 11:
            lb = np.where(wsv >= 1.0, 1.1 * np.maximum(wsv, 1.0) ** 0.464, 1.0)
        else:
            lb = 1.0 + 8.729 * (1.0 - np.exp(-0.030 * wsv)) ** 2.155
        a, b, c = (hros + bros) / 2.0, (hros + bros) / (2.0 * lb), (hros - bros) / 2.0
        e = np.sqrt(1.0 - 1.0 / (lb * lb))
        hros_all[at] = hros
        r2 = math.sqrt(0.5)
        for k, (x, y) in enumerate(((1, 0), (r2, r2), (0, 1), (-r2, r2), (-1, 0), (-r2, -r2), (0, -1), (r2, -r2))):
            cos = x * ux + y * uy
            if ellipse == 0:
                ros8[at, k] = np.where(cos > 0, a * (1.0 - e * e) / (1.0 - e * np.maximum(cos, 0.0)), a * (1.0 - e * e))
            else:
                sin2 = np.maximum(1.0 - cos * cos, 0.0)
                root = np.sqrt(b * b * cos * cos + hros * bros * sin2)
                ros8[at, k] = np.where(cos >= 0, (b * b * c * cos + a * b * root) / (b * b * cos * cos + a * a * sin2),
                                       b * b * hros * bros / (a * b * root - b * b * c * cos))
    return ros8, hros_all


def exact(case, seed):
    if case["kind"] != "rates":
        # counts, steps, scars and counters are whole numbers; the comparison's metrics are functions of scars
        # that only a whole run of the method gives
        return None
    rng = np.random.default_rng([seed, 1905])
    land = _landscape(int(rng.integers(1 << 30)), case["rows"], case["cols"])
    ros8, hros = _exact_rates(*land, _weather(rng, case["hours"])[case["hours"] // 2], case["ellipse"])
    return dict(ros8=ros8, hros=hros, base=None)
