"""Frontier windows and the integer rate arithmetic at their edges, against the oracle (needs a GB300).

A frontier warp handles at most 32 entries, 32 crossings and 32 burn-outs at a
time and shortens its window when there are more, so fires are run whose
fronts cross all at once (equal rates, no perturbation) or one period apart,
on grids inside, across and beyond the plane window and at the grid's borders.
The rates are checked bit for bit where the integer division, root and
fixed-point conversion leave their usual range.
"""
import numpy as np
import pytest

import c2f_synth as S
import oracle
import paper_1905_09317_gb300 as c2f

pytestmark = pytest.mark.gpu

_KEYS = {f[0] for f in c2f.SimParams._fields_}
_OUT = c2f.OUT_SCARS | c2f.OUT_COUNTERS | c2f.OUT_IGN_STEPS


@pytest.fixture(scope="module")
def ctx():
    c2f.build()
    with c2f.Context(0) as c:
        yield c


def _params(d):
    return c2f.default_params(**{k: v for k, v in dict(d, outputs=_OUT).items() if k in _KEYS})


@pytest.mark.parametrize("smem", [1, 0])
@pytest.mark.parametrize("over", [
    dict(const_ros=25.0),                                  # whole rings cross at once
    dict(const_ros=100.0),                                 # orthogonal neighbours every period
    dict(const_ros=150.0, minutes_per_step=5),             # every axis every period
    dict(const_ros=9.0, const_bros=3.0, const_lb=1.5),     # an ellipse: fronts a few periods apart
    dict(const_ros=25.0, ros_sigma=0.5),
    dict(const_ros=25.0, burnout_delta=1.0, ros_sigma=0.3),
    dict(const_ros=40.0, ros_threshold=38.0, ros_sigma=0.2),
    dict(const_ros=25.0, burnout_delta=30.0),              # every cell dies as it ignites
    dict(burn_hours_min=1, burn_hours_max=2, const_ros=30.0),
])
def test_simultaneous_fronts_equal_the_oracle(ctx, over, smem):
    rows, cols, hours = 150, 301, 4   # wider than the 256-column plane window
    rng = np.random.default_rng(7)
    fuel = np.full((rows, cols), 3, dtype=np.uint8)
    fuel[rng.random((rows, cols)) < 0.05] = 0
    weather = S.constant_weather(hours)
    ctx.set_frontier_config(32, smem)
    lid = ctx.load_landscape(fuel)
    ctx.set_weather(lid, weather)
    try:
        for cell in (75 * cols + 150, 0, 149 * cols + 300, 20 * cols + 255):   # centre, corners, window edge
            fuel_ok = fuel.ravel()[cell] != 0
            d = dict(seed=11, n_replicas=2, hours=hours, minutes_per_step=1, ignition_mode=0 if fuel_ok else 1,
                     ignition_cell=cell, ros_sigma=0.0)
            d.update(over)
            p = _params(d)
            sid = ctx.simulate(lid, p)
            _, ign = ctx.get_scars(sid, 2, fuel.size, ign_steps=True)
            work, nign, _ = ctx.get_counters(sid, 2)
            counts = ctx.burn_prob(sid, fuel.size)
            ctx.release(sid)
            z = np.zeros(fuel.shape, dtype=np.float32)
            o = oracle.Oracle(fuel, z, z, cell_size=100.0, weather=weather, **d)
            ref = [o.run_replica(r) for r in range(2)]
            for r in range(2):
                assert np.array_equal(ign[r], ref[r]["ign"].ravel()), (cell, r)
                assert work[r] == ref[r]["work"] and nign[r] == ref[r]["n_ignited"], (cell, r)
            assert np.array_equal(counts, sum(x["scar"].ravel().astype(np.uint32) for x in ref))
            o.close()
    finally:
        ctx.set_frontier_config(32, 1)
        ctx.release(lid)


@pytest.mark.parametrize("minutes", [1, 3, 4, 60])
@pytest.mark.parametrize("ellipse_mode", [0, 1])
def test_rates_at_the_ends_of_the_range(ctx, ellipse_mode, minutes):
    w = S.config2(side=45, n_replicas=1, hours=8)
    L = w.landscape
    L.fuel[0, :15] = np.arange(1, 16)
    L.fuel[1, :15] = np.arange(1, 16)
    L.slope[0, :15] = 0.0
    L.slope[1, :15] = 500.0
    weather = w.weather.copy()
    weather[0] = (0.0, 0.0, 90.0, 80.0)        # calm: no net wind on flat cells
    weather[1] = (0.4, 90.0, 90.0, 80.0)       # grass below 1 km/h: a circle
    weather[2] = (900.0, 45.0, 99.0, 200.0)    # extreme length-to-breadth ratios
    weather[3] = (20.0, 10.0, 0.0, 80.0)       # wet: vanishing rates
    weather[4] = (20.0, 10.0, 92.0, 0.05)      # build-up effect underflows: no spread
    weather[5] = (20.0, 180.0, 100.9, 9e5)
    weather[6] = (40.0, 270.0, 90.0, 80.0)     # the wind function's switch
    d = dict(w.params, hours=8, minutes_per_step=minutes, ellipse_mode=ellipse_mode)
    lid = ctx.load_landscape(L.fuel, L.slope, L.aspect, cell_size=L.cell_size)
    ctx.set_weather(lid, weather)
    o = oracle.Oracle(L.fuel, L.slope, L.aspect, cell_size=L.cell_size, weather=weather, **d)
    n = L.fuel.size
    cells = [c for c in range(n) if L.fuel.ravel()[c] and (c < 2 * 45 or c % 11 == 0)]
    for h in range(8):
        _, hros, base = ctx.get_ros(lid, _params(d), h, n)
        for c in cells:
            b, hr = o.base_inc(c, h)
            assert np.array_equal(base[c], b), (h, c, L.fuel.ravel()[c])
            assert hros[c] == hr, (h, c)
    o.close()
    ctx.release(lid)


@pytest.mark.parametrize("replicas", [1, 5, 320])
@pytest.mark.parametrize("smem", [1, 0])
def test_helped_on_demand_rows_equal_the_eager_table(ctx, smem, replicas):
    """On-demand tables: one replica, a few, and more than two an SM (no helper warps); a window of new
    chunks from one to thirty-two at a time."""
    w = S.config2(side=301, n_replicas=replicas, hours=6)
    L = w.landscape
    p = _params(dict(w.params, ros_threshold=1.0))
    ctx.set_frontier_config(32, smem)
    out = []
    try:
        for eager in (False, True):
            ctx.set_table_mode(eager)
            lid = ctx.load_landscape(L.fuel, L.slope, L.aspect, cell_size=L.cell_size)
            ctx.set_weather(lid, w.weather)
            sid = ctx.simulate(lid, p)
            out.append((ctx.get_counters(sid, replicas), ctx.burn_prob(sid, L.fuel.size),
                        ctx.get_replica_scar(sid, replicas - 1, L.fuel.size, ign_steps=True)))
            ctx.release(sid)
            ctx.release(lid)
    finally:
        ctx.set_frontier_config(32, 1)
        ctx.set_table_mode(True)
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    assert np.array_equal(out[0][1], out[1][1])
    for a, b in zip(out[0][2], out[1][2]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("replicas", [1215, 1217, 2500])
def test_crowded_launches_equal_small_ones(ctx, replicas):
    """Above eight replicas an SM the frontier takes global lists: the same replicas, alone and in the crowd."""
    w = S.config2(side=90, n_replicas=replicas, hours=5)
    L = w.landscape
    lid = ctx.load_landscape(L.fuel, L.slope, L.aspect, cell_size=L.cell_size)
    ctx.set_weather(lid, w.weather)
    n = L.fuel.size
    sid = ctx.simulate(lid, _params(w.params))
    work, nign, _ = ctx.get_counters(sid, replicas)
    few = ctx.simulate(lid, _params(dict(w.params, n_replicas=300)))
    w300, n300, _ = ctx.get_counters(few, 300)
    assert np.array_equal(work[:300], w300) and np.array_equal(nign[:300], n300)
    for r in (0, 299):
        for a, b in zip(ctx.get_replica_scar(sid, r, n, ign_steps=True), ctx.get_replica_scar(few, r, n, ign_steps=True)):
            assert np.array_equal(a, b)
    ctx.release(sid)
    ctx.release(few)
    ctx.release(lid)


@pytest.mark.parametrize("smem", [1, 0])
@pytest.mark.parametrize("capacity", [0, 300, 2100])   # default; retried at four times as many; nearly full of live entries
@pytest.mark.parametrize("over", [
    dict(const_ros=100.0),                   # rings of up to 660 cells ignite in one period
    dict(const_ros=60.0, ros_sigma=0.4, burnout_delta=30.0),   # some burn out at each hour's start
    dict(const_ros=60.0, ros_sigma=0.3),     # up to 348 cells in one period
])
def test_periods_of_many_windows_equal_the_oracle(ctx, over, capacity, smem):
    """Lists of more than one scan round (1,024 entries) whose periods take many windows, and compactions among them."""
    rows, cols, hours = 330, 340, 3
    fuel = np.full((rows, cols), 3, dtype=np.uint8)
    weather = S.constant_weather(hours)
    d = dict(dict(seed=5, n_replicas=1, hours=hours, minutes_per_step=1, ignition_mode=0,
                  ignition_cell=165 * cols + 170, ros_sigma=0.0), **over)
    ctx.set_frontier_config(32, smem)
    ctx.set_list_capacity(capacity)
    lid = ctx.load_landscape(fuel)
    ctx.set_weather(lid, weather)
    try:
        sid = ctx.simulate(lid, _params(d))
        _, ign = ctx.get_scars(sid, 1, fuel.size, ign_steps=True)
        work, nign, _ = ctx.get_counters(sid, 1)
        ctx.release(sid)
    finally:
        ctx.set_frontier_config(32, 1)
        ctx.set_list_capacity(0)
        ctx.release(lid)
    z = np.zeros(fuel.shape, dtype=np.float32)
    o = oracle.Oracle(fuel, z, z, cell_size=100.0, weather=weather, **d)
    ref = o.run_replica(0)
    o.close()
    assert np.array_equal(ign[0], ref["ign"].ravel())
    assert work[0] == ref["work"] and nign[0] == ref["n_ignited"]
