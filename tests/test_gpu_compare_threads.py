"""Scar comparison over its CTA sizes (needs a GB300).

The CTA takes 128 to 1,024 threads by the replica count and the grid size; the
metrics are functions of whole-number counts, so they are compared with the
same functions of counts taken from the ignition steps: MSE and the norm
exactly (one rounding of exact integers), SSIM to 1e-12 (a dozen roundings).
"""
import numpy as np
import pytest

import c2f_synth as S
import paper_1905_09317_gb300 as c2f

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols,replicas", [
    (3, 5, 2),          # fewer cells than threads
    (60, 61, 3),        # 128 threads
    (70, 61, 4),        # 256, cells not a multiple of four
    (100, 90, 5),       # 512
    (131, 127, 7),      # 1,024, ragged
    (192, 180, 2),      # 1,024, 16-byte loads
    (100, 90, 1300),    # many replicas: 128 again
])
def test_metrics_equal_counts(rows, cols, replicas):
    hours = 5
    L = S.heterogeneous_landscape(rows, cols, seed=rows)
    c2f.build()
    n = rows * cols
    with c2f.Context(0) as ctx:
        lid = ctx.load_landscape(L.fuel, L.slope, L.aspect, cell_size=L.cell_size)
        p = c2f.default_params(seed=5, n_replicas=replicas, hours=hours, ignition_mode=1, ros_sigma=0.1,
                               outputs=c2f.OUT_SCARS | c2f.OUT_COUNTERS | c2f.OUT_IGN_STEPS)
        sims, steps = [], []
        for k in range(2):
            ctx.set_weather(lid, S.weather_stream(hours, seed=40 + k))
            sims.append(ctx.simulate(lid, p))
            steps.append(ctx.get_scars(sims[-1], replicas, n, ign_steps=True)[1])
        mse, ssim, norm = ctx.compare_scars(sims[0], sims[1], replicas, hours)
    for r in range(0, replicas, max(1, replicas // 8)):
        x, y = steps[0][r], steps[1][r]
        for t in range(hours):
            sx, sy = (x >= 0) & (x <= (t + 1) * 60), (y >= 0) & (y <= (t + 1) * 60)
            a, b, c = float(sx.sum()), float(sy.sum()), float((sx & sy).sum())
            assert mse[r, t] == (a + b - 2.0 * c) / n
            mx, my, nn = a / n, b / n, n * (n - 1.0)
            vx, vy, cxy = a * (n - a) / nn, b * (n - b) / nn, (c * n - a * b) / nn
            ref = ((2 * mx * my + 1e-4) * (2 * cxy + 9e-4)) / ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4))
            assert abs(ssim[r, t] - ref) <= 1e-12 * max(1.0, abs(ref))
        assert norm[r] == np.sqrt(float(((x >= 0) != (y >= 0)).sum()))
