"""How much of the FP64 projection mode's error bound is used, and that its checks can fail: over random convergent tiles the
largest error of the FP32 local position against the FP64 projection, as a share of the staged bound; on the near-tie
rig evaluations left to FP64 in every box; for homographies whose magnitudes FP32 bounds cannot hold, every entry left
to FP64."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
import test_precise_round_cpu as rounding
from ieee32 import fma32
from test_precise_bound32_cpu import stage32
from test_precise_bound_cpu import _near_tie_table


def _tiles(seed, n):
    rng = np.random.default_rng(seed)
    W, H = 3840, 2160
    for _ in range(n):
        cams = synth.arc_rig(4, 3.0, float(rng.uniform(4, 60)), float(rng.uniform(800, 4000)), W, H,
                             seed=int(rng.integers(1 << 30)), roll_deg=5.0)
        table = oracle.homography_table_f64(cams, 1, [0, 2, 3], 30, 0.8, 15.0)
        for _ in range(8):
            h = [float(v) for v in table[int(rng.integers(3)), int(rng.integers(30))]]
            bw, bh = int(rng.integers(1, 130)), int(rng.integers(1, 20))
            yield h, int(rng.integers(0, W - bw)), int(rng.integers(0, H - bh)), bw, bh, W, H


def test_the_bound_holds_and_is_used():
    worst, boxes = 0.0, 0
    for h, xb, yb, bw, bh, W, H in _tiles(12, 20):
        xs, ys = [a.ravel() for a in np.meshgrid(np.arange(xb, xb + bw), np.arange(yb, yb + bh))]
        x0, y0 = (2 * xb + bw - 1) >> 1, (2 * yb + bh - 1) >> 1
        mode, st = stage32(h, x0, y0, max(x0 - xb, xb + bw - 1 - x0), max(y0 - yb, yb + bh - 1 - y0), W, H)
        if mode != "general":
            continue
        boxes += 1
        c, U0, V0, thr_u, thr_v = st
        xl, yl = (xs - x0).astype(np.float32), (ys - y0).astype(np.float32)
        r = (np.float32(1) / fma32(c[6], xl, fma32(c[7], yl, c[8]))).astype(np.float32)
        W64 = (h[6] * xs + h[7] * ys) + h[8]
        for k, at, thr in ((0, U0, thr_u), (3, V0, thr_v)):
            t = (fma32(c[k], xl, fma32(c[k + 1], yl, c[k + 2])) * r).astype(np.float32)
            exact = ((h[k] * xs + h[k + 1] * ys) + h[k + 2]) / W64 - at
            bound = 0.5 - float(thr) - 2.0 ** -22  # the staged bound, rounded up
            worst = max(worst, float(np.abs(t - exact).max()) / bound)
    print(f"largest error {worst:.3f} of the bound over {boxes} boxes")
    assert boxes > 60
    assert 0.05 < worst < 1.0


@pytest.mark.parametrize("box,outside", [((100, 10, 40, 9), False), ((3700, 0, 130, 16), False), ((0, 50, 8, 1), True)])
def test_samples_next_to_a_boundary_are_left_to_fp64(monkeypatch, box, outside):
    """The last box's columns 0 to 7 move 10.5 px and more to the left: it is decided as a whole, the others pixel by pixel."""
    monkeypatch.setattr(rounding, "stage", stage32)
    table, W, H = _near_tie_table()
    tables = [[float(v) for v in table[0, d]] for d in range(table.shape[1])]
    counts = [rounding._check(h, W, H, *box) for h in tables]
    x0, y0 = (2 * box[0] + box[2] - 1) >> 1, (2 * box[1] + box[3] - 1) >> 1
    rx, ry = max(x0 - box[0], box[0] + box[2] - 1 - x0), max(y0 - box[1], box[1] + box[3] - 1 - y0)
    modes = {stage32(h, x0, y0, rx, ry, W, H)[0] for h in tables}
    if outside:
        assert modes == {"out"} and all(a == box[2] * box[3] for a, _ in counts)
    else:
        assert modes == {"rect"}  # the decision check is reached
        assert all(near == box[2] * box[3] for _, near in counts)


@pytest.mark.parametrize("scale", [2.0 ** 140, 2.0 ** -140])
def test_magnitudes_beyond_fp32_leave_every_entry_to_fp64(scale):
    n = 0
    for h, xb, yb, bw, bh, W, H in _tiles(13, 8):
        mode, _ = stage32([v * scale for v in h], (2 * xb + bw - 1) >> 1, (2 * yb + bh - 1) >> 1, bw, bh, W, H)
        assert mode == "slow"
        n += 1
    assert n == 64
