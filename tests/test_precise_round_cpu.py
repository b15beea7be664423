"""CPU check of the FP64 projection mode's rounding form: the kernel takes the integer nearest to the FP32 local
position by adding 1.5 * 2^23 and compares the exact remainder with the staged threshold. On random convergent
tiles and on a rig whose every sample lies next to a rounding boundary, each evaluation that this decides must be
the FP64 projection's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from ieee32 import fma32
from test_precise_bound_cpu import _near_tie_table, project_f64, stage

F32 = np.float32
ROUND = F32(1.5 * 2.0 ** 23)
BITS = 0x4B400000


def nearest(t):
    """The integer nearest to t and the magnitude of the exact remainder."""
    s = (t + ROUND).astype(np.float32)
    return s.view(np.int32).astype(np.int64) - BITS, np.abs((t - (s - ROUND).astype(np.float32)).astype(np.float32))


def _check(h, W, H, x0b, y0b, bw, bh):
    xs, ys = [a.ravel() for a in np.meshgrid(np.arange(x0b, x0b + bw), np.arange(y0b, y0b + bh))]
    x0, y0 = (x0b + x0b + bw - 1) >> 1, (y0b + y0b + bh - 1) >> 1
    rx, ry = max(x0 - x0b, x0b + bw - 1 - x0), max(y0 - y0b, y0b + bh - 1 - y0)
    mode, st = stage(h, x0, y0, rx, ry, W, H)
    ok64, fu, fv = project_f64(h, xs.astype(np.float64), ys.astype(np.float64), W, H)
    if mode == "out":
        assert not ok64.any()
        return len(xs), 0
    if mode == "slow":
        return 0, len(xs)
    c, U0, V0, thr_u, thr_v = st
    xl, yl = (xs - x0).astype(np.float32), (ys - y0).astype(np.float32)
    if mode == "rect":
        ui, eu = nearest((xl + c[2]).astype(np.float32))
        ui, vi, near = ui + U0, ys + (V0 - y0), eu >= thr_u
    else:
        X, Y = fma32(c[0], xl, fma32(c[1], yl, c[2])), fma32(c[3], xl, fma32(c[4], yl, c[5]))
        r = (F32(1.0) / fma32(c[6], xl, fma32(c[7], yl, c[8]))).astype(np.float32)
        (ui, eu), (vi, ev) = nearest((X * r).astype(np.float32)), nearest((Y * r).astype(np.float32))
        ui, vi, near = ui + U0, vi + V0, (eu >= thr_u) | (ev >= thr_v)
    ok = (ui >= 0) & (ui < W) & (vi >= 0) & (vi < H)
    bad = (ok != ok64) | (ok64 & ((ui != np.where(ok64, fu, 0)) | (vi != np.where(ok64, fv, 0))))
    assert not np.any(bad & ~near)
    return int((~near).sum()), int(near.sum())


def test_convergent_tiles():
    rng = np.random.default_rng(77)
    decided = near = 0
    for _ in range(16):
        cams = synth.arc_rig(4, 3.0, float(rng.uniform(4, 30)), float(rng.uniform(800, 4000)), 3840, 2160,
                             seed=int(rng.integers(1 << 30)), roll_deg=5.0)
        table = oracle.homography_table_f64(cams, 1, [0, 2, 3], 30, 0.8, 15.0)
        for _ in range(6):
            h = [float(v) for v in table[int(rng.integers(3)), int(rng.integers(30))]]
            bw, bh = int(rng.integers(1, 130)), int(rng.integers(1, 20))
            a, b = _check(h, 3840, 2160, int(rng.integers(0, 3840 - bw)), int(rng.integers(0, 2160 - bh)), bw, bh)
            decided, near = decided + a, near + b
    assert decided > 30000 and near < 0.01 * decided


@pytest.mark.parametrize("box", [(100, 10, 40, 9), (3700, 0, 130, 16), (0, 50, 8, 1)])
def test_samples_next_to_a_rounding_boundary(box):
    table, W, H = _near_tie_table()
    total = [0, 0]
    for d in range(table.shape[1]):
        a, b = _check([float(v) for v in table[0, d]], W, H, *box)
        total = [total[0] + a, total[1] + b]
    assert sum(total) > 0
