"""CPU check of the FP64 projection mode's staging in FP32 arithmetic (the cost kernel's stage_precise): its bounds are
restated in IEEE float32 and every decision that they let stand is compared with the FP64 projection, over random
convergent tiles, tiles beyond each image edge, homographies of very large and very small scale and a rig whose
every sample lies next to a rounding boundary."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
import test_precise_round_cpu as rounding
from test_precise_bound_cpu import _near_tie_table, f32_down, stage

F = np.float32


def stage32(h, x0, y0, rx, ry, wv, hv):
    h = np.asarray(h, np.float64)
    hx = lambda s: F(float.fromhex(s))
    x0d, y0d = np.float64(x0), np.float64(y0)
    X0, Y0, W0 = (h[i] * x0d + (h[i + 1] * y0d + h[i + 2]) for i in (0, 3, 6))
    with np.errstate(all="ignore"):
        X0f, Y0f, c = F(X0), F(Y0), [None] * 6 + [F(h[6]), F(h[7]), F(W0)]
        up, frx, fry = F(1.0 + 2.0 ** -18), F(rx), F(ry)
        ax, ay = abs(F(x0)) + frx, abs(F(y0)) + fry
        c0, c1, c2 = (abs(v) for v in c[6:])
        AW = up * (F(2) * (c0 * ax + c1 * ay) + c2) + F(2.0 ** -120)
        Rc = c0 * frx + c1 * fry
        gW = up * Rc + F(2.0 ** -48) * AW + hx("0x1.1p-24") * c2 + F(2.0 ** -120)
        if c[8] + gW < 0:
            return "out", None
        Wlo = (c[8] - gW) * (F(2) - up)
        if not (Wlo > F(2.0 ** -60) and Wlo < F(2.0 ** 100)):
            return "slow", None
        U0, V0 = (np.rint(np.fmin(np.fmax(q / c[8], F(-2.0 ** 24)), F(2.0 ** 24))) for q in (X0f, Y0f))
        for i, P, C in ((0, U0, X0), (3, V0, Y0)):
            P = np.float64(P)
            c[i], c[i + 1], c[i + 2] = F(h[i] - P * h[6]), F(h[i + 1] - P * h[7]), F(C - P * W0)
        M = [up * (abs(c[i]) * frx + abs(c[i + 1]) * fry + abs(c[i + 2])) + F(2.0 ** -120) for i in (0, 3)]
        Mc = up * (Rc + c2) + F(2.0 ** -120)
        A = [up * (F(2) * ((abs(c[i]) + abs(P) * c0) * ax + (abs(c[i + 1]) + abs(P) * c1) * ay) + abs(C)) + F(2.0 ** -100)
             for i, P, C in ((0, U0, X0f), (3, V0, Y0f))]
        k3 = hx("0x1.82p-23")
        e = [k3 * M[i] + F(2.0 ** -50) * (M[i] + A[i] + abs(P) * AW) for i, P in ((0, U0), (1, V0))]
        eW = k3 * Mc + F(2.0 ** -50) * (Mc + AW)
        if not Wlo > F(2) * eW:
            return "slow", None
        rW = up * (F(1) / (Wlo - eW))
        B = [up * (M[i] + F(2) * e[i]) * rW for i in (0, 1)]
        d = [F(1.0625) * ((e[i] + B[i] * eW + hx("0x1.8p-52") * (A[i] + (abs(P) + B[i]) * AW)) * rW + hx("0x1.01p-23") * B[i] +
                     hx("0x1.02p-52") * (abs(P) + B[i] + F(1))) + F(2.0 ** -30)
             for i, P in ((0, U0), (1, V0))]
        l = [up * (B[i] + d[i]) for i in (0, 1)]
        if (U0 < F(-0.501) - l[0] or F(int(U0) - wv) > l[0] - F(0.499) or V0 < F(-0.501) - l[1]
                or F(int(V0) - hv) > l[1] - F(0.499)):
            return "out", None
        if not (d[0] < 0.25 and d[1] < 0.25 and max(B) < 2.0 ** 21):
            return "slow", None
    assert all(v.dtype == np.float32 for v in (U0, V0, eW, rW, *M, *A, *e, *B, *d))
    rect = (c[0] == 1 and c[1] == 0 and c[3] == 0 and c[4] == 1 and c[6] == 0 and c[7] == 0 and c[8] == 1
            and abs(c[5]) + d[1] < F(0.49))
    thr = [f32_down(0.5 - float(np.nextafter(v + F(2.0 ** -22), F(1)))) for v in d]
    return ("rect" if rect else "general"), (c, int(U0), int(V0), thr[0], thr[1])


@pytest.mark.parametrize("scale", [1.0, 2.0 ** 60, 2.0 ** -40, 2.0 ** 140, 2.0 ** -140])
def test_convergent_tiles(monkeypatch, scale):
    monkeypatch.setattr(rounding, "stage", stage32)
    rng = np.random.default_rng(3)
    W, H = 3840, 2160
    decided = near = near64 = 0
    modes = []
    for _ in range(12):
        cams = synth.arc_rig(4, 3.0, float(rng.uniform(4, 60)), float(rng.uniform(800, 4000)), W, H,
                             seed=int(rng.integers(1 << 30)), roll_deg=5.0)
        table = oracle.homography_table_f64(cams, 1, [0, 2, 3], 30, 0.8, 15.0)
        for _ in range(6):
            h = [float(v) * scale for v in table[int(rng.integers(3)), int(rng.integers(30))]]
            bw, bh = int(rng.integers(1, 130)), int(rng.integers(1, 20))
            x, y = int(rng.choice([0, W - bw, rng.integers(0, W - bw)])), int(rng.integers(0, H - bh))
            a, b = rounding._check(h, W, H, x, y, bw, bh)
            decided, near = decided + a, near + b
            x0, y0 = (2 * x + bw - 1) >> 1, (2 * y + bh - 1) >> 1
            modes.append((stage(h, x0, y0, bw, bh, W, H)[0], stage32(h, x0, y0, bw, bh, W, H)[0]))
            monkeypatch.setattr(rounding, "stage", stage)
            near64 += rounding._check(h, W, H, x, y, bw, bh)[1] if 2.0 ** -60 < scale < 2.0 ** 100 else 0
            monkeypatch.setattr(rounding, "stage", stage32)
    if 2.0 ** -60 < scale < 2.0 ** 100:  # outside, the FP32 bounds leave every evaluation to FP64
        assert decided > 20000 and near <= 1.01 * near64  # as few left to FP64 as with bounds formed in FP64
        assert sum(a != b for a, b in modes) <= 1 and any(b == "out" for _, b in modes)


@pytest.mark.parametrize("box", [(100, 10, 40, 9), (3700, 0, 130, 16), (0, 50, 8, 1)])
def test_samples_next_to_a_rounding_boundary(monkeypatch, box):
    monkeypatch.setattr(rounding, "stage", stage32)
    table, W, H = _near_tie_table()
    total = [rounding._check([float(v) for v in table[0, d]], W, H, *box) for d in range(table.shape[1])]
    assert sum(a + b for a, b in total) > 0


def test_homographies_with_w_near_zero_or_negative(monkeypatch):
    monkeypatch.setattr(rounding, "stage", stage32)
    rng = np.random.default_rng(8)
    for _ in range(60):
        h = [1.0, 0.01, 3.0, -0.02, 1.0, 5.0, float(rng.uniform(-2e-3, 2e-3)), float(rng.uniform(-2e-3, 2e-3)),
             float(rng.uniform(-1.5, 1.5))]
        with np.errstate(all="ignore"):
            rounding._check(h, 1920, 1080, int(rng.integers(0, 1800)), int(rng.integers(0, 1060)), 100, 12)
