"""ftv_skipped_evaluations on rigs where every tile of the cost kernel is one segment (32 x 32 pixels), so that the
evaluations decided for a whole tile can be counted from the homography tables: whole-number shifts that move all
columns of a tile out of the view, in both precisions, and a convergent rig, where they are the culled ones."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

ftv = pytest.importorskip("paper_1909_02294_gb300")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
from gpu_runs import dev  # noqa: E402

W, H, L, CELL = 512, 64, 9, 32  # CELL * CELL: the kernel's tile


def _run(cams, precision, combine):
    rng = np.random.default_rng(1)
    views = [synth.View(*(rng.integers(0, 256, (H, W)).astype(np.uint8) for _ in range(3))) for _ in cams]
    ys, xs = np.mgrid[0:H, 0:W]
    lab = (ys // CELL * (W // CELL) + xs // CELL).astype(np.int32)
    S = int(lab.max()) + 1
    refs = list(range(len(cams)))
    ctx = ftv.ftv_depth_init(cams, refs, L, 1.0, 6.0, sample_bytes=1, bit_depth=8, oob_penalty=300, max_segments=S,
                             precision=precision, combine=combine)
    cost = [torch.zeros((S, L), dtype=torch.int32, device="cuda") for _ in refs]
    ftv.ftv_cost_volume(ctx, [[dev(a) for a in (v.Y, v.U, v.V)] for v in views], [dev(lab)] * len(refs), [S] * len(refs), cost)
    assert ftv.ftv_check(ctx) == 0
    counts = ftv.ftv_skipped_evaluations(ctx), ftv.ftv_culled_evaluations(ctx)
    table = oracle.homography_table_f64 if precision == ftv.FTV_PRECISION_FP64 else oracle.homography_table
    tables = []
    for r in refs:
        nb = [v for v in refs if v != r]
        tables.append(table(cams, r, nb, L, 1.0, 6.0))
        want = oracle.cost_volume(cams, views, 1, r, nb, tables[-1], L, lab, S, 300,
                                  combine="min" if combine == ftv.FTV_COMBINE_MIN else "sum")
        assert np.array_equal(cost[r].cpu().numpy(), want)
    ctx.close()
    return counts, tables


@pytest.mark.parametrize("precision", [ftv.FTV_PRECISION_FP32, ftv.FTV_PRECISION_FP64])
@pytest.mark.parametrize("combine", [ftv.FTV_COMBINE_MIN, ftv.FTV_COMBINE_SUM])
def test_linear_rig(precision, combine):
    (skipped, culled), tables = _run(synth.linear_rig(4, 0.25, 717.7, W, H), precision, combine)
    h = np.concatenate([t.reshape(-1, 9) for t in tables]).astype(np.float64)
    assert np.array_equal(h[:, [0, 1, 3, 4, 5, 6, 7, 8]], np.tile([1, 0, 0, 1, 0, 0, 0, 1], (len(h), 1)))
    frac = (h[:, 2] + 0.5) % 1.0
    assert np.all((frac > 0.02) & (frac < 0.98))  # no entry near a rounding boundary: all are whole-number shifts
    D = np.floor(h[:, 2] + 0.5)[:, None]
    x0 = np.tile(np.arange(0, W, CELL), H // CELL)[None, :]
    out = (x0 + CELL - 1 + D < 0) | (x0 + D >= W)
    assert 0.05 < out.mean() < 0.95
    assert skipped == int(out.sum()) * CELL * CELL
    assert culled == 0


def test_convergent_rig():
    (skipped, culled), _ = _run(synth.arc_rig(3, 3.0, 25.0, 700.0, W, H, seed=2), ftv.FTV_PRECISION_FP32, ftv.FTV_COMBINE_MIN)
    assert skipped == culled > 0
