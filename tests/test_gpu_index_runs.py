"""Segment index of label maps whose runs are shorter and longer than a thread's four and a warp's 128 pixels, at widths
around both, through the cost volume of every segment against the oracle; labels outside the segments are reported."""
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


@pytest.mark.parametrize("w", [3, 4, 127, 128, 132, 515, 640])
@pytest.mark.parametrize("mean", [1, 3, 40, 300, 0])
def test_runs_of_equal_labels(w, mean):
    h, L, S = 9, 2, 6
    rng = np.random.default_rng(w + 7 * mean)
    lab = np.zeros(w * h, np.int64) if mean == 0 else np.repeat(rng.integers(0, S, w * h), rng.geometric(1 / mean, w * h))[: w * h]
    lab = lab.reshape(h, w).astype(np.int32)
    cams = synth.linear_rig(2, 0.2, 80.0, w, h)
    views = [synth.View(*(rng.integers(0, 256, (h, w)).astype(np.uint8) for _ in range(3))) for _ in cams]
    ctx = ftv.ftv_depth_init(cams, [0], L, 1.0, 6.0, sample_bytes=1, bit_depth=8, oob_penalty=765, max_segments=S)
    planes = [[dev(a) for a in (v.Y, v.U, v.V)] for v in views]
    cost = torch.full((S, L), -1, dtype=torch.int32, device="cuda")
    ftv.ftv_cost_volume(ctx, planes, [dev(lab)], [S], [cost])
    assert ftv.ftv_check(ctx) == 0
    H = oracle.homography_table(cams, 0, [1], L, 1.0, 6.0)
    assert np.array_equal(cost.cpu().numpy(), oracle.cost_volume(cams, views, 1, 0, [1], H, L, lab, S, 765))
    lab[h // 2, w // 2] = S if mean % 2 else -1
    ftv.ftv_segment_index(ctx, 0, dev(lab), S)
    assert ftv.ftv_check(ctx) == ftv.FTV_ERR_INVALID_ARG
