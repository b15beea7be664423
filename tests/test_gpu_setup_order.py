"""Objects created while the default stream still has work to do, then used at once on a non-blocking stream (which is
not ordered after it): what creation clears and uploads has arrived. Results against the oracle."""
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

BUSY = 100_000_000  # clock ticks of waiting on the default stream, about 50 ms


def test_created_behind_a_busy_default_stream():
    w, h, L, bits = 96, 40, 5, 8
    rng = np.random.default_rng(4)
    cams = synth.linear_rig(2, 0.2, 80.0, w, h)
    views = [synth.View(*(rng.integers(0, 256, (h, w)).astype(np.uint8) for _ in range(3))) for _ in cams]
    ys, xs = np.mgrid[0:h, 0:w]
    lab = (ys // 8 * 12 + xs // 8).astype(np.int32)
    S = int(lab.max()) + 1
    planes, lm = [[dev(a) for a in (v.Y, v.U, v.V)] for v in views], dev(lab)
    out = [torch.zeros(S, dtype=torch.int16, device="cuda") for _ in cams]
    seg = torch.zeros((h, w), dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY)
    ctx = ftv.ftv_depth_init(cams, [0, 1], L, 1.0, 6.0, sample_bytes=1, bit_depth=bits, oob_penalty=765, max_segments=S)
    torch.cuda._sleep(BUSY)
    ftv.ftv_stream_init(ctx, [lm, lm], [S, S], 3, 1, ftv.FTV_TM_ALL_YUV, stream=side)
    torch.cuda._sleep(BUSY)
    batch = ftv.ftv_batch_create(1, 2, 2)
    assert ftv.ftv_batch_prepare(batch, [dict(ctx=ctx, planes=planes, frame_type=ftv.FTV_FRAME_I, label_out=out)]) == 0
    ftv.ftv_batch_launch(batch, stream=side)
    assert ftv.ftv_batch_wait(batch) == 0
    torch.cuda._sleep(BUSY)
    sg = ftv.Segmenter([(w, h)], 1, bits, 8, 5, 3)
    ftv.ftv_superpixels(sg, [planes[0]], [seg], stream=side)
    assert ftv.ftv_segmenter_check(sg, stream=side) == 0
    side.synchronize()
    for r in range(2):
        H = oracle.homography_table(cams, r, [1 - r], L, 1.0, 6.0)
        want = oracle.wta(oracle.cost_volume(cams, views, 1, r, [1 - r], H, L, lab, S, 765))
        assert np.array_equal(out[r].cpu().numpy().view(np.uint16), want)
    assert np.array_equal(seg.cpu().numpy(), oracle.superpixels(views[0], 1, bits, 8, 5, 3))
    sg.close()
