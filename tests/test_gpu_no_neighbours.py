"""A context without neighbours (temporal test, adjacency: it samples nothing) beside a convergent one: its volume is
zero, and a batch of the two, whose texel formats differ, gives the convergent stream the oracle's labels."""
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


@pytest.mark.parametrize("bits", [10, 12])
@pytest.mark.parametrize("precision", [ftv.FTV_PRECISION_FP32, ftv.FTV_PRECISION_FP64])
def test_alone_and_in_a_batch(bits, precision):
    w, h, L = 61, 37, 5
    rng = np.random.default_rng(bits)
    cams = synth.arc_rig(3, 3.0, 10.0, 70.0, w, h, seed=3)
    views = [synth.View(*(rng.integers(0, 1 << bits, (h, w)).astype(np.uint16) for _ in range(3))) for _ in cams]
    planes = [[dev(a.view(np.int16)) for a in (v.Y, v.U, v.V)] for v in views]
    ys, xs = np.mgrid[0:h, 0:w]
    lab = (ys // 6 * 11 + xs // 6).astype(np.int32)
    S, penalty = int(lab.max()) + 1, 3 * ((1 << bits) - 1)
    ctx = [ftv.ftv_depth_init(cams, [0, 1, 2], L, 1.0, 6.0, sample_bytes=2, bit_depth=bits, oob_penalty=penalty,
                              max_segments=S, nbr_lists=nb, precision=precision) for nb in (None, [[], [], []])]
    cost = [torch.full((S, L), 7, dtype=torch.int32, device="cuda") for _ in cams]
    ftv.ftv_cost_volume(ctx[1], planes, [dev(lab)] * 3, [S] * 3, cost)
    assert ftv.ftv_check(ctx[1]) == 0
    assert all(int(c.abs().max()) == 0 for c in cost)
    out = [[torch.full((S,), 9, dtype=torch.int16, device="cuda") for _ in cams] for _ in ctx]
    for c in ctx:
        ftv.ftv_stream_init(c, [dev(lab)] * 3, [S] * 3, 3, 1, ftv.FTV_TM_ALL_YUV)
    batch = ftv.ftv_batch_create(2, 6, 6)
    assert ftv.ftv_batch_prepare(batch, [dict(ctx=c, planes=planes, frame_type=ftv.FTV_FRAME_I, label_out=o)
                                         for c, o in zip(ctx, out)]) == 0
    ftv.ftv_batch_launch(batch)
    assert ftv.ftv_batch_wait(batch) == 0
    table = oracle.homography_table_f64 if precision == ftv.FTV_PRECISION_FP64 else oracle.homography_table
    for r in range(3):
        nb = [k for k in range(3) if k != r]
        H = table(cams, r, nb, L, 1.0, 6.0)
        want = oracle.wta(oracle.cost_volume(cams, views, 2, r, nb, H, L, lab, S, penalty))
        assert np.array_equal(out[0][r].cpu().numpy().view(np.uint16), want)
        assert int(out[1][r].abs().max()) == 0
