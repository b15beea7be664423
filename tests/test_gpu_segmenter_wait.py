"""The bounded wait of the segmentation's last kernel: with a limit of one poll its blocks do not wait for one another, the
kernel ends early and the check reports it; the next call with the default limit is complete and exact."""
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


def test_a_wait_that_runs_out_is_reported():
    w, h = 900, 700
    view = synth.mosaic(w, h, 300, bit_depth=8, noise_sigma=5.0, seed=3)
    planes = [tuple(dev(a) for a in (view.Y, view.U, view.V))]
    out = torch.full((h, w), -3, dtype=torch.int32, device="cuda")
    sg = ftv.Segmenter([(w, h)], 1, 8, 10, 5, 3)
    for _ in range(2):
        ftv.ftv_segmenter_set_poll_limit(sg, 1)
        ftv.ftv_superpixels(sg, planes, [out])
        assert ftv.ftv_segmenter_check(sg) == ftv.FTV_ERR_TIMEOUT
        assert ftv.ftv_segmenter_check(sg) == 0  # cleared by the report
        ftv.ftv_segmenter_set_poll_limit(sg, 0)
        ftv.ftv_superpixels(sg, planes, [out])
        assert ftv.ftv_segmenter_check(sg) == 0
        assert np.array_equal(out.cpu().numpy(), oracle.superpixels(view, 1, 8, 10, 5, 3))
    with pytest.raises(ftv.FtvError):
        ftv.ftv_segmenter_set_poll_limit(sg, -1)
    sg.close()
