"""Two segmenters of one assignment form and different grid steps, the one with the larger tiles created first and used
after the other: neither's set-up may change the other's launches."""
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


@pytest.mark.parametrize("bits,steps", [(8, (4, 10)), (10, (13, 64)), (12, (9, 20)), (12, (1, 64))])
def test_used_in_turn(bits, steps):
    w, h, sb = 150, 90, 1 if bits <= 8 else 2
    view = synth.mosaic(w, h, 40, bit_depth=bits, noise_sigma=(1 << bits) / 60, seed=steps[0])
    planes = [tuple(dev(a) for a in (view.Y, view.U, view.V))]
    segs = [ftv.Segmenter([(w, h)], sb, bits, S, 5, 3) for S in steps]
    for k in (0, 1, 0):
        out = torch.full((h, w), -3, dtype=torch.int32, device="cuda")
        ftv.ftv_superpixels(segs[k], planes, [out])
        assert ftv.ftv_segmenter_check(segs[k]) == 0
        assert np.array_equal(out.cpu().numpy(), oracle.superpixels(view, sb, bits, steps[k], 5, 3))
    for sg in segs:
        sg.close()
