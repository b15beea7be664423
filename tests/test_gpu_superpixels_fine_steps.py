"""Segmentation with grid steps of one to three pixels on images large enough for several row groups per thread (steps 1
and 2 have kernels of their own), at odd sizes, against the oracle."""
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


@pytest.mark.parametrize("w,h,step", [(701, 523, 1), (1003, 771, 2), (1090, 801, 3)])
@pytest.mark.parametrize("bits", [8, 10, 12])
def test_fine_steps_equal_the_oracle(w, h, step, bits):
    sb = 1 if bits <= 8 else 2
    view = synth.mosaic(w, h, 60, bit_depth=bits, noise_sigma=(1 << bits) / 40, seed=step + bits)
    sg = ftv.Segmenter([(w, h)], sb, bits, step, 5, 2)
    out = [torch.full((h, w), -3, dtype=torch.int32, device="cuda")]
    ftv.ftv_superpixels(sg, [tuple(dev(a) for a in (view.Y, view.U, view.V))], out)
    assert ftv.ftv_segmenter_check(sg) == 0
    assert np.array_equal(out[0].cpu().numpy(), oracle.superpixels(view, sb, bits, step, 5, 2))
    sg.close()


@pytest.mark.parametrize("step,compactness", [(6, 5), (11, 10), (18, 20)])
def test_distance_form_of_the_64_column_tile(step, compactness):
    """6-bit sets whose 32-bit form the tile of 64 columns admits and one of 128 would not."""
    w, h = 203, 151
    view = synth.mosaic(w, h, 60, bit_depth=6, noise_sigma=4.0, seed=step)
    sg = ftv.Segmenter([(w, h)], 1, 6, step, compactness, 4)
    out = [torch.full((h, w), -3, dtype=torch.int32, device="cuda")]
    ftv.ftv_superpixels(sg, [tuple(dev(a) for a in (view.Y, view.U, view.V))], out)
    assert ftv.ftv_segmenter_check(sg) == 0
    assert np.array_equal(out[0].cpu().numpy(), oracle.superpixels(view, 1, 6, step, compactness, 4))
    sg.close()
