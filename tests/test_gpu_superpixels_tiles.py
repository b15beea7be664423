"""Superpixel segmentation at the edges of its tilings, against the oracle: widths and heights around the 32- and
64-pixel tiles, steps around the five rows of a group, every distance form, one and several images, and an image large
enough for the assignment's four groups per thread."""
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


@pytest.mark.parametrize("sizes,bits,step,compactness,iters", [
    ([(33, 31)], 8, 1, 5, 2), ([(64, 20), (65, 21), (63, 19)], 8, 5, 5, 3), ([(97, 66)], 8, 6, 0, 4),
    ([(128, 96), (31, 200)], 10, 10, 5, 5), ([(130, 70)], 10, 11, 255, 3), ([(200, 130)], 12, 16, 5, 4),
    ([(190, 150)], 16, 64, 5, 3), ([(1, 1), (1, 90), (90, 1)], 16, 7, 20, 2), ([(1537, 1093)], 10, 9, 5, 3),
    ([(1024, 1030), (700, 800)], 8, 3, 5, 2)])
def test_tilings_equal_the_oracle(sizes, bits, step, compactness, iters):
    rng = np.random.default_rng(step + bits)
    views = [synth.mosaic(w, h, max(1, w * h // 300), bit_depth=bits, noise_sigma=(1 << bits) / 60, seed=int(rng.integers(1 << 30)))
             for w, h in sizes]
    sb = 1 if bits <= 8 else 2
    sg = ftv.Segmenter(sizes, sb, bits, step, compactness, iters)
    planes = [tuple(dev(a) for a in (v.Y, v.U, v.V)) for v in views]
    out = [torch.full((h, w), -3, dtype=torch.int32, device="cuda") for w, h in sizes]
    for _ in range(2):  # the second call finds the first one's scratch
        ftv.ftv_superpixels(sg, planes, out)
        assert ftv.ftv_segmenter_check(sg) == 0
        for v, o in zip(views, out):
            assert np.array_equal(o.cpu().numpy(), oracle.superpixels(v, sb, bits, step, compactness, iters))
    sg.close()


def test_an_image_of_noise_large_enough_to_draw_turns():
    """5.3 million pixels of noise: nearly every pixel is its own component, the lists and tile loops of the merge are long
    enough for the drawn turns."""
    w, h = 2636, 2011
    rng = np.random.default_rng(6)
    view = synth.View(*(rng.integers(0, 256, (h, w)).astype(np.uint8) for _ in range(3)))
    sg = ftv.Segmenter([(w, h)], 1, 8, 12, 0, 1)
    out = [torch.full((h, w), -3, dtype=torch.int32, device="cuda")]
    ftv.ftv_superpixels(sg, [tuple(dev(a) for a in (view.Y, view.U, view.V))], out)
    assert ftv.ftv_segmenter_check(sg) == 0
    assert np.array_equal(out[0].cpu().numpy(), oracle.superpixels(view, 1, 8, 12, 0, 1))
    sg.close()
