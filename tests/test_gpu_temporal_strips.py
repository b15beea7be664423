"""The temporal test's four-column strips against the oracle: widths around the strip and the tile, segments one to five
pixels wide (two, three and four labels in a strip), samples at both ends of the 8- and 16-bit ranges, planes on and
off the vector loads' alignment."""
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


@pytest.mark.parametrize("w,h", [(1, 1), (3, 9), (4, 7), (5, 8), (127, 3), (128, 8), (129, 17), (132, 16), (244, 33)])
@pytest.mark.parametrize("sample_bytes", [1, 2])
@pytest.mark.parametrize("aligned", [True, False])
def test_strips_equal_the_oracle(w, h, sample_bytes, aligned):
    bits = 8 * sample_bytes
    top, dtype = (1 << bits) - 1, (np.uint8 if sample_bytes == 1 else np.uint16)
    rng = np.random.default_rng(w + h)
    frames = [synth.View(*(np.where(rng.random((h, w)) < 0.3, rng.choice([0, top], (h, w)), rng.integers(0, top + 1, (h, w)))
                           .astype(dtype) for _ in range(3))) for _ in range(3)]
    cam = synth.Camera(synth.intrinsics(100.0, w, h), np.eye(3), np.zeros(3), w, h)
    ctx = ftv.ftv_depth_init([cam], [0], 2, 1.0, 9.0, nbr_lists=[[]], sample_bytes=sample_bytes, bit_depth=bits,
                             max_segments=w * h + 700)

    def place(a):
        a = a.view(np.int16) if a.dtype == np.uint16 else a
        if aligned:
            return dev(a)
        buf = torch.zeros(h * (w + 3) + 1, dtype=torch.int16 if a.dtype == np.int16 else torch.uint8, device="cuda")
        out = torch.as_strided(buf, (h, w), (w + 3, 1), 1)
        out.copy_(dev(a))
        return out

    planes = [[place(a) for a in (f.Y, f.U, f.V)] for f in frames]
    ys, xs = np.mgrid[0:h, 0:w]
    maps = [(ys // 4 * w + xs // k).astype(np.int32) for k in (1, 2, 3, 5)]
    maps += [rng.integers(0, w * h, (h, w)).astype(np.int32), (xs % 2 * 600).astype(np.int32), np.zeros((h, w), np.int32)]
    for lab in maps:
        S = int(lab.max()) + 2
        for mode, ifr in ((ftv.FTV_TM_ALL_YUV, 0), (ftv.FTV_TM_Y_ONLY, None), (ftv.FTV_TM_ALL_YUV, None)):
            t_p, t_i = top // 4, top // 8
            mask = torch.full((S,), 9, dtype=torch.uint8, device="cuda")
            changed, n = torch.zeros(S, dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
            ftv.ftv_temporal_mask(ctx, 0, planes[2], planes[1], planes[ifr] if ifr is not None else None, dev(lab), S, t_p,
                                  t_i, mode, mask, changed, n)
            assert ftv.ftv_check(ctx) == 0
            m, c, k = oracle.temporal_mask(lab, S, frames[2], frames[1], frames[ifr] if ifr is not None else None,
                                           sample_bytes, t_p, t_i, mode)
            assert np.array_equal(mask.cpu().numpy(), m)
            assert int(n.item()) == k and np.array_equal(changed.cpu().numpy()[:k], c[:k])
    ctx.close()
