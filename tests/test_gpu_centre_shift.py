"""The centre table's integer-shift entries and packed 8-bit comparison against the oracle: disparities on, next to and
away from half-integers, neighbours wider, narrower and lower than the reference, segments of one to many pixels (centres in
every corner and border), samples at both ends of the range. Everything is exact."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

ftv = pytest.importorskip("paper_1909_02294_gb300")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from gpu_runs import dev  # noqa: E402


@pytest.mark.parametrize("bits", [8, 10])
@pytest.mark.parametrize("first,step", [(0.5, 1.0), (0.25, 0.25), (1.50001, 0.5), (3.0, 7.0)])
def test_rectified_rig(bits, first, step):
    w, h, L, f, B = 45, 14, 9, 64.0, 0.25
    K = synth.intrinsics(f, w, h)
    sizes = [(w, h), (w, h), (w + 6, h + 3), (w - 9, h), (w, h - 5)]
    cams = [synth.Camera(K, np.eye(3), np.array([-B * k, 0.0, 0.0]), *s) for k, s in enumerate(sizes)]
    z_near, z_far = f * B / (first + step * (L - 1)), f * B / first
    rng = np.random.default_rng(bits)
    top, dtype = (1 << bits) - 1, (np.uint8 if bits == 8 else np.uint16)
    views = [synth.View(*(np.where(rng.random((c.height, c.width)) < 0.3, rng.choice([0, top], (c.height, c.width)),
                                   rng.integers(0, top + 1, (c.height, c.width))).astype(dtype) for _ in range(3)))
             for c in cams]
    sb, penalty = (1 if bits == 8 else 2), 3 * top
    for cell in (1, 4):
        maps = [(np.arange(c.height)[:, None] // cell * ((c.width + cell - 1) // cell) + np.arange(c.width) // cell)
                .astype(np.int32) for c in cams]
        S = int(maps[0].max()) + 1
        ctx = ftv.ftv_depth_init(cams, [0], L, z_near, z_far, sample_bytes=sb, bit_depth=bits, oob_penalty=penalty,
                                 max_segments=S)
        planes = [[dev(a.view(np.int16) if a.dtype == np.uint16 else a) for a in (v.Y, v.U, v.V)] for v in views]
        m, sp = (torch.empty((S, L, 4), dtype=torch.int32, device="cuda") for _ in range(2))
        ftv.ftv_centre_table(ctx, planes, [dev(x) for x in maps], [S], 3, [m], [sp])
        assert ftv.ftv_check(ctx) == 0
        nb = [1, 2, 3, 4]
        H = oracle.homography_table(cams, 0, nb, L, z_near, z_far)
        mo, spo = oracle.centre_table(cams, views, sb, 0, nb, H, L, maps, S, 3, penalty)
        assert np.array_equal(m.cpu().numpy(), mo)
        assert np.array_equal(sp.cpu().numpy(), spo)
