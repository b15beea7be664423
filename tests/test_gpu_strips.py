"""The kernels that take four adjacent pixels per thread (packing and depth maps, alone and in a batch) and the
least-cost label, at widths around the strip and the row block, with maps and planes on and off the vector accesses'
alignment. Everything is exact."""
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


def _off(shape, dtype, by):
    """A contiguous tensor that starts `by` elements past an allocation."""
    n = int(np.prod(shape))
    return torch.zeros(n + by, dtype=dtype, device="cuda")[by:].view(shape)


@pytest.mark.parametrize("w,h", [(1, 2), (4, 1), (7, 5), (508, 2), (513, 3), (516, 2)])
@pytest.mark.parametrize("L", [1, 31, 33, 64, 250])
def test_least_label_and_depth_map(w, h, L):
    rng = np.random.default_rng(w * 31 + L)
    S = w * h + 2
    cam = synth.Camera(synth.intrinsics(100.0, w, h), np.eye(3), np.zeros(3), w, h)
    ctx = ftv.ftv_depth_init([cam], [0], L, 1.0, 9.0, nbr_lists=[[]], max_segments=S)
    cost = rng.integers(-3, 3, (S, L)).astype(np.int32)  # ties
    cost[0] = np.iinfo(np.int32).max
    cost[1, -1] = np.iinfo(np.int32).min
    want = cost.argmin(1)
    z = ftv.ftv_get_label_depths(ctx)
    lab = rng.integers(0, S, (h, w)).astype(np.int32)
    for by in (0, 1):
        lm, depth = _off((h, w), torch.int32, by), _off((h, w), torch.float32, by)
        lm.copy_(dev(lab))
        out = torch.zeros(S, dtype=torch.int16, device="cuda")
        ftv.ftv_wta_depth(ctx, 0, dev(cost), S, out, labels_pix=lm, depth_map=depth)
        assert ftv.ftv_check(ctx) == 0
        assert np.array_equal(out.cpu().numpy().view(np.uint16), want)
        assert np.array_equal(depth.cpu().numpy(), z[want[lab]])


@pytest.mark.parametrize("w", [61, 64, 516])
@pytest.mark.parametrize("sample_bytes,bits", [(1, 8), (2, 10), (2, 12), (2, 16)])
@pytest.mark.parametrize("rig", ["linear", "arc"])
def test_batch_of_one_frame(w, sample_bytes, bits, rig):
    h, L = 24, 6
    rng = np.random.default_rng(w + bits)
    cams = synth.linear_rig(3, 0.2, 80.0, w, h) if rig == "linear" else synth.arc_rig(3, 3.0, 12.0, 80.0, w, h, seed=5)
    dtype = np.uint8 if sample_bytes == 1 else np.uint16
    views = [synth.View(*(rng.integers(0, 1 << bits, (h, w)).astype(dtype) for _ in range(3))) for _ in cams]
    ys, xs = np.mgrid[0:h, 0:w]
    lab = (ys // 6 * ((w + 6) // 7) + xs // 7).astype(np.int32)
    S = int(lab.max()) + 1
    penalty = 3 * ((1 << bits) - 1)
    for by in (0, 1):
        ctx = ftv.ftv_depth_init(cams, [0, 1, 2], L, 1.0, 6.0, sample_bytes=sample_bytes, bit_depth=bits,
                                 oob_penalty=penalty, max_segments=S)
        ftv.ftv_stream_init(ctx, [dev(lab)] * 3, [S] * 3, 3, 1, ftv.FTV_TM_ALL_YUV)
        planes = []
        for v in views:
            planes.append([])
            for a in (v.Y, v.U, v.V):
                t = _off((h, w), torch.uint8 if sample_bytes == 1 else torch.int16, by)
                t.copy_(dev(a.view(np.int16) if a.dtype == np.uint16 else a))
                planes[-1].append(t)
        out = [torch.zeros(S, dtype=torch.int16, device="cuda") for _ in cams]
        depth = [_off((h, w), torch.float32, by) for _ in cams]
        batch = ftv.ftv_batch_create(1, 3, 3)
        assert ftv.ftv_batch_prepare(batch, [dict(ctx=ctx, planes=planes, frame_type=ftv.FTV_FRAME_I, label_out=out,
                                                  depth_out=depth)]) == 0
        ftv.ftv_batch_launch(batch)
        assert ftv.ftv_batch_wait(batch) == 0
        z = ftv.ftv_get_label_depths(ctx)
        for r in range(3):
            nb = [k for k in range(3) if k != r]
            H = oracle.homography_table(cams, r, nb, L, 1.0, 6.0)
            want = oracle.wta(oracle.cost_volume(cams, views, sample_bytes, r, nb, H, L, lab, S, penalty))
            assert np.array_equal(out[r].cpu().numpy().view(np.uint16), want)
            assert np.array_equal(depth[r].cpu().numpy(), z[want[lab]])
