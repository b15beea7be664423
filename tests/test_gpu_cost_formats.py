"""The cost kernel's texel formats and tile classes against the oracle: every bit depth at which the format
changes, samples at both ends of the range, tiles wholly and partly in view, label maps whose tiles span
more than 2^16 empty segments."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import synth
from synth.configs import Workload

pytestmark = pytest.mark.gpu

ftv = pytest.importorskip("paper_1909_02294_gb300")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle  # noqa: E402
import oracle_runs  # noqa: E402
from gpu_runs import Run  # noqa: E402


def _workload(rig, bits, W=211, H=77, L=13, n=4, cell=9):
    """Random views whose samples are 0, the maximum or anything between, a third each."""
    cams = synth.linear_rig(n, 0.3, 150.0, W, H) if rig == "linear" else synth.arc_rig(n, 3.0, 12.0, 150.0, W, H, 5)
    wl = Workload(f"{rig}{bits}", cams, list(range(n)), L, 1.0, 9.0, bits, [], cell=cell, jitter=2)
    rng = np.random.default_rng(bits)
    top = (1 << bits) - 1
    for v in range(n):
        p = []
        for _ in range(3):
            a = rng.integers(0, top + 1, (H, W))
            k = rng.integers(0, 3, (H, W))
            p.append(np.where(k == 0, 0, np.where(k == 1, top, a)).astype(np.uint8 if bits <= 8 else np.uint16))
        wl._views[(v, 0, False)] = synth.View(*p)
    return wl


@pytest.mark.parametrize("rig", ["linear", "arc"])
@pytest.mark.parametrize("bits", [7, 8, 9, 10, 11, 14, 15, 16])
@pytest.mark.parametrize("combine,precision", [("min", 0), ("sum", 0), ("min", 1)])
def test_every_texel_format_is_exact_at_the_ends_of_its_range(rig, bits, combine, precision):
    wl = _workload(rig, bits)
    run = Run(wl, combine=combine, precision=precision)
    costs = run.volumes()
    assert run.check() == 0
    table = oracle.homography_table_f64 if precision else oracle.homography_table
    for i, r in enumerate(wl.ref_views):
        H = table(wl.cams, r, wl.neighbours(r), wl.n_labels, wl.z_near, wl.z_far)
        lab, S = wl.labels(r)
        want = oracle.cost_volume(wl.cams, wl.views(), wl.sample_bytes, r, wl.neighbours(r), H, wl.n_labels, lab, S,
                                  wl.oob_penalty, combine)
        assert np.array_equal(costs[i].cpu().numpy(), want), (rig, bits, r)
    run.close()


@pytest.mark.parametrize("rig", ["linear", "arc"])
def test_tiles_that_span_many_empty_segments(rig):
    """Label values 0 .. 200000 spread over 16247 pixels: a tile's segments lie further apart than 16 bits."""
    wl = _workload(rig, 8, L=5)
    rng = np.random.default_rng(3)
    for r in wl.ref_views:
        c = wl.cams[r]
        runs = np.sort(rng.choice(200001, (c.width * c.height + 6) // 7, replace=False)).astype(np.int32)
        wl._labels[r] = (np.repeat(runs, 7)[: c.width * c.height].reshape(c.height, c.width).copy(), 200001)
    run = Run(wl)
    costs = run.volumes()
    assert run.check() == 0
    for i, r in enumerate(wl.ref_views):
        assert np.array_equal(costs[i].cpu().numpy(), oracle_runs.volume(wl, r)), (rig, r)
    run.close()


def test_streams_of_different_bit_depth_share_a_batch():
    """11- to 16-bit streams share a batch (one sample format); the 12-bit ones alone have the narrower texels."""
    wls = [_workload("arc", 12), _workload("arc", 16), _workload("arc", 12, W=140)]
    runs = [Run(w) for w in wls]
    for r in runs:
        ftv.ftv_stream_init(r.ctx, r.labels, r.S, 3, 1, ftv.FTV_TM_ALL_YUV)
    outs = [[torch.zeros(S, dtype=torch.int16, device="cuda") for S in r.S] for r in runs]
    batch = ftv.ftv_batch_create(3, 16, 16)
    for group in ([0, 1], [0, 2], [1, 2]):
        jobs = [dict(ctx=runs[k].ctx, planes=runs[k].planes(), frame_type=ftv.FTV_FRAME_I, label_out=outs[k])
                for k in group]
        assert ftv.ftv_batch_prepare(batch, jobs) == ftv.FTV_OK
        ftv.ftv_batch_replay(batch)
        assert ftv.ftv_batch_wait(batch) == ftv.FTV_OK
        for k in group:
            for i, r in enumerate(wls[k].ref_views):
                want = oracle.wta(oracle_runs.volume(wls[k], r))
                assert np.array_equal(outs[k][i].cpu().numpy().view(np.uint16), want), (group, k, r)
    batch.close()
    for r in runs:
        r.close()
