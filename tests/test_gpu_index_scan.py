"""Prefix sums over several blocks (the segment index and the edge offsets of the adjacency): segment counts around
one, two and three blocks' share of 8192, against the oracle. Everything is exact but the weights, which are the same
operations in the same order."""
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


@pytest.mark.parametrize("S", [8191, 8192, 8193, 16384, 16385, 24577])
def test_offsets_of_many_segments(S):
    w, h, L, bits = 307, 97, 2, 8
    rng = np.random.default_rng(S)
    lab = rng.permutation(S)[np.arange(w * h) * S // (w * h)].reshape(h, w).astype(np.int32)  # one to four pixels of a row each
    cams = synth.linear_rig(2, 0.2, 80.0, w, h)
    views = [synth.View(*(rng.integers(0, 256, (h, w)).astype(np.uint8) for _ in range(3))) for _ in cams]
    ctx = ftv.ftv_depth_init(cams, [0], L, 1.0, 6.0, sample_bytes=1, bit_depth=bits, oob_penalty=765, max_segments=S)
    planes = [[dev(a) for a in (v.Y, v.U, v.V)] for v in views]
    cost = torch.full((S, L), -1, dtype=torch.int32, device="cuda")
    ftv.ftv_cost_volume(ctx, planes, [dev(lab)], [S], [cost])
    assert ftv.ftv_check(ctx) == 0
    H = oracle.homography_table(cams, 0, [1], L, 1.0, 6.0)
    assert np.array_equal(cost.cpu().numpy(), oracle.cost_volume(cams, views, 1, 0, [1], H, L, lab, S, 765))
    es_r, et_r, b_r = oracle.adjacency(lab, S, views[0], 1, 4, beta0=2.0, min_diff=0.5)
    n = len(es_r)
    es, et = (torch.full((n,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    beta, count = torch.zeros(n, dtype=torch.float32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    ftv.ftv_adjacency(ctx, 0, planes[0], dev(lab), S, 4, 2.0, 0.5, es, et, beta, count)
    assert ftv.ftv_check(ctx) == 0 and int(count.item()) == n
    assert np.array_equal(es.cpu().numpy(), es_r) and np.array_equal(et.cpu().numpy(), et_r)
    assert np.array_equal(beta.cpu().numpy().view(np.uint32), b_r.view(np.uint32))
