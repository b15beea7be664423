"""Segment lists and plane layouts the preparation kernels take by different routes: lists out of order, with repeats,
invalid and absent entries, against the oracle; planes whose rows start off the vector loads' alignment."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from synth.configs import make_workload

pytestmark = pytest.mark.gpu

ftv = pytest.importorskip("paper_1909_02294_gb300")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import oracle_runs  # noqa: E402
from gpu_runs import Run, dev  # noqa: E402


@pytest.mark.parametrize("kind", ["increasing", "reversed", "repeats", "one_repeated", "invalid", "empty"])
def test_listed_rows_equal_the_oracle(kind):
    wl = make_workload("tiny")
    run = Run(wl)
    S = run.S[0]
    rng = np.random.default_rng(4)
    some = np.sort(rng.choice(S, S // 3, replace=False)).astype(np.int32)
    lst = {"increasing": some, "reversed": some[::-1].copy(), "repeats": np.repeat(some, 3)[:S],
           "one_repeated": np.full(S, some[5], np.int32),
           "invalid": np.where(rng.random(len(some)) < 0.2, rng.choice([-1, S, 1 << 30], len(some)), some).astype(np.int32),
           "empty": some[:0]}[kind]
    d_list = dev(np.concatenate([lst, np.zeros(4, np.int32)]))
    n = torch.tensor([len(lst)], dtype=torch.int32, device="cuda")
    costs = run.volumes(fill=-7, seg_lists=[d_list], n_listed=[n])
    assert run.check() == 0
    want = np.full((S, wl.n_labels), -7, np.int32)
    rows = np.unique(lst[(lst >= 0) & (lst < S)])
    full = oracle_runs.volume(wl, wl.ref_views[0])
    want[rows] = full[rows]
    assert np.array_equal(costs[0].cpu().numpy(), want)
    run.close()


@pytest.mark.parametrize("name", ["tiny", "hd8", "uhd15"])
@pytest.mark.parametrize("offset,extra", [(1, 3), (4, 4), (2, 5)])
def test_plane_offsets_and_pitches(name, offset, extra):
    """hd8: 244 samples a row (a multiple of four), uhd15: 390 (not one), tiny: 8-bit."""
    wl = make_workload(name, reduced=name != "tiny")
    run = Run(wl)
    planes = []
    for trip in run.planes():
        out = []
        for p in trip:
            h, w = p.shape
            buf = torch.zeros(h * (w + extra) + offset, dtype=torch.int16 if p.element_size() == 2 else torch.uint8,
                              device="cuda")
            view = torch.as_strided(buf, (h, w), (w + extra, 1), offset)
            view.copy_(p.view(torch.int16) if p.element_size() == 2 else p)
            out.append(view)
        planes.append(tuple(out))
    got = run.volumes(planes=planes)
    assert run.check() == 0
    for a, b in zip(got, run.volumes()):
        assert torch.equal(a, b)
    run.close()
