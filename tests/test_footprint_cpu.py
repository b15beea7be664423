"""ftv_job_footprint decides from few labels whether a rig has affine homographies (which sets the size of the cost
kernel's texels); here it is compared with the whole tables. The affine and the projective answer differ by four bytes
per padded view pixel for 10-bit samples."""
from __future__ import annotations

import copy

import numpy as np
import pytest

import synth

W, H, L = 64, 40, 9


@pytest.fixture(scope="module")
def ftv():
    return pytest.importorskip("paper_1909_02294_gb300")


def _bytes(ftv, cams, lists=None, mode=0, centre=0):
    import ctypes
    cfg, keep = ftv.ftv._config(cams, list(range(len(lists or cams))), L, 1.0, 8.0, lists, mode, centre, 2, 10, -1,
                                ftv.FTV_COMBINE_MIN, 40)
    n = ctypes.c_int64()
    assert ftv.ftv.lib.ftv_job_footprint(ctypes.byref(cfg), 0, ctypes.byref(n)) == 0
    return n.value


def _cancelling(z):
    """A reference, its neighbour and a centre camera, tilted alike: the third row of the pair's homography vanishes at
    the label of depth z and at no other."""
    K = synth.intrinsics(64.0, W, H)
    tilt = np.array([[1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.25, 0.5, 1.0]])
    return [synth.Camera(K.copy(), R.copy(), np.array([0.0, 0.0, t]), W, H) for R, t in ((np.eye(3), 0.0), (tilt, -z), (tilt, 0.0))]


def _rigs():
    lin = synth.linear_rig(3, 0.1, 64.0, W, H)
    arc = synth.arc_rig(3, 3.0, 8.0, 64.0, W, H, seed=1, roll_deg=3.0)
    flat = synth.arc_rig(3, 3.0, 8.0, 64.0, W, H, seed=1, roll_deg=0.0)
    mixed = copy.deepcopy(arc)
    mixed.append(synth.Camera(arc[0].K.copy(), arc[0].R.copy(), arc[0].t + np.array([0.05, 0.0, 0.2]), W, H))
    return {"linear": lin, "arc": arc, "arc without rolls": flat, "mixed": mixed}


@pytest.mark.parametrize("name", list(_rigs()))
@pytest.mark.parametrize("centre", [None, 0, 1])
def test_same_as_the_whole_table(ftv, name, centre):
    cams = _rigs()[name]
    _check(ftv, cams, centre)


@pytest.mark.parametrize("z", [1.0, 8.0, 3.0])
def test_affine_at_one_label_only(ftv, z):
    cams = _cancelling(z)
    t = ftv.ftv_compute_homographies(cams, [0], 0, L, 1.0, 8.0, nbr_lists=[[1]], plane_mode=ftv.FTV_PLANES_CENTRE, centre_view=2)
    assert int(((t[0, :, 6] == 0) & (t[0, :, 7] == 0)).sum()) == (1 if z in (1.0, 8.0) else 0)
    _check(ftv, cams, 2, [[1]])


def _check(ftv, cams, centre, lists=None):
    mode = ftv.FTV_PLANES_REF if centre is None else ftv.FTV_PLANES_CENTRE
    refs = list(range(len(lists or cams)))
    tables = [ftv.ftv_compute_homographies(cams, refs, r, L, 1.0, 8.0, nbr_lists=lists, plane_mode=mode, centre_view=centre or 0)
              for r in refs]
    affine = any(np.any((t[..., 6] == 0) & (t[..., 7] == 0)) for t in tables)
    base = _bytes(ftv, synth.linear_rig(len(cams), 0.1, 64.0, W, H), lists)
    pad = lambda b: (b + 255) & ~255
    wide = 0 if affine else len(cams) * (pad(W * H * 8) - pad(W * H * 4))
    assert _bytes(ftv, cams, lists, mode, centre or 0) == base + wide


def test_context_without_neighbours_takes_the_smaller_texels(ftv):
    arc = synth.arc_rig(3, 3.0, 8.0, 64.0, W, H, seed=1)
    lin = synth.linear_rig(3, 0.1, 64.0, W, H)
    assert _bytes(ftv, arc, [[], [], []]) == _bytes(ftv, lin, [[], [], []])
