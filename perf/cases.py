"""The work this library's users have it do, as cases that can be timed and compared.

A case is a dict of plain values. Its "kind" is one of
  volume       cost volume of every reference from fresh label maps, then the winner-take-all readout with
               depth maps: an I-type depth frame through the direct entry points
  p_frame      temporal test of every reference, cost volume of the changed segments from the cached index,
               readout with adoption: a P-type depth frame through the direct entry points
  temporal     the temporal test of every reference of a rig alone
  gop          an I frame and a P frame of several camera streams through the batched, graph-replayed form
  superpixels  the segmentation that produces the label maps
  centre       the centre table (matching cost and correspondence at segment centres)
  adjacency    adjacent segment pairs and smoothing weights of every reference
The sizes are those of the repository's workloads (480x270 to 3840x2160, 3 to 15 views, 64 to 400 labels, 10
to 16 px segments), with odd and ragged ones between them. Scenes are textured planes rendered on the GPU by
ray casting, with sensor noise; label maps are the Voronoi cells of a jittered grid, like superpixels.
"""
import math

import numpy as np
import torch

import paper_1909_02294_gb300 as ftv

DEV = "cuda"


def listed():
    return [
        # one small 8-bit frame, one reference: the latency of a call
        dict(name="volume_270p_8bit", kind="volume", rig="linear", views=3, refs=1, nearest=0, w=480, h=270, labels=64,
             cell=16, bits=8, combine="min", precision=32),
        # 12-bit samples, ragged size, the two nearest views, summed: the wide texel format and the other combination
        dict(name="volume_541_12bit_sum", kind="volume", rig="arc", views=5, refs=5, nearest=2, w=957, h=541, labels=100,
             cell=9, bits=12, combine="sum", precision=32),
        # the rectified rig of the broadcast sequences: all views are references
        dict(name="volume_1080p_linear", kind="volume", rig="linear", views=8, refs=8, nearest=0, w=1920, h=1080,
             labels=250, cell=10, bits=10, combine="min", precision=32),
        # the largest: a convergent arc at 4K, the default benchmark's shape
        dict(name="volume_2160p_arc", kind="volume", rig="arc", views=15, refs=15, nearest=0, w=3840, h=2160, labels=400,
             cell=13, bits=10, combine="min", precision=32),
        # sample positions in double precision on a convergent arc of odd size
        dict(name="volume_545_arc_fp64", kind="volume", rig="arc", views=7, refs=3, nearest=0, w=975, h=545, labels=100,
             cell=11, bits=10, combine="min", precision=64),
        # the everyday frame of a small stream: most segments adopt, a few are estimated
        dict(name="p_frame_540p", kind="p_frame", rig="linear", views=3, refs=3, nearest=0, w=960, h=540, labels=64,
             cell=10, bits=10, combine="min", precision=32),
        # the per-frame test of a whole rig, against the previous and the I frame
        dict(name="temporal_1080p", kind="temporal", rig="linear", views=8, refs=8, w=1920, h=1080, cell=10, bits=10,
             yuv=True, iframe=True),
        # four small camera streams served together
        dict(name="gop_540p_streams", kind="gop", streams=4, views=3, w=960, h=540, labels=64, cell=10, bits=10),
        # segmentation of one small 8-bit image, and of every view of a 1080p rig
        dict(name="superpixels_270p_8bit", kind="superpixels", images=1, w=480, h=270, bits=8, step=16, iters=10),
        dict(name="superpixels_1080p", kind="superpixels", images=8, w=1920, h=1080, bits=10, step=10, iters=10),
        # what a graph-cut consumer reads: the paper's 3x3 window at every segment centre of the 1080p rig
        dict(name="centre_1080p", kind="centre", rig="linear", views=8, refs=8, nearest=0, w=1920, h=1080, labels=250,
             cell=10, bits=10, window=3),
        # and its smoothing weights
        dict(name="adjacency_1080p", kind="adjacency", views=8, w=1920, h=1080, cell=10, bits=10, conn=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["volume", "volume", "volume", "p_frame", "temporal", "gop", "superpixels", "superpixels", "centre",
                       "adjacency"])
    w = _log(rng, 240, 2600)
    h = max(96, int(w * rng.uniform(0.5, 0.75)))
    cell = rng.randint(8, 18)
    bits = rng.choice([8, 10, 10, 12])
    rig = rng.choice(["linear", "arc"])
    views = rng.randint(2, 10)
    if kind == "volume":
        nearest = rng.choice([0, 0, 2]) if views > 3 else 0
        labels = _log(rng, 32, 400)
        refs = rng.randint(1, views)
        precision = rng.choice([32, 32, 32, 64])
        n = (nearest or views - 1) * refs
        while w * h * labels * n > 3e10 / (1 if precision == 32 else 2):  # well below the largest listed case
            w, h = w * 3 // 4, h * 3 // 4
        return dict(kind=kind, rig=rig, views=views, refs=refs, nearest=nearest, w=w, h=h, labels=labels, cell=cell,
                    bits=bits, combine=rng.choice(["min", "min", "sum"]), precision=precision)
    if kind == "p_frame":
        labels = _log(rng, 32, 250)
        while w * h * labels * views * (views - 1) > 3e10:
            w, h = w * 3 // 4, h * 3 // 4
        return dict(kind=kind, rig=rig, views=views, refs=views, nearest=0, w=w, h=h, labels=labels, cell=cell, bits=bits,
                    combine="min", precision=32)
    if kind == "temporal":
        return dict(kind=kind, rig=rig, views=views, refs=views, w=w, h=h, cell=cell, bits=bits, yuv=rng.random() < 0.7,
                    iframe=rng.random() < 0.7)
    if kind == "gop":
        w, h = min(w, 1280), min(h, 720)
        return dict(kind=kind, streams=rng.randint(1, 4), views=rng.randint(2, 4), w=w, h=h, labels=_log(rng, 32, 128),
                    cell=cell, bits=rng.choice([8, 10]))
    if kind == "superpixels":
        return dict(kind=kind, images=rng.randint(1, 8), w=w, h=h, bits=bits, step=rng.randint(8, 32),
                    iters=rng.choice([5, 10]))
    if kind == "centre":
        labels = _log(rng, 32, 250)
        while (w // cell + 1) * (h // cell + 1) * labels * views * (views - 1) > 3e8:
            w, h = w * 3 // 4, h * 3 // 4
        return dict(kind=kind, rig=rig, views=views, refs=views, nearest=0, w=w, h=h, labels=labels, cell=cell, bits=bits,
                    window=rng.choice([3, 3, 5]))
    return dict(kind=kind, views=rng.randint(1, 8), w=w, h=h, cell=cell, bits=bits, conn=rng.choice([4, 8]))


# ------------------------------------------------------------------------------------------------ inputs

class Camera:
    def __init__(self, K, R, t, w, h):
        self.K, self.R, self.t, self.width, self.height = K, R, t, w, h


def _intrinsics(f, w, h):
    return np.array([[f, 0.0, (w - 1) / 2.0], [0.0, f, (h - 1) / 2.0], [0.0, 0.0, 1.0]])


def _rig(rig, n, w, h, rng):
    f = w / 1.28  # 1500 px at 1920
    cams = []
    for i in range(n):
        if rig == "linear":  # parallel cameras 10 cm apart
            R, C, fi = np.eye(3), np.array([(i - (n - 1) / 2.0) * 0.10, 0.0, 0.0]), f
        else:  # a convergent arc of radius 3 m, 8 degrees apart, small rolls and focal spread
            th = math.radians((i - (n - 1) / 2.0) * 8.0)
            C = np.array([3.0 * math.sin(th), 0.0, -3.0 * math.cos(th)])
            fwd = -C / 3.0
            right = np.array([math.cos(th), 0.0, math.sin(th)])
            a = math.radians(rng.uniform(-2.0, 2.0))
            roll = np.array([[math.cos(a), -math.sin(a), 0.0], [math.sin(a), math.cos(a), 0.0], [0.0, 0.0, 1.0]])
            R, fi = roll @ np.stack([right, np.cross(fwd, right), fwd]), f * (1.0 + rng.uniform(-0.03, 0.03))
        cams.append(Camera(_intrinsics(fi, w, h), R, -R @ C, w, h))
    return cams


def _planes(ref, w, h, zmin, zmax, rng):
    """A background plane and a few bounded ones in front of it, parallel to `ref`'s image plane or slanted:
    (point, two edge vectors, half size or 0, texel size, texture number)."""
    f = ref.K[0, 0]
    Rt, C = ref.R.T, -ref.R.T @ ref.t
    out = [(C + Rt @ np.array([0.0, 0.0, zmax]), Rt[:, 0], Rt[:, 1], 0.0, 6.0 * zmax / f, 0)]
    for k in range(1, 8):
        z = math.exp(rng.uniform(math.log(zmin), math.log(0.7 * zmax)))
        p = np.array([rng.uniform(-0.4, 0.4) * w / f * z, rng.uniform(-0.4, 0.4) * h / f * z, z])
        a = math.radians(rng.uniform(0.0, 35.0)) if k % 2 else 0.0
        e1 = np.array([math.cos(a), 0.0, math.sin(a)])
        out.append((C + Rt @ p, Rt @ e1, Rt[:, 1], rng.uniform(0.05, 0.12) * w / f * z, rng.uniform(3.0, 9.0) * z / f, k))
    return out


def _render(cam, planes, textures, bits, noise, gen, shift=0.0):
    """(Y, Cb, Cr) of one view: nearest plane per pixel, bilinear texture, rounded noise. shift moves the
    bounded planes along their first edge (metres), for the frames of a sequence."""
    w, h = cam.width, cam.height
    y, x = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float32),
                          torch.arange(w, device=DEV, dtype=torch.float32), indexing="ij")
    Ki = np.linalg.inv(cam.K)
    D = cam.R.T @ Ki
    C = -cam.R.T @ cam.t
    d = [D[i, 0] * x + D[i, 1] * y + D[i, 2] for i in range(3)]
    best = torch.full((h, w), 1e9, device=DEV)
    U, V = torch.zeros((h, w), device=DEV), torch.zeros((h, w), device=DEV)
    T = torch.zeros((h, w), device=DEV, dtype=torch.int64)
    for p0, e1, e2, half, texel, k in planes:
        p0 = p0 + (shift * e1 if half > 0 else 0.0)
        n = np.cross(e1, e2)
        s = float(n @ (p0 - C)) / (n[0] * d[0] + n[1] * d[1] + n[2] * d[2])
        q = [C[i] - p0[i] + s * d[i] for i in range(3)]
        u = e1[0] * q[0] + e1[1] * q[1] + e1[2] * q[2]
        v = e2[0] * q[0] + e2[1] * q[1] + e2[2] * q[2]
        hit = (s > 0.05) & (s < best)
        if half > 0:
            hit &= (u.abs() < half) & (v.abs() < half)
        best = torch.where(hit, s, best)
        U, V = torch.where(hit, u / texel, U), torch.where(hit, v / texel, V)
        T = torch.where(hit, torch.full_like(T, k), T)
    i, j = torch.floor(U), torch.floor(V)
    fu, fv = U - i, V - j
    i, j = i.to(torch.int64), j.to(torch.int64)
    n = textures.shape[-1]
    vmax = (1 << bits) - 1
    dtype = torch.uint8 if bits <= 8 else torch.int16
    out = []
    for c in range(3):
        t = textures[c]
        a, b = t[T, j % n, i % n], t[T, j % n, (i + 1) % n]
        e, g = t[T, (j + 1) % n, i % n], t[T, (j + 1) % n, (i + 1) % n]
        v = ((a * (1 - fu) + b * fu) * (1 - fv) + (e * (1 - fu) + g * fu) * fv) * vmax
        v = v + noise * torch.randn(v.shape, device=DEV, generator=gen)
        out.append(v.round().clamp_(0, vmax).to(dtype).contiguous())
    return tuple(out)


def _label_map(w, h, cell, gen):
    """Voronoi cells of a jittered grid: (int32 [h][w], number of segments)."""
    gw, gh = -(-w // cell), -(-h // cell)
    sx = (torch.arange(gw, device=DEV).float()[None, :] + 0.5 + 0.7 * (torch.rand((gh, gw), device=DEV, generator=gen) - 0.5))
    sy = (torch.arange(gh, device=DEV).float()[:, None] + 0.5 + 0.7 * (torch.rand((gh, gw), device=DEV, generator=gen) - 0.5))
    y, x = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    best = torch.full((h, w), 1e9, device=DEV)
    lab = torch.zeros((h, w), device=DEV, dtype=torch.int64)
    for dy in (-1, 0, 1):
        for dx in (-1, 0, 1):
            ci, cj = (x // cell + dx).clamp(0, gw - 1), (y // cell + dy).clamp(0, gh - 1)
            k = cj * gw + ci
            d = (sx.reshape(-1)[k] * cell - x - 0.5) ** 2 + (sy.reshape(-1)[k] * cell - y - 0.5) ** 2
            lab = torch.where(d < best, k, lab)
            best = torch.minimum(d, best)
    return lab.to(torch.int32).contiguous(), gw * gh


class Scene:
    """Cameras, frames and label maps of one rig, from a seed."""

    def __init__(self, case, seed, frames=1):
        w, h, n = case["w"], case["h"], case["views"]
        rng = np.random.default_rng(seed)
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed))
        arc = case.get("rig", "linear") == "arc"
        self.cams = _rig(case.get("rig", "linear"), n, w, h, rng)
        self.z_near, self.z_far = (0.8, 15.0) if arc else (1.0, 20.0)
        mid = self.cams[n // 2]
        planes = _planes(mid, w, h, 1.6, 12.0 if arc else 18.0, rng)
        textures = torch.rand((3, 8, 256, 256), device=DEV, generator=gen)
        noise = 2.0 * (1 << case["bits"]) / 1024.0
        step = 4.0 * 2.5 / mid.K[0, 0]  # the bounded planes move about 4 px a frame
        self.frames = [[_render(c, planes, textures, case["bits"], noise, gen, k * step) for c in self.cams]
                       for k in range(frames)]
        self.labels, self.segments = [], []
        for _ in range(n if "cell" in case else 0):
            lab, s = _label_map(w, h, case["cell"], gen)
            self.labels.append(lab)
            self.segments.append(s)


def _refs(case):
    """The reference views (the first ones from the centre outwards) and their neighbour lists."""
    n = case["views"]
    order = sorted(range(n), key=lambda v: (abs(v - n // 2), v))
    refs = sorted(order[: case["refs"]])
    nbrs = None
    if case.get("nearest"):
        nbrs = [sorted(sorted((v for v in range(n) if v != r), key=lambda v: (abs(v - r), v))[: case["nearest"]])
                for r in refs]
    return refs, nbrs


def _context(case, sc, refs, nbrs):
    return ftv.ftv_depth_init(
        sc.cams, refs, case.get("labels", 2), sc.z_near, sc.z_far, nbr_lists=nbrs,
        sample_bytes=1 if case["bits"] <= 8 else 2, bit_depth=case["bits"],
        combine=ftv.FTV_COMBINE_SUM if case.get("combine") == "sum" else ftv.FTV_COMBINE_MIN,
        max_segments=max(sc.segments),
        precision=ftv.FTV_PRECISION_FP64 if case.get("precision") == 64 else ftv.FTV_PRECISION_FP32)


def _empty(shape, dtype=torch.int32):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def prepare(case, seed):
    s = {"case": case}
    kind = case["kind"]
    if kind == "gop":
        scenes = [Scene(case, 1000 * seed + 17 * k, frames=2) for k in range(case["streams"])]
        refs = list(range(case["views"]))
        s["ctx"] = [_context(case, sc, refs, None) for sc in scenes]
        for ctx, sc in zip(s["ctx"], scenes):
            ftv.ftv_stream_init(ctx, sc.labels, sc.segments, 3 << (case["bits"] - 8), 1 << (case["bits"] - 8),
                                ftv.FTV_TM_ALL_YUV)
        n = case["streams"] * case["views"]
        s["batch"] = ftv.ftv_batch_create(case["streams"], n, n)
        s["win"] = [[[_empty(S, torch.int16) for S in sc.segments] for sc in scenes] for _ in range(2)]
        s["depth"] = [[[_empty((case["h"], case["w"]), torch.float32) for _ in refs] for _ in scenes] for _ in range(2)]
        s["jobs"] = [[dict(ctx=c, planes=sc.frames[k], frame_type=(ftv.FTV_FRAME_I, ftv.FTV_FRAME_P)[k],
                           label_out=s["win"][k][i], depth_out=s["depth"][k][i])
                      for i, (c, sc) in enumerate(zip(s["ctx"], scenes))] for k in range(2)]
        s["scenes"] = scenes
        return s
    if kind == "superpixels":
        sc = Scene(dict(case, views=case["images"]), seed)
        s["seg"] = ftv.ftv_segmenter_init([(case["w"], case["h"])] * case["images"], 1 if case["bits"] <= 8 else 2,
                                          case["bits"], case["step"], 5, case["iters"])
        s["planes"] = sc.frames[0]
        s["labels"] = [_empty((case["h"], case["w"])) for _ in range(case["images"])]
        return s
    if kind == "adjacency":
        case = dict(case, refs=case["views"], rig="linear")
    refs, nbrs = _refs(case)
    sc = Scene(case, seed, frames=3 if kind in ("p_frame", "temporal") else 1)
    L = case.get("labels", 2)
    if kind in ("temporal", "adjacency"):  # neither reads the neighbours
        nbrs = [[] for _ in refs]
    s["refs"], s["scene"], s["nbrs"] = refs, sc, nbrs
    s["ctx"] = _context(case, sc, refs, nbrs)
    s["labels"] = [sc.labels[r] for r in refs]
    s["nseg"] = [sc.segments[r] for r in refs]
    if kind in ("volume", "p_frame"):
        s["cost"] = [_empty((S, L)) for S in s["nseg"]]
        s["win"] = [_empty(S, torch.int16) for S in s["nseg"]]
        s["depth"] = [_empty((case["h"], case["w"]), torch.float32) for _ in refs]
    if kind in ("temporal", "p_frame"):
        s["mask"] = [_empty(S, torch.uint8) for S in s["nseg"]]
        s["list"] = [_empty(S) for S in s["nseg"]]
        s["count"] = [_empty(1) for _ in refs]
    if kind == "p_frame":  # the stream so far: its index, and the labels of the previous and the I frame
        for i in range(len(refs)):
            ftv.ftv_segment_index(s["ctx"], i, s["labels"][i], s["nseg"][i])
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 5)
        s["prev"] = [torch.randint(0, L, (S,), device=DEV, generator=gen).to(torch.int16) for S in s["nseg"]]
        s["ifr"] = [torch.randint(0, L, (S,), device=DEV, generator=gen).to(torch.int16) for S in s["nseg"]]
    if kind == "centre":
        n = [len(nbrs[i]) if nbrs else case["views"] - 1 for i in range(len(refs))]
        s["m"] = [_empty((S, L, k)) for S, k in zip(s["nseg"], n)]
        s["sp"] = [_empty((S, L, k)) for S, k in zip(s["nseg"], n)]
    if kind == "adjacency":
        cap = [8 * S for S in s["nseg"]]
        s["es"], s["et"] = [_empty(c) for c in cap], [_empty(c) for c in cap]
        s["beta"] = [_empty(c, torch.float32) for c in cap]
        s["count"] = [_empty(1) for _ in refs]
    return s


def _temporal(s, frames, iframe, t, mode):
    cur, prev = [frames[2][r] for r in s["refs"]], [frames[1][r] for r in s["refs"]]
    ifr = [frames[0][r] for r in s["refs"]] if iframe else None
    ftv.ftv_temporal_mask_views(s["ctx"], list(range(len(s["refs"]))), cur, prev, ifr, s["labels"], s["nseg"], 3 * t, t,
                                mode, s["mask"], s["list"], s["count"])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "volume":
        ftv.ftv_cost_volume(s["ctx"], s["scene"].frames[0], s["labels"], s["nseg"], s["cost"])
        for i in range(len(s["refs"])):
            ftv.ftv_wta_depth(s["ctx"], i, s["cost"][i], s["nseg"][i], s["win"][i], labels_pix=s["labels"][i],
                              depth_map=s["depth"][i])
        return {"cost": s["cost"], "win": s["win"], "depth": s["depth"]}
    if kind == "p_frame":
        frames = s["scene"].frames
        _temporal(s, frames, True, 1 << (case["bits"] - 8), ftv.FTV_TM_ALL_YUV)
        ftv.ftv_cost_volume(s["ctx"], frames[2], None, None, s["cost"], s["list"], s["count"])
        for i in range(len(s["refs"])):
            ftv.ftv_wta_depth(s["ctx"], i, s["cost"][i], s["nseg"][i], s["win"][i], mask=s["mask"][i],
                              prev_label=s["prev"][i], iframe_label=s["ifr"][i], labels_pix=s["labels"][i],
                              depth_map=s["depth"][i])
        return {k: s[k] for k in ("mask", "list", "count", "cost", "win", "depth")}
    if kind == "temporal":
        _temporal(s, s["scene"].frames, case["iframe"], 1 << (case["bits"] - 8),
                  ftv.FTV_TM_ALL_YUV if case["yuv"] else ftv.FTV_TM_Y_ONLY)
        return {k: s[k] for k in ("mask", "list", "count")}
    if kind == "gop":
        for jobs in s["jobs"]:
            if ftv.ftv_batch_prepare(s["batch"], jobs) != ftv.FTV_OK:
                raise RuntimeError("the batch was not prepared")
            ftv.ftv_batch_replay(s["batch"])
            if ftv.ftv_batch_wait(s["batch"]) != ftv.FTV_OK:  # a stream has one frame in flight
                raise RuntimeError("a job of the batch failed")
        return {"win": s["win"], "depth": s["depth"]}
    if kind == "superpixels":
        ftv.ftv_superpixels(s["seg"], s["planes"], s["labels"])
        return s["labels"]
    if kind == "centre":
        ftv.ftv_centre_table(s["ctx"], s["scene"].frames[0], s["scene"].labels, s["nseg"], case["window"], s["m"], s["sp"])
        return {"m": s["m"], "sp": s["sp"]}
    for i, r in enumerate(s["refs"]):
        ftv.ftv_adjacency(s["ctx"], i, s["scene"].frames[0][r], s["labels"][i], s["nseg"][i], case["conn"], 1.0,
                          1.0 / 64, s["es"][i], s["et"][i], s["beta"][i], s["count"][i])
    return {"s": s["es"], "t": s["et"], "beta": s["beta"], "count": s["count"]}


# ------------------------------------------------------------------------------------------------- work

def work(case):
    kind, px = case["kind"], case["w"] * case["h"]
    frame = 3 * px * (1 if case["bits"] <= 8 else 2)
    segs = -(-case["w"] // case["cell"]) * -(-case["h"] // case["cell"]) if "cell" in case else 0
    if kind == "superpixels":  # colours in, labels out; nine candidates of 18 operations per pixel and pass
        return {"bytes": case["images"] * (frame + 4 * px), "flops": case["images"] * px * case["iters"] * 162}
    if kind == "temporal":
        return {"bytes": case["refs"] * ((3 if case["iframe"] else 2) * frame * (3 if case["yuv"] else 1) // 3 + 4 * px +
                                         5 * segs),
                "flops": case["refs"] * px * (3 if case["yuv"] else 1) * (4 if case["iframe"] else 2)}
    if kind == "adjacency":
        return {"bytes": case["views"] * (frame + 4 * px + 3 * segs * 12), "flops": case["views"] * px * (3 + case["conn"])}
    if kind == "gop":  # an I frame and a P frame of which about a fifth is estimated
        v = case["views"]
        return {"bytes": case["streams"] * 2 * v * (frame + 8 * px + 2 * segs),
                "flops": case["streams"] * v * (v - 1) * px * case["labels"] * 9 * 1.2}
    n = case["refs"] * (case.get("nearest") or case["views"] - 1)
    per = 9 + (16 if case["rig"] == "arc" else 0)  # three differences, their sum and the minimum; the projection
    if kind == "centre":
        e = segs * case["labels"] * n
        return {"bytes": case["views"] * (frame + 4 * px) + 8 * e, "flops": e * (case["window"] ** 2 * 9 + 16)}
    if kind == "p_frame":
        return {"bytes": case["views"] * 3 * frame + case["refs"] * (8 * px + segs * 12 + segs * case["labels"]),
                "flops": n * px * case["labels"] * per * 0.2}
    return {"bytes": case["views"] * frame + case["refs"] * (8 * px + segs * (4 * case["labels"] + 2)),
            "flops": n * px * case["labels"] * per}


# ------------------------------------------------------------------------------------------------ exact

def _exact_depth(case, seed):
    """Depth maps of a volume case: every step of the estimator in 64 bits."""
    refs, nbrs = _refs(case)
    sc = Scene(case, seed)
    L, w, h = case["labels"], case["w"], case["h"]
    a, b = 1.0 / sc.z_far, 1.0 / sc.z_near
    iz = [a + d * ((b - a) / (L - 1)) for d in range(L)]
    y, x = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float64),
                          torch.arange(w, device=DEV, dtype=torch.float64), indexing="ij")
    penalty = 3 * ((1 << case["bits"]) - 1)
    frames = [torch.stack([p.to(torch.int32) for p in f]) for f in sc.frames[0]]
    out = []
    for i, r in enumerate(refs):
        cr, S = sc.cams[r], sc.segments[r]
        lab = sc.labels[r].long().reshape(-1)
        cost = torch.empty((L, S), dtype=torch.int64, device=DEV)
        for d in range(L):
            acc = None
            for v in (nbrs[i] if nbrs else [v for v in range(case["views"]) if v != r]):
                cv = sc.cams[v]
                A = cv.R @ cr.R.T
                M = A + np.outer(cv.t - A @ cr.t, [0.0, 0.0, 1.0]) * iz[d]
                H = cv.K @ M @ np.linalg.inv(cr.K)
                W = H[2, 0] * x + H[2, 1] * y + H[2, 2]
                u = torch.floor((H[0, 0] * x + H[0, 1] * y + H[0, 2]) / W + 0.5)
                t = torch.floor((H[1, 0] * x + H[1, 1] * y + H[1, 2]) / W + 0.5)
                ok = (W > 0) & (u >= 0) & (u < w) & (t >= 0) & (t < h)
                q = (torch.where(ok, t, 0.0) * w + torch.where(ok, u, 0.0)).long().reshape(-1)
                c = (frames[v].reshape(3, -1)[:, q] - frames[r].reshape(3, -1)).abs().sum(0)
                c = torch.where(ok.reshape(-1), c, penalty)
                acc = c if acc is None else (acc + c if case["combine"] == "sum" else torch.minimum(acc, c))
            cost[d] = torch.zeros(S, dtype=torch.int64, device=DEV).index_add_(0, lab, acc.long())
        win = (cost * L + torch.arange(L, device=DEV)[:, None]).min(0).values % L  # the smallest label on ties
        z = torch.tensor([1.0 / v for v in iz], dtype=torch.float64, device=DEV)
        out.append(z[win][lab].reshape(h, w))
    k = len(refs)
    return {"cost": [None] * k, "win": [None] * k, "depth": out}


def _exact_adjacency(case, seed):
    sc = Scene(dict(case, rig="linear"), seed)
    out = {"s": [], "t": [], "beta": [], "count": []}
    for r in range(case["views"]):
        lab, S = sc.labels[r].long(), sc.segments[r]
        pairs = [(lab[:, :-1], lab[:, 1:]), (lab[:-1], lab[1:])]
        if case["conn"] == 8:
            pairs += [(lab[:-1, :-1], lab[1:, 1:]), (lab[:-1, 1:], lab[1:, :-1])]
        keys = torch.cat([(torch.minimum(p, q) * S + torch.maximum(p, q))[p != q] for p, q in pairs])
        keys = torch.unique(keys)
        es, et = keys // S, keys % S
        n = torch.bincount(lab.reshape(-1), minlength=S).double()
        dist = torch.zeros(len(keys), dtype=torch.float64, device=DEV)
        for c in range(3):
            m = torch.zeros(S, dtype=torch.float64, device=DEV).index_add_(0, lab.reshape(-1),
                                                                           sc.frames[0][r][c].reshape(-1).double()) / n
            dist += (m[es] - m[et]).abs()
        beta = torch.zeros(8 * S, dtype=torch.float64, device=DEV)
        beta[: len(keys)] = 1.0 / dist.clamp(min=1.0 / 64)
        out["s"].append(None), out["t"].append(None), out["count"].append(None)
        out["beta"].append(beta)
    return out


def exact(case, seed):
    """Whole outputs (costs, labels, masks, tables, label maps) are compared as they are; depth maps and smoothing
    weights are computed here in 64 bits where that takes seconds."""
    if case["kind"] == "adjacency":
        return _exact_adjacency(case, seed)
    if case["kind"] == "volume":
        n = case["refs"] * (case["nearest"] or case["views"] - 1)
        if case["w"] * case["h"] * case["labels"] * n < 3e9:
            return _exact_depth(case, seed)
    return None
