"""Performance cases of the stereo frontend: what users of the library have it do.

Each case is one call sequence through the public Python binding: one stereo
pair at a time from a camera (plain calls or replays of a captured graph),
batches of many streams resident on the device, batches from pinned host
memory, the learned cell-skip mode, the optional readings, and the sub-pixel
refinement.  Sizes, depths, thresholds and feature counts are those of the
workloads in ``scenes`` and of the tests; images are seeded synthetic scenes
of the same kinds with fresh sensor noise per frame.

Outputs are the result blocks (keypoints, descriptors, matches), on the host
where the call downloads them and in the library's device buffers otherwise,
and the floating outputs of the modes that have some.
"""
import ctypes
import json
import os

import numpy as np
import torch

from paper_2410_04090_gb300 import jslam, scenes

_PACKAGE = os.path.dirname(os.path.abspath(jslam.__file__))
_BF = 386.1448  # fx * baseline of a KITTI-like rig (pixels x metres)
_BORDER = 19    # evaluation border of the default configuration
_DEFAULTS = dict(scale=1.2, thresh=20, lo=7, cell=32, p_min=9, p_max=13, k=1, q=3, rule=0, arc=0, cascade=0)


def _case(name, kind, scene, width, height, levels, feats, pairs=1, **options):
    return dict(dict(_DEFAULTS, name=name, kind=kind, scene=scene, width=width, height=height, levels=levels,
                     feats=feats, pairs=pairs), **options)


def listed():
    return [
        # one small camera, one pair per call, results on the host: latency
        _case("pair_320x240_L4", "pair", "planes", 320, 240, 4, 400),
        # one pair through the whole middle-end of a SLAM step: extraction,
        # matching, refinement, tracking of the last frame's keypoints
        _case("step_1241x376_L8", "step", "planes", 1241, 376, 8, 2000),
        # the largest camera of the workloads, one pair per call
        _case("pair_1920x1080_L8", "pair", "planes", 1920, 1080, 8, 3000),
        # a camera stream replayed through a captured graph, new frames each call
        _case("graph_752x480_L8", "graph", "euroc", 752, 480, 8, 1200),
        # many small single-level cameras at once
        _case("batch_640x480_L1", "batch", "checker", 640, 480, 1, 300, 100, lo=0),
        # the headline sequence: 100 frames in one call
        _case("batch_1241x376_L8", "batch", "planes", 1241, 376, 8, 2000, 100),
        # 16 concurrent streams of four sizes and depths
        _case("mixed16", "mixed", "mixed", 1920, 1080, 8, 3000, 16),
        # three keypoints per cell, arc response, wider NMS, lexicographic
        # rule, odd size and another scale factor
        _case("options_647x363_k3", "batch", "planes", 647, 363, 5, 1500, 24, scale=1.3, thresh=15, cell=24, k=3, q=5,
              rule=1, arc=1),
        # other run bounds (the general ring test) on a cascaded pyramid
        _case("bounds_800x602_cascade", "batch", "euroc", 800, 602, 6, 1200, 16, p_min=10, p_max=14, cascade=1),
        # the learned cell-skip proposal with its logits
        _case("skip_752x480_L8", "skip", "euroc", 752, 480, 8, 1200, 12),
        # sub-pixel refinement of a matched batch
        _case("refine_1241x376", "refine", "planes", 1241, 376, 8, 2000, 20),
        # frames that come from, and results that go to, pinned host memory
        _case("host_1241x376_L8", "host", "planes", 1241, 376, 8, 2000, 25),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["pair", "step", "graph", "batch", "batch", "batch", "skip", "refine", "host"])
    scene = rng.choice(["planes", "euroc", "checker"])
    width = _log_uniform(rng, 240, 1920)
    height = min(1080, max(180, int(width * rng.uniform(0.3, 0.75))))
    scale = rng.choice([1.2, 1.2, 1.2, 1.25, 1.3, 1.5])
    # every level has to hold the border on both sides and a pixel between
    deepest = 1
    while deepest < 8 and min(width, height) / scale ** deepest >= 2 * _BORDER + 4:
        deepest += 1
    levels = rng.randint(max(1, deepest - 3), deepest)
    feats = _log_uniform(rng, 200, 3000)
    pairs = 1
    if kind in ("batch", "host"):
        most = max(2, int(100 * 1241 * 376 / (width * height)))
        pairs = min(_log_uniform(rng, 2, most), 100 if kind == "batch" else 25)
    elif kind in ("skip", "refine"):
        pairs = rng.randint(2, 12 if kind == "skip" else 20)
    options = dict(scale=scale, thresh=rng.choice([15, 20, 20, 25]), lo=rng.choice([0, 7, 7]),
                   cell=rng.choice([32, 32, 32, 24, 16]))
    if kind == "batch" and rng.random() < 0.4:
        options.update(rng.choice([dict(k=2), dict(k=3, q=5), dict(arc=1), dict(rule=1, q=5), dict(cascade=1),
                                   dict(p_min=10, p_max=14), dict(p_min=9, p_max=16)]))
    if kind == "skip":
        options["cell"] = 32  # the model was trained for these cells
    case = _case("", kind, scene, width, height, levels, feats, pairs, **options)
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs

def _base_pair(scene, width, height, seed):
    if scene == "checker":
        return scenes.checker_pair(width, height, seed, sigma=0.0)
    if scene == "euroc":
        return scenes.euroc_pair(width, height, 0, seed, seed + 1)
    return scenes.planes_pair(width, height, 0, seed, seed + 1, sigma=0.0)


def _frames(scene, width, height, count, seed):
    """`count` stereo frames [count, 2, height, width] u8 on the GPU: one scene
    of the seed seen by a camera that pans (both views by the same columns)
    and turns over on odd frames, with fresh sensor noise (sigma 2)."""
    seed = int(seed) % 1_000_000_007
    pair = _base_pair(scene, width, height, seed)
    base = torch.from_numpy(np.stack([pair.left, pair.right])).cuda().half()
    gen = torch.Generator(device="cuda").manual_seed(seed + 17)
    out = torch.empty((count, 2, height, width), dtype=torch.uint8, device="cuda:0")
    for i in range(count):
        f = torch.roll(base, shifts=(37 * i) % width, dims=2)
        if i & 1:
            f = f.flip(1)
        noise = torch.randn(f.shape, generator=gen, device="cuda", dtype=torch.float16) * 2.0
        out[i] = (f + noise.round_()).clamp_(0, 255).to(torch.uint8)
    return out


def _streams(case):
    """(scene, width, height, levels, feats) of every pair of the case."""
    if case["kind"] == "mixed":
        return [(s["kind"], s["width"], s["height"], s["levels"], s["max_feats"]) for s in scenes.MIXED_STREAMS]
    one = (case["scene"], case["width"], case["height"], case["levels"], case["feats"])
    return [one] * case["pairs"]


def _all_frames(case, seed):
    """Per pair a [2, height, width] u8 CUDA tensor (pairs of one size share one buffer)."""
    streams = _streams(case)
    out, i = [], 0
    while i < len(streams):
        j = i
        while j < len(streams) and streams[j][:3] == streams[i][:3]:
            j += 1
        out.extend(_frames(*streams[i][:3], j - i, seed + 31 * i))
        i = j
    return out


# ------------------------------------------------------------------ state

class _State:
    pass


def _frontend(case, streams, stream=None):
    return jslam.Frontend(device=0, stream=stream, max_width=max(s[1] for s in streams),
                          max_height=max(s[2] for s in streams), max_levels=max(s[3] for s in streams),
                          max_feats=max(s[4] for s in streams), max_pairs=len(streams),
                          fast_thresh_lo=case["lo"], p_min=case["p_min"], p_max=case["p_max"],
                          k_per_cell=case["k"], nms_q=case["q"], pfa_rule=case["rule"],
                          response_mode=case["arc"], pyramid_mode=case["cascade"])


def _args(case, stream):
    return dict(levels=stream[3], scale=case["scale"], fast_thresh=case["thresh"], cell=case["cell"],
                max_feats=stream[4])


def _jobs(case, streams, frames):
    return [jslam.Job(f[0], f[1], **_args(case, s)) for s, f in zip(streams, frames)]


class _DeviceArray:
    """Device memory of a frontend, which lives as long as a tensor made of it."""

    def __init__(self, owner, ptr, shape, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": tuple(shape), "typestr": typestr, "data": (ptr, False), "version": 3}


def _kept(fe, view):
    """`view` (a device view of the frontend's results) as a tensor that keeps the frontend."""
    if view.numel() == 0:
        return view
    kind = {torch.float32: "<f4", torch.uint32: "<u4", torch.uint8: "|u1"}[view.dtype]
    return torch.as_tensor(_DeviceArray(fe, view.data_ptr(), view.shape, kind), device="cuda:0")


def _device_blocks(fe, pairs):
    """The result blocks of all pairs as one device tensor, for a consumer on
    the GPU: their size from result_range, their place from the device
    address of pair 0's descriptors and those descriptors' offset in a block."""
    size, _ = fe.result_range(0, pairs)
    host = np.zeros(fe.result_bytes(0), np.uint8)
    in_block, on_device = jslam.Keypoints(), jslam.Keypoints()
    jslam.lib().jslam_result_view(fe._h, 0, host.ctypes.data, 0, ctypes.byref(in_block), None)
    jslam.lib().jslam_get_keypoints(fe._h, 0, 0, ctypes.byref(on_device))
    base = on_device.desc - (in_block.desc - host.ctypes.data)
    return torch.as_tensor(_DeviceArray(fe, base, (size,), "|u1"), device="cuda:0")


def _skip_model():
    with open(os.path.join(_PACKAGE, "skipnet_v1.bin"), "rb") as f:
        blob = f.read()
    with open(os.path.join(_PACKAGE, "skipnet_v1.json")) as f:
        return blob, json.load(f)["thresh"]


def prepare(case, seed):
    kind, streams = case["kind"], _streams(case)
    s = _State()
    s.kind, s.n, s.args = kind, len(streams), _args(case, streams[0])
    s.frames = _all_frames(case, seed)
    # device-resident batches run on torch's current stream, in order with
    # the rest of a program; the others own a stream and wait for their result
    on = torch.cuda.current_stream() if kind in ("batch", "mixed", "skip", "refine") else None
    s.fe = _frontend(case, streams, on)
    torch.cuda.synchronize()
    if kind == "skip":
        s.fe.set_skip_model(*_skip_model())
    if kind == "host":
        # one pinned buffer for a step's frames: left 0, right 0, left 1, ...
        s.pinned = torch.stack(s.frames).cpu().pin_memory()
        views = s.pinned.numpy()
        s.batch = s.fe.prepare_batch([jslam.Job(v[0], v[1], **s.args) for v in views])
        s.frames = None
    elif kind in ("batch", "mixed", "skip", "refine"):
        s.batch = s.fe.prepare_batch(_jobs(case, streams, s.frames))
    elif kind == "graph":
        # captured on frames of its own; the calls bring theirs
        first = [f.flip(2).contiguous() for f in s.frames]
        s.fe.graph_capture(_jobs(case, streams, first))
        s.first = first
    if kind in ("pair", "step"):
        if kind == "step":  # the keypoints of the last frame, to track into this one
            last = torch.roll(s.frames[0], 1, 2)
            s.fe.extract(last[0], last[1], **s.args)
            s.fe.sync()
            kp = s.fe.keypoints(0, 0)
            s.queries = (kp["X"].float() - 1.0, kp["Y"].float(), kp["level"].clone(),
                         kp["desc"].view(torch.int32).clone())
            torch.cuda.synchronize()
        s.fe.extract(s.frames[0][0], s.frames[0][1], **s.args)
        s.fe.match()
    elif kind == "host" or kind in ("batch", "mixed", "skip", "refine"):
        s.fe.extract_batch(s.batch)
        s.fe.match()
    s.fe.sync()
    if kind in ("pair", "step", "graph", "host"):
        size, _ = s.fe.result_range(0, s.n)
        s.result = torch.zeros(size, dtype=torch.uint8).pin_memory()
    elif kind == "refine":
        s.fe.refine_matches(5, 5, _BF)
        s.fe.sync()
        s.out = [{k: _kept(s.fe, v) for k, v in s.fe.refined(p).items() if k != "count"} for p in range(s.n)]
    else:
        s.out = {"block": _device_blocks(s.fe, s.n)}
        if kind == "skip":
            views = [s.fe.skip_view(p, side) for p in range(s.n) for side in (0, 1)]
            s.out["logits"] = [_kept(s.fe, v["logits"]) for v in views]
            s.out["skip"] = [_kept(s.fe, v["skip"]) for v in views]
    return s


def run(s):
    fe, kind = s.fe, s.kind
    if kind in ("batch", "mixed", "skip"):
        fe.extract_batch(s.batch)
        fe.match()
        return s.out
    if kind == "refine":
        fe.refine_matches(5, 5, _BF)
        return s.out
    out = {"block": s.result}
    if kind == "host":
        fe.extract_batch(s.batch)
        fe.match()
    elif kind == "graph":
        f = s.frames[0]
        fe.graph_launch([jslam.Job(f[0], f[1], **s.args)])
    else:
        f = s.frames[0]
        fe.extract(f[0], f[1], **s.args)
        fe.match()
        if kind == "step":
            fe.refine_matches(5, 5, _BF)
            out["track"] = fe.track(0, 0, *s.queries, radius=8.0)
    fe.download_range(0, s.n, s.result)
    fe.sync()
    return out


# ------------------------------------------------------------------ work, exact values

def _level_pixels(width, height, levels, scale):
    return [round(width / scale ** n) * round(height / scale ** n) for n in range(levels)]


def work(case):
    total, flops = 0, 0
    for _, width, height, levels, feats in _streams(case):
        px = _level_pixels(width, height, levels, case["scale"])
        if case["kind"] == "refine":
            # per left keypoint: its 11 x 11 window, the 11 x 21 strip of the
            # other view, the match in, disparity, depth and SAD out
            total += feats * (121 + 231 + 4 + 12)
            flops += feats * 2 * 11 * 121
            continue
        # per image: level 0 read, the deeper raw levels and every blurred
        # level written, keypoint records and descriptors; per pair matches
        total += 2 * (px[0] + sum(px[1:]) + sum(px) + 48 * feats) + 8 * feats
        if case["kind"] in ("host", "pair", "step", "graph"):
            total += 2 * 56 * feats + 8 * feats  # the download
        if case["kind"] == "host":
            total += 2 * px[0]                    # the upload
        if case["kind"] == "step":
            total += feats * (121 + 231 + 4 + 12) + feats * (9 + 32 + 6)
        if case["kind"] == "skip":
            cells = ((width + 7) // 8) * ((height + 7) // 8)
            total += 2 * cells * 4
            flops += 2 * cells * 2 * 9 * (16 + 256 + 16)
    return {"bytes": total, "flops": flops}


def _exact_logits(image, blob):
    """The three convolutions of the skip model in 64 bits, on the 8x8 box means of one image."""
    c = 16
    bias = np.frombuffer(blob, np.float32, 2 * c + 1, 16)
    raw = np.frombuffer(blob, np.uint16, c * 9 + c * c * 9 + c * 9, 16 + 4 * (2 * c + 1))
    weight = torch.from_numpy((raw.astype(np.uint32) << 16).view(np.float32).astype(np.float64)).cuda()
    w1, w2, w3 = weight[:c * 9], weight[c * 9:c * 9 + c * c * 9], weight[-c * 9:]
    b = torch.from_numpy(bias.astype(np.float64)).cuda()
    height, width = image.shape
    h8, w8 = (height + 7) // 8, (width + 7) // 8
    pad = torch.zeros((2, h8 * 8, w8 * 8), dtype=torch.float64, device="cuda:0")
    pad[0, :height, :width] = image.double()
    pad[1, :height, :width] = 1.0
    box = pad.view(2, h8, 8, w8, 8).sum((2, 4))
    x = (box[0] / box[1] / 255.0 - 0.5)[None, None]
    conv = torch.nn.functional.conv2d
    x = conv(x, w1.view(c, 1, 3, 3), b[:c], padding=1).relu()
    x = conv(x, w2.view(c, c, 3, 3), b[c:2 * c], padding=1).relu()
    return conv(x, w3.view(1, c, 3, 3), b[2 * c:], padding=1)[0, 0]


def exact(case, seed):
    """The skip model's logits in 64 bits; the other outputs are whole numbers
    and packed result blocks, and the refinement's follow from them."""
    if case["kind"] != "skip":
        return None
    blob, _ = _skip_model()
    logits = [_exact_logits(f[side], blob) for f in _all_frames(case, seed) for side in (0, 1)]
    return {"block": None, "logits": logits, "skip": None}
