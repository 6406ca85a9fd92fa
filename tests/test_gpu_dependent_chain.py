"""The whole chain enqueued back to back with other frames in every pair and
call: extraction, matching, refinement and tracking, graph replays, host frames
in parts and cascaded pyramids of a large scale, each against the oracle for
the first, a middle and the last pair."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes
from parity_util import compare_keypoints, compare_matches, frontend_for, params_from
from test_gpu_refine import BF, _compare as compare_refined

pytestmark = pytest.mark.gpu

CALLS = 6
RADIUS = 6.0


def _scene(width, height, count=3):
    pairs = [scenes.planes_pair(width, height, 0, s, s + 1) for s in (3, 8, 13)[:count]]
    return [(np.ascontiguousarray(f.left), np.ascontiguousarray(f.right)) for f in pairs]


def _device(frames):
    import torch
    dev = [[torch.from_numpy(im).cuda() for im in f] for f in frames]
    torch.cuda.synchronize()
    return dev


def _jobs(J, images, p, pairs, call):
    """Pair i of a call shows frame (call + i) mod 3."""
    return [J.Job(*images[(call + i) % len(images)], levels=p.levels, scale=p.scale, fast_thresh=p.fast_thresh,
                  cell=p.cell, max_feats=p.max_feats) for i in range(pairs)]


def _check(J, fe, want, pairs, call, what):
    for i in sorted({0, pairs // 2, pairs - 1}):
        kl, kr, m = want[(call + i) % len(want)]
        compare_keypoints(J.to_numpy(fe.keypoints(i, 0)), kl, f"{what} {i} left")
        compare_keypoints(J.to_numpy(fe.keypoints(i, 1)), kr, f"{what} {i} right")
        compare_matches(J.to_numpy(fe.matches(i)), m, f"{what} {i}")


@pytest.mark.parametrize("width,height,levels,pairs,options,window", [
    (320, 240, 4, 1, {}, (5, 5)), (752, 480, 8, 3, {}, (3, 4)), (640, 480, 4, 24, {}, (5, 5)),
    (320, 240, 4, 3, dict(pyramid_mode=1), (7, 2)), (640, 480, 6, 24, dict(pyramid_mode=1), (5, 3)),
])
def test_chain_back_to_back(J, oracle, width, height, levels, pairs, options, window):
    import torch
    p = params_from(oracle, levels=levels, max_feats=700, fast_thresh_lo=7, **options)
    frames = _scene(width, height)
    want = [oracle.extract_pair(a, b, p) for a, b in frames]
    queries = want[0][0]  # the first frame's left keypoints, looked for in every frame
    n = queries["count"]
    q = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
         (queries["X"][:n].astype(np.float32), queries["Y"][:n].astype(np.float32),
          queries["level"][:n].astype(np.uint8), queries["desc"][:n].view(np.int32))]
    dev = _device(frames)
    fe = frontend_for(J, p, max_width=width, max_height=height, max_pairs=pairs)
    mid, kept = pairs // 2, []
    for first in range(2):
        for call in range(first, first + CALLS):  # no wait between the calls
            fe.extract_batch(_jobs(J, dev, p, pairs, call))
            fe.match()
            fe.refine_matches(*window, BF)
            kept.append(fe.track(mid, 0, *q, RADIUS))
        fe.sync()
        _check(J, fe, want, pairs, call, f"from {first}")
        for i in sorted({0, mid, pairs - 1}):
            f = (call + i) % 3
            kl, kr, m = want[f]
            compare_refined(J.to_numpy(fe.refined(i)), oracle.subpixel(*frames[f], kl, kr, m[0], p, *window, BF),
                            f"{first} {i}")
        idx, dist = kept[-1]
        wi, wd = oracle.track(want[(call + mid) % 3][0], p.scale, queries["X"][:n].astype(np.float32),
                              queries["Y"][:n].astype(np.float32), queries["level"][:n], queries["desc"][:n], RADIUS)
        assert np.array_equal(idx.cpu().numpy(), wi)
        assert np.array_equal(dist.cpu().numpy().view(np.uint16), wd)
    fe.close()


@pytest.mark.parametrize("pairs", [1, 9])
def test_graph_replays_back_to_back(J, oracle, pairs):
    import torch
    p = params_from(oracle, levels=5, max_feats=600, fast_thresh_lo=7)
    frames = _scene(420, 300)
    want = [oracle.extract_pair(a, b, p) for a, b in frames]
    dev = _device(frames)
    fe = frontend_for(J, p, max_width=420, max_height=300, max_pairs=pairs, stream=torch.cuda.Stream())
    fe.graph_capture(_jobs(J, dev, p, pairs, 0))
    for last in range(1, 4):
        batches = [fe.prepare_batch(_jobs(J, dev, p, pairs, call)) for call in range(last, last + CALLS)]
        for b in batches:
            fe.graph_launch(b)
        fe.refine_matches(5, 5, BF)  # enqueued after the last replay
        fe.sync()
        call = last + CALLS - 1
        _check(J, fe, want, pairs, call, f"replays from {last}")
        f = (call + pairs - 1) % 3
        kl, kr, m = want[f]
        compare_refined(J.to_numpy(fe.refined(pairs - 1)), oracle.subpixel(*frames[f], kl, kr, m[0], p, 5, 5, BF), "graph")
    fe.close()


def test_host_frames_back_to_back(J, oracle):
    """Twelve pairs of 752x480 (8.7 MB) go up in two parts; the frames of the
    next call are other buffers, uploaded while the call before runs."""
    import torch
    pairs, w, h = 12, 752, 480
    p = params_from(oracle, levels=4, max_feats=500, fast_thresh_lo=7)
    frames = _scene(w, h)
    want = [oracle.extract_pair(a, b, p) for a, b in frames]
    fe = frontend_for(J, p, max_width=w, max_height=h, max_pairs=pairs)
    batches, keep = [], []
    for call in range(3):
        pinned = torch.empty((pairs, 2, h, w), dtype=torch.uint8).pin_memory()
        host = pinned.numpy()
        for i in range(pairs):
            host[i, 0], host[i, 1] = frames[(call + i) % 3]
        keep.append(pinned)
        batches.append(fe.prepare_batch([J.Job(host[i, 0], host[i, 1], levels=p.levels, scale=p.scale,
                                               fast_thresh=p.fast_thresh, cell=p.cell, max_feats=p.max_feats)
                                         for i in range(pairs)]))
    for call in (0, 1, 2, 1):
        fe.extract_batch(batches[call])
        fe.match()
    fe.sync()
    _check(J, fe, want, pairs, 1, "host")
    fe.close()


@pytest.mark.parametrize("pairs", [1, 3])
def test_cascade_of_scale_seven(J, oracle, pairs):
    """Taps too far apart for byte windows: levels 1 and 2 read single bytes of
    the level above, in launches that start while that level is written."""
    p = params_from(oracle, levels=3, scale=7.0, max_feats=500, fast_thresh_lo=7, border=16, pyramid_mode=1)
    frames = _scene(2020, 1820, 2)
    want = [oracle.extract_pair(a, b, p) for a, b in frames]
    dev = _device(frames)
    fe = frontend_for(J, p, max_width=2020, max_height=1820, max_pairs=pairs)
    for last in range(2):
        for call in range(last, last + CALLS):
            fe.extract_batch(_jobs(J, dev, p, pairs, call))
            fe.match()
        fe.sync()
        _check(J, fe, want, pairs, call, f"scale 7 from {last}")
        for side in (0, 1):
            img = frames[(call + pairs - 1) % 2][side]
            for n in range(3):
                got = fe.level(pairs - 1, side, n)["raw"].cpu().numpy()
                if n:
                    img = oracle.pyramid_level_sized(img, p.scale, 1, got.shape[1], got.shape[0])
                assert np.array_equal(got, img), (side, n)
    fe.close()
