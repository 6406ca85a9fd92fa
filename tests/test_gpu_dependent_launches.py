"""Calls enqueued back to back with other frames each time, on both sides of the
detection tiles that run at once: every kernel sees the results of the one
before it, against the oracle."""
import numpy as np
import pytest

from paper_2410_04090_gb300 import scenes
from parity_util import compare_keypoints, frontend_for, params_from

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def J():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_04090_gb300 import build
    build.build()
    from paper_2410_04090_gb300 import jslam
    return jslam


@pytest.mark.parametrize("width,height,levels,pairs,options", [
    (160, 120, 1, 1, {}), (320, 240, 4, 1, {}), (752, 480, 8, 2, {}), (640, 480, 4, 40, {}),
    (320, 240, 4, 1, dict(pyramid_mode=1)), (640, 480, 4, 40, dict(pyramid_mode=1)),
])
def test_back_to_back_calls(J, oracle, width, height, levels, pairs, options):
    import torch
    p = params_from(oracle, levels=levels, max_feats=700, fast_thresh_lo=7, **options)
    pairs_of = [scenes.planes_pair(width, height, 0, s, s + 1) for s in (3, 8, 13)]
    frames = [(f.left, f.right) for f in pairs_of]
    want = [[oracle.extract_image(im, p) for im in f] for f in frames]
    fe = frontend_for(J, p, max_width=width, max_height=height, max_pairs=pairs)
    dev = [[torch.from_numpy(np.ascontiguousarray(im)).cuda() for im in f] for f in frames]
    torch.cuda.synchronize()
    for last in range(3):
        for k in range(7):  # no wait between the calls; the last one has frame pair `last`
            a, b = dev[(last + k + 1) % 3] if k < 6 else dev[last]
            fe.extract_batch([J.Job(a, b, levels=levels, scale=p.scale, fast_thresh=p.fast_thresh, cell=p.cell,
                                    max_feats=p.max_feats)] * pairs)
            fe.match()
        fe.sync()
        for pair in {0, pairs - 1}:
            for side in (0, 1):
                compare_keypoints(J.to_numpy(fe.keypoints(pair, side)), want[last][side], f"{last} {pair} {side}")
    fe.close()
