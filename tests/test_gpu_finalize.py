"""The aggregation's finalisation over every number of CTAs an image: caps
below, at and above the survivors, ties at the threshold, empty levels and
more segments than the kernel keeps on chip, against the oracle."""
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


def _tied(h, w):
    """Dots of equal contrast on a flat image: equal priorities almost everywhere."""
    img = np.full((h, w), 90, np.uint8)
    img[24:h - 24:16, 24:w - 24:16] = 150
    img[25:h - 24:16, 24:w - 24:16] = 150
    return img


# slots an image from below one CTA's share to eight CTAs', caps that bind
# and that do not; cell 4 on a tall image: more than 1024 segments
@pytest.mark.parametrize("width,height,levels,cell,k,pairs,cap", [
    (160, 120, 2, 32, 1, 1, 5), (160, 120, 1, 32, 1, 1, 500), (640, 480, 4, 32, 1, 1, 300),
    (1241, 376, 8, 32, 1, 1, 1), (1241, 376, 8, 32, 1, 1, 2000), (800, 600, 5, 16, 1, 2, 3999),
    (1920, 1080, 8, 32, 1, 1, 3000), (1920, 1080, 8, 32, 1, 1, 20000), (640, 480, 3, 8, 3, 3, 4000),
    (300, 1500, 4, 4, 1, 1, 7000), (640, 480, 2, 32, 1, 100, 123),
])
@pytest.mark.parametrize("tied", [False, True])
def test_finalize_parity(J, oracle, width, height, levels, cell, k, pairs, cap, tied):
    import torch
    p = params_from(oracle, levels=levels, max_feats=cap, cell=cell, k_per_cell=k, fast_thresh_lo=7)
    img = _tied(height, width) if tied else scenes.random_image(height, width, 3)
    flat = np.full_like(img, 77)
    want = oracle.extract_image(img, p)
    fe = frontend_for(J, p, max_width=width, max_height=height, max_pairs=pairs)
    a, z = torch.from_numpy(img).cuda(), torch.from_numpy(flat).cuda()
    torch.cuda.synchronize()
    job = J.Job(a, z, levels=p.levels, scale=p.scale, fast_thresh=p.fast_thresh, cell=cell, max_feats=cap)
    for _ in range(2):  # the second run finds the score map as the first one left it
        fe.extract_batch([job] * pairs)
        fe.match()
        fe.sync()
        compare_keypoints(J.to_numpy(fe.keypoints(pairs - 1, 0)), want, "left")
        assert fe.keypoints(pairs - 1, 1)["count"] == 0
    fe.close()
